// Single-precision rotational M2L with the whole pair in registers (orders
// 1..12 of the mixed form).
//
// One weak pair per thread. Its (p+1)^2 real coefficient values (the m = 0
// imaginary parts are zero by the real-source symmetry) stay in registers
// between the stages, and every entry of the fixed matrices d^n(pi/2) and of
// the axial translation is an immediate operand of its multiply-add: no table
// reads and no storage between the stages. Zero entries (k = 0 or m = 0 of
// the imaginary part) drop out at compile time: 4,381 multiply-adds per pair
// at p = 12 instead of 4,914, in about 7,300 instructions (the kernel that
// kept the pair in tensor and shared memory and read the tables from shared
// memory took 12,300).
//
// What bounds it: instruction issue of two warps per scheduler (255
// registers), over 60% busy, with the straight-line code (120 KB at p = 12)
// read through the instruction caches, and the 32-lane sums into the targets
// (0.9 of 5.4 ms). 1.62e7 pairs of 2M Plummer points, 14 levels, M2L stage
// before and now: p = 12 10.74 -> 5.18 ms, p = 10 6.91 -> 3.40, p = 8 4.39 ->
// 1.75, p = 4 1.64 -> 0.55; odd orders (formerly tensor-core products) p = 9
// 81.5 -> 2.75.
#pragma once

#include <algorithm>
#include <type_traits>
#include <utility>

#include "fmm_internal.cuh"
#include "m2l_common.cuh"

namespace fmm {
namespace reg {

// ---- the fixed matrices as compile-time constants
constexpr double c_sqrt(double x) {
    double y = x > 1.0 ? x : 1.0;
    for (int i = 0; i < 400; i++) {
        const double z = 0.5 * (y + x / y);
        if (z >= y) break;  // Newton from above decreases until it rounds to the root
        y = z;
    }
    return y;
}
constexpr double c_fact(int n) {
    double r = 1.0;
    for (int i = 2; i <= n; i++) r *= i;
    return r;
}
constexpr long long c_binom(int n, int k) {
    if (k < 0 || k > n) return 0;
    long long r = 1;
    for (int i = 1; i <= k; i++) r = r * (n - k + i) / i;
    return r;
}
// d^n_{km}(pi/2) = 2^-n sqrt((n+k)!(n-k)! / ((n+m)!(n-m)!)) sum_s (-1)^(k-m+s) C(n+m, s) C(n-m, n-k-s):
// the alternating sum is an integer, so zeros are exact
constexpr double c_wigner(int n, int k, int m) {
    long long t = 0;
    for (int s = 0; s <= n + m; s++) {
        const long long v = c_binom(n + m, s) * c_binom(n - m, n - k - s);
        t += ((k - m + s) & 1) ? -v : v;
    }
    double sc = 1.0;
    for (int i = 0; i < n; i++) sc *= 0.5;
    return sc * (double)t * c_sqrt(c_fact(n + k) / c_fact(n + m) * (c_fact(n - k) / c_fact(n - m)));
}
constexpr double c_F(int n, int m) { return c_sqrt(c_fact(n + m)) * c_sqrt(c_fact(n - m)); }
// entry (K, M) of the folds of degree N: forward first / second, inverse first / second
enum { kFwd1, kFwd2, kInv1, kInv2 };
constexpr float c_fold(int tab, int n, int k, int m) {
    const bool tr = tab == kFwd2 || tab == kInv2;
    double g = tr ? c_wigner(n, m, k) : c_wigner(n, k, m);
    if (!tr) g *= (m ? 2.0 : 1.0) * (k ? 2.0 : 1.0);
    if (tab == kFwd1) g *= c_F(n, m);
    if (tab == kInv2) g *= c_F(n, k);
    return (float)g;
}
constexpr float c_axial(int l, int k, int n) {
    const double a = c_fact(n + k) / (c_F(n, l) * c_F(k, l));
    return (float)(((k + l) & 1) ? -a : a);
}
template <int TAB, int N, int K, int M>
struct Fold {
    static constexpr float v = c_fold(TAB, N, K, M);
};
template <int L, int K, int N>
struct Axial {
    static constexpr float v = c_axial(L, K, N);
};

template <int... I, typename F>
__device__ __forceinline__ void for_impl(std::integer_sequence<int, I...>, F &&f) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F &&f) {
    for_impl(std::make_integer_sequence<int, N>{}, static_cast<F &&>(f));
}

// sum of the fold's row K over m = M0, M0 + 2, ... <= N of v[m]
template <int TAB, int N, int K, int M0>
__device__ __forceinline__ float row(const float (&v)[N + 1]) {
    float a = 0.f;
    bool first = true;
    static_for<(N - M0) / 2 + (M0 <= N ? 1 : 0)>([&](auto j) {
        constexpr int M = M0 + 2 * decltype(j)::value;
        constexpr float c = Fold<TAB, N, K, M>::v;
        if constexpr (c != 0.f) {
            a = first ? c * v[M] : fmaf(c, v[M], a);
            first = false;
        }
    });
    return a;
}

// out = fold of v: re_k over the m of parity n + k, im_k over the others
template <int TAB, int N>
__device__ __forceinline__ void fold(const float (&vr)[N + 1], const float (&vi)[N + 1], float (&re)[N + 1],
                                     float (&im)[N + 1]) {
    static_for<N + 1>([&](auto kk) {
        constexpr int K = decltype(kk)::value, par = (N + K) & 1;
        re[K] = row<TAB, N, K, par>(vr);
        im[K] = row<TAB, N, K, 1 - par>(vi);
    });
}

// per-pair state: coefficient (n, m) at tri(n, m)
template <int P>
struct State {
    float r[(P + 1) * (P + 2) / 2], i[(P + 1) * (P + 2) / 2];
};

// powers 1..P of a unit complex number
template <int P>
struct Phases {
    float2 z[P + 1];
    __device__ __forceinline__ void set(float2 b) {
        z[0] = make_float2(1.f, 0.f);
        if constexpr (P >= 1) z[1] = b;
#pragma unroll
        for (int k = 2; k <= P; k++)
            z[k] = make_float2(z[k - 1].x * b.x - z[k - 1].y * b.y, z[k - 1].x * b.y + z[k - 1].y * b.x);
    }
};

template <int N>
__device__ __forceinline__ void phase(float (&r)[N + 1], float (&i)[N + 1], const float2 *z) {
#pragma unroll
    for (int m = 1; m <= N; m++) {
        const float a = r[m] * z[m].x - i[m] * z[m].y;
        i[m] = r[m] * z[m].y + i[m] * z[m].x;
        r[m] = a;
    }
}

// ---- staging of the source multipoles
// A warp's 32 source rows sit in its slice of shared memory at their stride in
// global memory, an odd number of 16-byte pieces (conflict-free 16-byte reads
// down the lanes).
__host__ __device__ constexpr int row_bytes(int p) { return 8 * mf_stride(p); }

// a read-only load that stays where it is written (the compiler would sink it
// to its use, past the arithmetic that is to hide it)
__device__ __forceinline__ float4 ld4(const void *p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}

// The lanes' source rows, counted on the warp's mbarrier: one bulk copy for
// each run of consecutive boxes (a target's sources ascend and siblings come
// together). A copy's operands are warp-uniform registers, so every copy is a
// trip of a loop: fewer copies, fewer instructions. (withhold >= 0, tests only:
// the run that holds this box is left out, and the wait for it runs out.)
template <int P>
__device__ __forceinline__ void copy_rows(const float2 *__restrict__ Mf, int gs, const char *row, uint32_t bar,
                                          int withhold) {
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(0xffffffffu, gs, 1);
    const bool head = lane == 0 || gs != prev + 1;
    const unsigned later = __ballot_sync(0xffffffffu, head) & (0xfffffffeu << lane);
    const int len = (later ? __ffs(later) - 1 : 32) - lane;
    if (lane == 0)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(32 * row_bytes(P))
                     : "memory");
    __syncwarp();
    if (head && !(withhold >= gs && withhold < gs + len))
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                (uint32_t)__cvta_generic_to_shared(row)),
            "l"(Mf + (int64_t)gs * mf_stride(P)), "r"(len * row_bytes(P)), "r"(bar)
            : "memory");
}

// Waits for phase `parity` of the warp's copies: a few tries that suspend in
// hardware (a copy takes microseconds), then `limit` sleeps of ~0.1 us. False if
// the bound ran out.
__device__ __forceinline__ bool wait_rows(uint32_t bar, uint32_t parity, long long limit) {
    uint32_t ok = 0;
    for (int i = 0; i < 8; i++) {
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    for (long long i = 0; i < limit; i++) {
        __nanosleep(100);
        asm volatile(
            "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// the waits' bound and the box whose row is not copied (-1: none), as set by fmm_set_wait_limit
struct Waits {
    long long limit;
    int withhold;
};

// degree N of this lane's row, two coefficients per 16-byte read where the pair is aligned
template <int N>
__device__ __forceinline__ void read_deg(const char *row, float (&r)[N + 1], float (&i)[N + 1]) {
    constexpr int c0 = N * (N + 1) / 2, m0 = c0 & 1;
    const float2 *Ms = (const float2 *)row;
    if constexpr (m0 == 1) {
        const float2 t = Ms[c0];
        r[0] = t.x, i[0] = t.y;
    }
#pragma unroll
    for (int m = m0; m + 1 <= N; m += 2) {
        const float4 t = *(const float4 *)(Ms + c0 + m);
        r[m] = t.x, i[m] = t.y, r[m + 1] = t.z, i[m + 1] = t.w;
    }
    if constexpr (((N + 1 - m0) & 1) == 1) {
        const float2 t = Ms[c0 + N];
        r[N] = t.x, i[N] = t.y;
    }
}

// Block-wide barriers at the start of the largest degrees and orders keep the
// warps of the SM together on the longest straight-line code, so that it is
// fetched once per SM and pass, not once per warp. Measured on 1.62e7 pairs
// with barriers from degree 4 on / P - 2 / P - 1 / none: p = 12 5.36 / 5.05 /
// 5.13 / 5.36 ms, p = 10 3.52 / 3.43 / 3.32 / 3.38, p = 8 2.01 / 1.97 / 1.85 /
// 1.72, p = 6 1.25 / 1.22 / 1.14 / 0.91 (with weighted sums): the code of the orders below 10 fits
// the instruction cache and the barriers only cost.
template <int P>
constexpr int sync_from() { return P >= 12 ? P - 2 : P >= 10 ? P - 1 : P + 1; }

// forward rotation of degree N, scaled by (r_s / rho)^N
template <int P, int N>
__device__ __forceinline__ void fwd(const char *rowp, const float2 *za, const float2 *zb, float qsn, State<P> &S) {
    constexpr int c0 = N * (N + 1) / 2;
    float ur[N + 1], ui[N + 1], xr[N + 1], xi[N + 1];
    read_deg<N>(rowp, ur, ui);
    if constexpr (N >= sync_from<P>()) __syncthreads();
    phase<N>(ur, ui, za);
    fold<kFwd1, N>(ur, ui, xr, xi);
    phase<N>(xr, xi, zb);
    fold<kFwd2, N>(xr, xi, ur, ui);
#pragma unroll
    for (int m = 0; m <= N; m++) {
        S.r[c0 + m] = ur[m] * qsn;
        S.i[c0 + m] = -ui[m] * qsn;
    }
}

// Translation along z of order L, in place. The terms fall with the degree (by
// (r_s / rho)^n), so the sums run from the highest degree down: a chain that
// starts from the small terms loses half as much as one that starts from the
// large ones (potential of a pair's translation, p = 12: 3.7e-8 against 7.2e-8
// relative; two chains added at the end 6.1e-8).
template <int P, int L>
__device__ __forceinline__ void axial(State<P> &S) {
    float sr[P + 1 - L], si[P + 1 - L];
#pragma unroll
    for (int n = L; n <= P; n++) sr[n - L] = S.r[n * (n + 1) / 2 + L], si[n - L] = S.i[n * (n + 1) / 2 + L];
    static_for<P + 1 - L>([&](auto kk) {
        constexpr int K = L + decltype(kk)::value, c = K * (K + 1) / 2 + L;
        float a = 0.f, b = 0.f;
        static_for<P + 1 - L>([&](auto nn) {
            constexpr int j = P - L - decltype(nn)::value;
            constexpr float w = Axial<L, K, L + j>::v;
            a = j == P - L ? w * sr[j] : fmaf(w, sr[j], a);
            if constexpr (L > 0) b = j == P - L ? w * si[j] : fmaf(w, si[j], b);
        });
        S.r[c] = a;
        if constexpr (L > 0) S.i[c] = b;
    });
}

// ---- the sum into the targets
// The inverse rotation leaves its results in columns of a transpose buffer of
// the warp, lane i of column c at 36 c + i (conflict-free writes, 16-byte
// column reads). Degree k takes 2k + 1 columns (Re of orders 0..k, then Im of
// 1..k); consecutive degrees of at most 32 columns in all are summed
// together, one column per lane.
constexpr int kCol = 36;
__host__ __device__ constexpr int group_first(int n) {  // first degree of degree n's group
    int g = 0;
    for (int k = 1; k <= n; k++)
        if ((k + 1) * (k + 1) - g * g > 32) g = k;
    return g;
}

// Column sums of degrees G..N over each of the warp's runs of equal target
// (the pair list is sorted by target; `ends`: the runs' last lanes), added to
// the run's target's scaled local in double. mask: of several runs, the lanes
// of the present one as bits all 1, the others 0, so that a warp with several
// targets costs a pass per run and not a loop over its lanes. (Bits and not
// weights of 0 and 1: another target's sum may hold an infinity. p = 12 5.18 ms
// against 5.10 with weights; weights, and the sums that come out not finite
// formed again, 5.33; loops over a run's quads 5.46.)
template <int P, int G, int N>
__device__ __forceinline__ void sum_group(const float *red, uint32_t *mask, int t32, unsigned ends,
                                          double2 *__restrict__ Lh) {
    constexpr int NC = (P + 1) * (P + 2) / 2, W = (N + 1) * (N + 1) - G * G;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const bool on = lane < W;
    const float4 *c4 = (const float4 *)(red + (on ? lane : 0) * kCol);
    const uint4 *m4 = (const uint4 *)mask;
    auto keep = [](float v, uint32_t m) { return __uint_as_float(__float_as_uint(v) & m); };
    int k = G;
#pragma unroll
    for (int d = G + 1; d <= N; d++) k += lane >= d * d - G * G;
    const int j = lane - (k * k - G * G);
    double *dst = (double *)Lh + 2 * (k * (k + 1) / 2) + (j <= k ? 2 * j : 2 * (j - k) + 1);
#pragma unroll 1
    for (unsigned m = ends; m; m &= m - 1) {  // warp-uniform
        const int t = __shfl_sync(0xffffffffu, t32, __ffs(m) - 1);
        if (ends != 0x80000000u) {
            __syncwarp();
            mask[lane] = t32 == t ? ~0u : 0u;
            __syncwarp();
        }
        float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
        if (ends == 0x80000000u) {  // one target: no mask
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const float4 v = c4[i];
                a0 = __fadd2_rn(a0, make_float2(v.x, v.y));
                a1 = __fadd2_rn(a1, make_float2(v.z, v.w));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const float4 v = c4[i];
                const uint4 u = m4[i];
                a0 = __fadd2_rn(a0, make_float2(keep(v.x, u.x), keep(v.y, u.y)));
                a1 = __fadd2_rn(a1, make_float2(keep(v.z, u.z), keep(v.w, u.w)));
            }
        }
        const float s = (a0.x + a0.y) + (a1.x + a1.y);
        if (on) atomicAdd(dst + (int64_t)t * (2 * NC), (double)s);
    }
    __syncwarp();  // the next group reuses the buffer
}

// inverse rotation of degree N into the transpose buffer, scaled by tp = qt^N / rho
template <int P, int N>
__device__ __forceinline__ void inv(State<P> &S, const float2 *za, const float2 *zb, float tp, float *red,
                                    uint32_t *mask, int t32, unsigned ends, double2 *__restrict__ Lh) {
    constexpr int c0 = N * (N + 1) / 2, G = group_first(N);
    if constexpr (N >= sync_from<P>()) __syncthreads();
    float ur[N + 1], ui[N + 1], xr[N + 1], xi[N + 1];
#pragma unroll
    for (int m = 0; m <= N; m++) ur[m] = S.r[c0 + m] * tp, ui[m] = m ? S.i[c0 + m] * tp : 0.f;
    fold<kInv1, N>(ur, ui, xr, xi);
    phase<N>(xr, xi, zb);
    fold<kInv2, N>(xr, xi, ur, ui);
    phase<N>(ur, ui, za);
    float *col = red + (N * N - G * G) * kCol + (threadIdx.x & 31);
#pragma unroll
    for (int l = 0; l <= N; l++) {
        col[l * kCol] = ur[l];
        if (l) col[(N + l) * kCol] = ui[l];
    }
    if constexpr (N == P || group_first(N + 1) != G) sum_group<P, G, N>(red, mask, t32, ends, Lh);
}

// bytes of a warp's slice of shared memory: its source rows, the run's mask, the transpose buffer, the mbarrier of the copies
template <int P>
__host__ __device__ constexpr int slice_bytes() {
    return 32 * row_bytes(P) + 128 + 4 * kCol * ((P + 1) * (P + 1) < 32 ? (P + 1) * (P + 1) : 32) + 16;
}
// Warps per SM (one block): what the registers of order P (65,536 per SM) and
// shared memory allow. On 1.62e7 pairs: p = 9 2.89 ms with 8 warps (2.91 with
// 11), p = 8 2.01 with 12 (2.31 with 8), p = 7 1.67 with 16 (1.73 with 12),
// p = 6 1.26 with 16 (1.33 with 12), p = 4 0.72 with 24 (0.80 with 16).
template <int P>
constexpr int warps() { return P >= 9 ? 8 : P >= 8 ? 12 : P >= 5 ? 16 : 24; }
template <int P>
constexpr size_t smem_bytes() { return (size_t)slice_bytes<P>() * warps<P>(); }

// One warp's 32 pairs: chunk w of the pair list (all of one system)
struct Cursor {
    int gt, gs;   // target and source box of this lane's pair
    int sys;      // system (batched)
    bool valid;   // lanes past the end repeat the last pair, for no target
};

// the pairs of one plan
struct OnePlan {
    const PairTable &PT;
    const float4 *cf_;
    const float2 *Mf_;
    double2 *Lh_;
    int *err_;
    int lev;
    __device__ __forceinline__ unsigned chunks() const { return (unsigned)((PT.off[PT.lmax + 1] + 31) >> 5); }
    __device__ __forceinline__ Cursor at(unsigned w) {
        int64_t g = (int64_t)w * 32 + (threadIdx.x & 31);
        const int64_t last = PT.off[PT.lmax + 1] - 1;
        Cursor c;
        c.valid = g <= last;
        c.sys = 0;
        if (!c.valid) g = last;
        while (lev < PT.lmax && g >= PT.off[lev + 1]) lev++;  // pairs only move forward
        const int64_t e = g - PT.off[lev];
        const int boff = (1 << lev) - 1;
        c.gt = boff + PT.tgt[lev][e];
        c.gs = boff + PT.src[lev][e];
        return c;
    }
    __device__ __forceinline__ const float4 *cf(const Cursor &) const { return cf_; }
    __device__ __forceinline__ const float2 *Mf(const Cursor &) const { return Mf_; }
    __device__ __forceinline__ double2 *Lh(const Cursor &) const { return Lh_; }
    __device__ __forceinline__ int *err(const Cursor &) const { return err_; }
};

// the pairs of every system of one order; off counts chunks of 128 pairs
struct Batched {
    const BatchSys *__restrict__ S;
    const int32_t *__restrict__ off;
    int nsys;
    __device__ __forceinline__ unsigned chunks() const { return (unsigned)off[nsys] * 4u; }
    __device__ __forceinline__ Cursor at(unsigned w) {
        const int ch = (int)(min(w, chunks() - 1u) >> 2);
        Cursor c;
        c.sys = batch_sys_of(off, nsys, ch);
        const BatchSys &y = S[c.sys];
        int64_t g = ((int64_t)w - (int64_t)off[c.sys] * 4) * 32 + (threadIdx.x & 31);
        c.valid = g < y.npairs;
        if (!c.valid) g = y.npairs - 1;
        int64_t gt, gs;
        pair_of(y.pt, g, gt, gs);
        c.gt = (int)gt;
        c.gs = (int)gs;
        return c;
    }
    __device__ __forceinline__ const float4 *cf(const Cursor &c) const { return S[c.sys].box_cf; }
    __device__ __forceinline__ const float2 *Mf(const Cursor &c) const { return S[c.sys].Mf; }
    __device__ __forceinline__ double2 *Lh(const Cursor &c) const { return S[c.sys].Lh; }
    __device__ __forceinline__ int *err(const Cursor &c) const { return S[c.sys].err; }
};

// The loop of one warp over its chunks, in step with the block's other warps.
// The next chunk's source rows are copied to shared memory while this one is
// translated and rotated back.
template <int P, typename Src>
__device__ __forceinline__ void run(Src &src, char *slice, const Waits &wt) {
    const unsigned W = blockDim.x >> 5, total = src.chunks(), stride = gridDim.x * W;
    unsigned w0 = blockIdx.x * W;  // the block's first chunk (device memory holds fewer than 2^31 chunks of pairs)
    if (w0 >= total) return;
    const char *rowp = slice + (threadIdx.x & 31) * row_bytes(P);
    uint32_t *mask = (uint32_t *)(slice + 32 * row_bytes(P));
    float *red = (float *)(mask + 32);
    Cursor nxt = src.at(w0 + (threadIdx.x >> 5));
    float4 th, tl, sh, sl;  // split centres and radii of the next target and source box
    auto geometry = [&](const Cursor &c) {
        const float4 *cf = src.cf(c);
        th = ld4(cf + 2 * (int64_t)c.gt), tl = ld4(cf + 2 * (int64_t)c.gt + 1);
        sh = ld4(cf + 2 * (int64_t)c.gs), sl = ld4(cf + 2 * (int64_t)c.gs + 1);
    };
    geometry(nxt);
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(slice + slice_bytes<P>() - 16);
    if ((threadIdx.x & 31) == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    copy_rows<P>(src.Mf(nxt), nxt.gs, rowp, bar, wt.withhold);
    uint32_t parity = 0;
    bool lost = false;  // a wait ran out (lanes of a warp agree: they test the same barrier phase)
    for (;; w0 += stride) {
        const Cursor cur = nxt;
        // the centre offset from the split centres: the hi difference and its
        // rounding error (TwoSum), plus the lo difference, rounded once
        const float dx = offset_f(th.x, sh.x, tl.x, sl.x), dy = offset_f(th.y, sh.y, tl.y, sl.y),
                    dz = offset_f(th.z, sh.z, tl.z, sl.z);
        const float rxy2 = fmaf(dx, dx, dy * dy);
        const float rxy = sqrtf(rxy2), rinv = rsqrtf(fmaf(dz, dz, rxy2));
        const float rxinv = rxy > 0.f ? 1.f / rxy : 0.f;
        const float2 ea = rxy > 0.f ? make_float2(dx * rxinv, dy * rxinv) : make_float2(1.f, 0.f);
        const float2 eb = make_float2(dz * rinv, rxy * rinv);
        const float2 eai = make_float2(ea.y, -ea.x);  // -i e^{ia}
        const float qs = (sh.w > 0.f ? sh.w : 1.f) * rinv, qt = (th.w > 0.f ? th.w : 1.f) * rinv;
        if (!lost && !wait_rows(bar, parity, wt.limit)) {
            lost = true;  // no more copies; the warp goes on, for the block's barriers (FMM_ETIMEDOUT: results invalid)
            atomicOr(src.err(cur) + 1, 16);
        }
        if (!lost) parity ^= 1;
        State<P> S;
        {
            Phases<P> A, B;
            A.set(eai);
            B.set(eb);
            float qp[P + 1];
            qp[0] = 1.f;
#pragma unroll
            for (int n = 1; n <= P; n++) qp[n] = qp[n - 1] * qs;
            // highest degree first: as the state grows, the degree's temporaries shrink
            static_for<P + 1>([&](auto d) {
                constexpr int N = P - decltype(d)::value;
                fwd<P, N>(rowp, A.z, B.z, qp[N], S);
            });
        }
        // the rows are read: the next ones may replace them (the bulk copies write through the async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        const bool more = w0 + stride < total;  // uniform over the block
        if (more) nxt = src.at(w0 + stride + (threadIdx.x >> 5));
        static_for<P + 1>([&](auto l) {
            constexpr int L = decltype(l)::value;
            if constexpr (P - L >= sync_from<P>()) __syncthreads();
            axial<P, L>(S);
            if constexpr (L == P / 6) {
                if (more && !__any_sync(0xffffffffu, lost)) copy_rows<P>(src.Mf(nxt), nxt.gs, rowp, bar, wt.withhold);
            }
        });
        {
            Phases<P> A, B;
            A.set(eai);
            B.set(eb);
            float tp = rinv;
            const int t32 = cur.valid ? cur.gt : -1, up = __shfl_down_sync(0xffffffffu, t32, 1);
            const unsigned ends = __ballot_sync(0xffffffffu, cur.valid && ((threadIdx.x & 31) == 31 || up != t32));
            double2 *Lh = src.Lh(cur);
            static_for<P + 1>([&](auto n) {
                constexpr int N = decltype(n)::value;
                if constexpr (N == (P * 9 + 9) / 10) {
                    if (more) geometry(nxt);
                }
                inv<P, N>(S, A.z, B.z, tp, red, mask, t32, ends, Lh);
                tp *= qt;
            });
        }
        if (!more) break;
    }
    if (lost) wait_rows(bar, parity, wt.limit);  // its copies still in flight
}

template <int P>
__global__ void __launch_bounds__(warps<P>() * 32, 1)
k_m2l_reg(PairTable PT, const float4 *__restrict__ cf, const float2 *__restrict__ Mf, double2 *__restrict__ Lh,
          int *err, Waits wt) {
    extern __shared__ float4 sm4[];
    OnePlan src{PT, cf, Mf, Lh, err, PT.lmin};
    run<P>(src, (char *)sm4 + (threadIdx.x >> 5) * slice_bytes<P>(), wt);
}

template <int P>
__global__ void __launch_bounds__(warps<P>() * 32, 1)
k_b_m2l_reg(const BatchSys *__restrict__ S, const int32_t *__restrict__ off, int nsys, Waits wt) {
    extern __shared__ float4 sm4[];
    Batched src{S, off, nsys};
    run<P>(src, (char *)sm4 + (threadIdx.x >> 5) * slice_bytes<P>(), wt);
}

template <int P>
cudaError_t reg_attr() {
    cudaError_t e = allow_max_smem((const void *)k_m2l_reg<P>, smem_bytes<P>());
    return e == cudaSuccess ? allow_max_smem((const void *)k_b_m2l_reg<P>, smem_bytes<P>()) : e;
}
// one block per SM, fewer where the pairs are few
template <int P>
unsigned grid(int64_t warp_chunks) {
    return (unsigned)std::min<int64_t>((warp_chunks + warps<P>() - 1) / warps<P>(), sm_count());
}
template <int P>
void reg_launch(const PairTable &PT, int64_t tot, const float4 *cf, const float2 *Mf, double2 *Lh, int *err,
                Waits wt, cudaStream_t st) {
    FMM_LAUNCH(k_m2l_reg<P>, grid<P>((tot + 31) / 32), warps<P>() * 32, smem_bytes<P>(), st, PT, cf, Mf, Lh, err, wt);
}
template <int P>
void reg_launch_batch(const BatchSys *S, const int32_t *off, int nsys, int64_t nchunks, Waits wt, cudaStream_t st) {
    FMM_LAUNCH(k_b_m2l_reg<P>, grid<P>(nchunks * 4), warps<P>() * 32, smem_bytes<P>(), st, S, off, nsys, wt);
}

// explicit instances of one order (each translation unit holds a few: they compile in parallel)
#define FMM_M2L_REG(PRE, P)                                                                                   \
    PRE template cudaError_t reg_attr<P>();                                                                   \
    PRE template void reg_launch<P>(const PairTable &, int64_t, const float4 *, const float2 *, double2 *,    \
                                    int *, Waits, cudaStream_t);                                              \
    PRE template void reg_launch_batch<P>(const BatchSys *, const int32_t *, int, int64_t, Waits, cudaStream_t);

}  // namespace reg
}  // namespace fmm
