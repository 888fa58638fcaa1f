// Near field of the FP64 form (P2P, Algorithm 4) in three-float arithmetic.
//
// What bounds it: the FP32 pipe. A pair takes ~295 packed operations
// (trifloat.cuh) where FP64 arithmetic takes 19 FP64 instructions at less than
// two per clock and SM, ~1,400 FP32 operations' time, and its terms are more
// accurate than those of plain double arithmetic. Sums run in compensated
// three-float accumulators. 200k Plummer points, 11 levels, 1.16e10 pairs: FP64
// arithmetic 412.6 ms (its pipe saturated), this 107.0; 20k uniform points, 8
// levels: 3.29 -> 0.96 ms. A unit is one warp and its 32 targets, staging its
// own sources: units of four warps held their registers until the slowest was
// done (110.7 ms; with block-wide staging and its barriers slower by a
// fifth). Registers: 16 warps per SM (128 registers; 18 warps 109.6 ms).
//
// Positions are taken relative to the root cell's centre on a common grid of
// 2^-72 of its extent (rounded up to a power of two): three floats of 24 bits
// each, whose differences are exact part by part. A double that does not fit
// the grid (a coordinate within 2^-19 of the extent of the centre has finer
// bits) is rounded to it and marked; a pair goes through FP64 arithmetic on the
// original doubles instead when its distance is below 2^-19 of the extent
// with a marked point, below 2^-23 otherwise (that includes r = 0), or when
// the charge is not finite or below 2^-60 of the largest. Such a pair costs
// both arithmetics: 200k Plummer points with one more at 1e5 of their size
// 121 ms, at 1e6 (all near pairs left to FP64) 447, charges over 24 decades
// 145, over 40 245; FP64 arithmetic alone 563 to 581 (whole evaluations).

#include <algorithm>
#include <type_traits>

#include "fmm_internal.cuh"
#include "trifloat.cuh"

namespace fmm {

namespace {

constexpr float kThrExact = 0x1p-46f, kThrRounded = 0x1p-38f;  // on r^2 over the squared extent

// exponent k of the grid's extent: 2^k > the root cell's longest side (a side
// outside the double range's middle: all pairs are left to FP64)
__device__ __forceinline__ bool grid_exponent(const double *__restrict__ lo, const double *__restrict__ hi, int &k) {
    const double w = fmax(fmax(hi[0] - lo[0], hi[1] - lo[1]), hi[2] - lo[2]);
    const int e = w > 0.0 ? ilogb(w) + 1 : 0;
    const bool ok = w < 0x1p1000 && e > -1000;
    k = ok ? e : 0;
    return ok;
}

// coordinate x (relative to centre c) in three floats; false if rounded
__device__ __forceinline__ bool grid_split(double x, double c, double inv, float (&f)[3]) {
    const double u = __dsub_rn(x, c), bb = __dsub_rn(u, x);
    const double e = __dadd_rn(__dsub_rn(x, __dsub_rn(u, bb)), __dsub_rn(-c, bb));  // x - c = u + e
    const double us = u * inv, es = e * inv;
    constexpr double M1 = 0x1.8p28, M2 = 0x1.8p4, M3 = 0x1.8p-20;  // grids 2^-24, 2^-48, 2^-72
    const double a = __dsub_rn(__dadd_rn(us, M1), M1), r = __dsub_rn(us, a);
    const double v = __dadd_rn(r, es), vb = __dsub_rn(v, r);
    const double ve = __dadd_rn(__dsub_rn(r, __dsub_rn(v, vb)), __dsub_rn(es, vb));
    const double b = __dsub_rn(__dadd_rn(v, M2), M2), s = __dsub_rn(v, b);
    const double d = __dsub_rn(__dadd_rn(s, M3), M3);
    f[0] = (float)a, f[1] = (float)b, f[2] = (float)d;
    return d == s && ve == 0.0;
}

// plan time: positions on the grid (component-major: [part][axis][n]) and the thresholds they give
__global__ void k_tf_points(int64_t n, const double *__restrict__ x, const double *__restrict__ y,
                            const double *__restrict__ z, const double *__restrict__ lo,
                            const double *__restrict__ hi, float *__restrict__ pos, float *__restrict__ thr) {
    int k;
    const bool ok = grid_exponent(lo, hi, k);
    const double inv = scalbn(1.0, -k);
    const double *src[3] = {x, y, z};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        bool exact = true;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            float f[3] = {0.f, 0.f, 0.f};
            if (ok) exact &= grid_split(src[a][i], 0.5 * lo[a] + 0.5 * hi[a], inv, f);
#pragma unroll
            for (int c = 0; c < 3; c++) pos[(3 * c + a) * n + i] = f[c];
        }
        thr[i] = !ok ? __int_as_float(0x7f800000) : exact ? kThrExact : kThrRounded;
    }
}

// the largest finite charge's exponent (bits of |q| >> 52)
__global__ void __launch_bounds__(256)
k_tf_qmax(int64_t n, const double *__restrict__ q, int *__restrict__ emax) {
    int m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)((__double_as_longlong(q[i]) >> 52) & 0x7ff);
        if (e < 0x7ff) m = max(m, e);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(emax, m);
}

// 2^q_exponent is above every finite charge (all subnormal or zero: 2^-1022)
__device__ __forceinline__ int q_exponent(int e) { return max(e, 1) - 1022; }

// a charge over 2^e in three floats; its pairs' threshold
__device__ __forceinline__ float charge_split(double q, int e, float thr, float (&f)[3]) {
    const double s = scalbn(q, -e), as = fabs(s);
    const bool ok = as == 0.0 || (as >= 0x1p-60 && as <= 1.0);  // NaN and infinities: no
    f[0] = ok ? (float)s : 0.f;
    const double r = ok ? s - (double)f[0] : 0.0;
    f[1] = (float)r;
    f[2] = (float)(r - (double)f[1]);
    return ok ? thr : __int_as_float(0x7f800000);
}

__device__ __forceinline__ void clear_x(tf::PairTerms<float2> &o) {
    o.phi.a.x = o.phi.b.x = o.phi.c.x = 0.f;
    o.w.a.x = o.w.b.x = o.w.c.x = 0.f;
}
__device__ __forceinline__ void clear_y(tf::PairTerms<float2> &o) {
    o.phi.a.y = o.phi.b.y = o.phi.c.y = 0.f;
    o.w.a.y = o.w.b.y = o.w.c.y = 0.f;
}

// the sums of positions over 2^k and charges over 2^eq, and the FP64 pairs
template <bool F>
__device__ __forceinline__ double4 result(const tf::Sums<float2, F> &A, const double (&slow)[4], int k, int eq) {
    double v[4] = {slow[0], slow[1], slow[2], slow[3]};
#pragma unroll
    for (int c = 0; c < tf::Sums<float2, F>::N; c++) {
        const double m = A.M[c > 0];
        v[c] += scalbn(((double)A.a[c].x + (double)A.a[c].y) +
                           ((((double)A.s[c].x - m) + ((double)A.s[c].y - m)) +
                            ((double)A.c[c].x + (double)A.c[c].y)),
                       c ? eq - 2 * k : eq - k);
    }
    return make_double4(v[0], v[1], v[2], v[3]);
}

// charges over 2^q_exponent in three floats, and the pair thresholds with the charges' own
__global__ void __launch_bounds__(256)
k_tf_charges(int64_t n, const double *__restrict__ q, const int *__restrict__ emax, const float *__restrict__ thr0,
             float *__restrict__ tq, float *__restrict__ thr) {
    const int e = q_exponent(*emax);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float f[3];
        thr[i] = charge_split(q[i], e, thr0[i], f);
#pragma unroll
        for (int c = 0; c < 3; c++) tq[c * n + i] = f[c];
    }
}

constexpr int kT = kP2PTile;  // threads and targets of a block of the direct sum
constexpr int kChunk = 64;    // sources staged at a time by a warp

// source j on target i in FP64 on the original positions, pairs at zero distance skipped
__device__ __noinline__ void pair_f64(const double *__restrict__ x, const double *__restrict__ y,
                                      const double *__restrict__ z, const double *__restrict__ q, int i, int j,
                                      double (&s)[4]) {
    const double dx = x[i] - x[j], dy = y[i] - y[j], dz = z[i] - z[j];
    const double r2 = dx * dx + dy * dy + dz * dz;
    const double rinv = r2 > 0.0 ? rsqrt(r2) : 0.0;
    const double qr = q[j] * rinv, qr3 = qr * rinv * rinv;
    s[0] += qr;
    s[1] += qr3 * dx;
    s[2] += qr3 * dy;
    s[3] += qr3 * dz;
}

template <typename OutT, bool F>  // F: with the field
__global__ void __launch_bounds__(kP2PTileTf, 16)
k_p2p_tf(int B, int64_t n, const double *__restrict__ x, const double *__restrict__ y, const double *__restrict__ z,
         const double *__restrict__ q, const float *__restrict__ pos, const float *__restrict__ tq,
         const float *__restrict__ thr0, const float *__restrict__ thr, const double *__restrict__ lo,
         const double *__restrict__ hi, const int *__restrict__ emax, const int32_t *__restrict__ begin,
         const int32_t *__restrict__ count, const int32_t *__restrict__ ssrc, const int4 *__restrict__ units,
         const int32_t *__restrict__ upart, const int32_t *__restrict__ nunits, const int32_t *__restrict__ perm,
         const double *__restrict__ far_phi, const double *__restrict__ far_E, double4 *__restrict__ partial,
         OutT *__restrict__ pot, OutT *__restrict__ field) {
    // per source pair: parts a, b, c of (x, y, z, q), the two sources side by
    // side. A unit is one warp: a chunk is some 20,000 cycles of arithmetic, so
    // several warps loading the same one cost nothing, and the short ones (a
    // leaf's last targets, sliced over the lanes) give their place up when done.
    constexpr int kT = kP2PTileTf;
    __shared__ float4 sm[6][kChunk / 2];
    __shared__ float2 sthr[kChunk / 2];
    __shared__ double4 red[kT];
    if ((int)blockIdx.x >= *nunits) return;  // launched for an upper bound on the units
    const int64_t off = ((int64_t)1 << B) - 1;
    const int4 unit = units[blockIdx.x];
    const int part = upart[blockIdx.x];
    const int t = unit.x, tid = threadIdx.x;
    const int bt = begin[off + t], nt = count[off + t];
    const P2PLane L(min(kT, nt - unit.y), kT, tid);
    const int i = unit.y + L.target, slot = bt + i;
    const bool busy = __any_sync(0xffffffffu, L.active);  // warp-uniform
    tf::Tri<float2> X[3];
    float thr_i = 0.f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        float f[3] = {0.f, 0.f, 0.f};
        if (L.active)
#pragma unroll
            for (int c = 0; c < 3; c++) f[c] = pos[(3 * c + a) * n + slot];
        X[a] = {make_float2(f[0], f[0]), make_float2(f[1], f[1]), make_float2(f[2], f[2])};
    }
    if (L.active) thr_i = thr0[slot];
    tf::Sums<float2, F> A(make_float2(0.f, 0.f));
    double slow[4] = {0.0, 0.0, 0.0, 0.0};
    float *fs = (float *)sm, *ft = (float *)sthr;
    for (int e = unit.z; e < (busy ? unit.w : 0); e++) {
        const int64_t gs = off + ssrc[e];
        const int bs = begin[gs], ns = count[gs];
        for (int sb = 0; sb < ns; sb += kChunk) {
            __syncwarp();
#pragma unroll
            for (int h = 0; h < kChunk; h += 32) {
                const int s = h + (tid & 31), j = sb + s;
                float v[12] = {}, th = 0.f;
                v[0] = -1.f;  // padding: a zero charge away from every target
                if (j < ns) {
#pragma unroll
                    for (int c = 0; c < 3; c++) {
#pragma unroll
                        for (int a = 0; a < 3; a++) v[4 * c + a] = -pos[(3 * c + a) * n + bs + j];
                        v[4 * c + 3] = tq[c * n + bs + j];
                    }
                    th = thr[bs + j];
                }
#pragma unroll
                for (int c = 0; c < 12; c++)
                    fs[((c >> 1) * (kChunk / 2) + (s >> 1)) * 4 + 2 * (c & 1) + (s & 1)] = v[c];
                ft[s] = th;
            }
            __syncwarp();
            const int np = (min(kChunk, ns - sb) + 1) >> 1;
#pragma unroll 1
            for (int pp = L.slice; pp < np; pp += L.slices) {
                const float4 a0 = sm[0][pp], a1 = sm[1][pp], b0 = sm[2][pp], b1 = sm[3][pp], c0 = sm[4][pp],
                             c1 = sm[5][pp];
                const float2 th = sthr[pp];
                const tf::Tri<float2> Y[3] = {
                    {make_float2(a0.x, a0.y), make_float2(b0.x, b0.y), make_float2(c0.x, c0.y)},
                    {make_float2(a0.z, a0.w), make_float2(b0.z, b0.w), make_float2(c0.z, c0.w)},
                    {make_float2(a1.x, a1.y), make_float2(b1.x, b1.y), make_float2(c1.x, c1.y)}};
                const tf::Tri<float2> Q = {make_float2(a1.z, a1.w), make_float2(b1.z, b1.w), make_float2(c1.z, c1.w)};
                tf::PairTerms<float2> o = tf::pair_terms<float2, F>(X, Y, Q);
                const bool bx = o.r2.x < fmaxf(th.x, thr_i), by = o.r2.y < fmaxf(th.y, thr_i);
                if (bx || by) {
                    const int j0 = sb + 2 * pp;  // the leaf's sources j0 and j0 + 1 (padding past its last one)
                    if (bx) {
                        // a target meets itself once: nothing, unless its charge is not finite
                        if (L.active && (bs + j0 != slot || isinf(th.x))) pair_f64(x, y, z, q, slot, bs + j0, slow);
                        clear_x(o);
                    }
                    if (by) {
                        if (L.active && j0 + 1 < ns && (bs + j0 + 1 != slot || isinf(th.y)))
                            pair_f64(x, y, z, q, slot, bs + j0 + 1, slow);
                        clear_y(o);
                    }
                }
                A.put_phi(o.phi);
                if constexpr (F) A.put_field(o.w, o.d);
            }
            A.settle();
        }
    }
    int k;
    grid_exponent(lo, hi, k);
    double4 r = result(A, slow, k, q_exponent(*emax));
    const bool owner = L.combine(r, red);
    if (owner && part >= 0) {  // one segment of a split leaf: its partial sums
        partial[part + i] = r;
    } else if (owner) {
        const int64_t o = perm[slot];
        pot[o] = (OutT)(far_phi[slot] + r.x);
        if constexpr (F) {
            field[3 * o] = (OutT)(far_E[slot] + r.y);
            field[3 * o + 1] = (OutT)(far_E[n + slot] + r.z);
            field[3 * o + 2] = (OutT)(far_E[2 * n + slot] + r.w);
        }
    }
}

// ---------------------------------------------------------------------------
// The exact sum at selected targets (fmm_direct) in the same arithmetic. The
// sources are split once into records of two (kRec float4: parts a, b, c of x,
// y, z, q, then the thresholds; every lane of a warp reads the same record), a
// slab of them at a time; a block takes 128 targets against a segment of the
// slab and adds its sums to the (segment, target) slot; a last pass adds the
// segments. Everything outside the three floats' own sums (pairs left to FP64,
// those sums every kFlush records, slices, slabs, segments) is added in doubles
// with Neumaier's compensation: with one segment a target's sum runs over the
// whole slab (100,000 targets, all pairs left to FP64: off by 2.4e-15 of the terms without
// it). 500k points, 1000 targets (5e8 pairs): one block per target in FP64
// arithmetic (square root, two divisions and Neumaier sums a pair) 58.6 ms,
// this 5.00 (4.92 with plain sums; ~365 instead of ~295 operations a pair: 5.48);
// all pairs left to FP64 51.8; 1 target: 8.40 -> 0.36 ms, 2000 points and 1000
// targets 0.38 -> 0.08.
// ---------------------------------------------------------------------------
constexpr int kRec = 7;
constexpr int kFlush = 1024;  // records between flushes: three-float sums of 1000 terms lose less than 2^-55 of them, of 10^6 2^-51
constexpr int64_t kSlab = 1 << 20;  // sources split at a time (58 MB of records)

// the grid of the points: centre, 2^-k, whether it holds (grid_exponent), and the charges' exponent
struct Grid {
    double c[3], inv;
    int k, ok, eq;
    // a point's parts and its threshold on r^2
    __device__ __forceinline__ float split(double x, double y, double z, float (&f)[3][3]) const {
        bool exact = true;
        const bool fine = ok && isfinite(x) && isfinite(y) && isfinite(z);
        const double v[3] = {x, y, z};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            f[a][0] = f[a][1] = f[a][2] = 0.f;
            if (fine) exact &= grid_split(v[a], c[a], inv, f[a]);
        }
        return !fine ? __int_as_float(0x7f800000) : exact ? kThrExact : kThrRounded;
    }
};

struct DirectBox {  // the finite coordinates' range (order-preserving keys) and the largest charge's exponent
    unsigned long long lo[3], hi[3];
    int emax;
    unsigned blocks;  // blocks done
    Grid grid;        // from the last one
};

__global__ void k_direct_box_init(DirectBox *b) {
    const int a = threadIdx.x;
    if (a < 3) b->lo[a] = ~0ull, b->hi[a] = 0ull;
    if (a == 0) b->emax = 0, b->blocks = 0;
}

template <typename T>
__global__ void __launch_bounds__(256)
k_direct_box(const T *__restrict__ pts, const T *__restrict__ q, int64_t n, DirectBox *b) {
    unsigned long long lo[3], hi[3];
    int em = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) lo[a] = ~0ull, hi[a] = 0ull;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const double v = (double)pts[3 * i + a];
            if (!isfinite(v)) continue;
            const unsigned long long k = dkey(v);
            lo[a] = min(lo[a], k);
            hi[a] = max(hi[a], k);
        }
        const int e = (int)((__double_as_longlong((double)q[i]) >> 52) & 0x7ff);
        if (e < 0x7ff) em = max(em, e);
    }
    em = __reduce_max_sync(0xffffffffu, em);
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = min(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = max(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            atomicMin(&b->lo[a], lo[a]);
            atomicMax(&b->hi[a], hi[a]);
        }
        if (em > 0) atomicMax(&b->emax, em);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&b->blocks, 1u) == gridDim.x - 1) {  // every block's part is in
        __threadfence();
        double l[3], h[3];
        Grid G;
        for (int a = 0; a < 3; a++) {
            const unsigned long long kl = __ldcg(&b->lo[a]), kh = __ldcg(&b->hi[a]);
            l[a] = kh ? dkey_inv(kl) : 0.0;  // no finite coordinate: an empty range at 0
            h[a] = kh ? dkey_inv(kh) : 0.0;
            G.c[a] = 0.5 * l[a] + 0.5 * h[a];
        }
        G.ok = grid_exponent(l, h, G.k);
        G.inv = scalbn(1.0, -G.k);
        G.eq = q_exponent(__ldcg(&b->emax));
        b->grid = G;
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_direct_split(const T *__restrict__ pts, const T *__restrict__ q, int64_t n, int64_t j0, int64_t j1,
               const DirectBox *__restrict__ box, float4 *__restrict__ rec) {
    const Grid G = box->grid;
    const int64_t m = (j1 - j0 + 1) & ~(int64_t)1;  // the last record is padded
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        float f[3][3] = {{1.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, qf[3] = {0.f, 0.f, 0.f}, th = 0.f;
        const int64_t j = j0 + i;
        if (j < j1) {
            th = G.split((double)pts[3 * j], (double)pts[3 * j + 1], (double)pts[3 * j + 2], f);
            th = charge_split((double)q[j], G.eq, th, qf);
        }
        float *r = (float *)(rec + (i >> 1) * kRec) + (i & 1);
#pragma unroll
        for (int c = 0; c < 3; c++) {
#pragma unroll
            for (int a = 0; a < 3; a++) r[2 * (4 * c + a)] = -f[a][c];
            r[2 * (4 * c + 3)] = qf[c];
        }
        r[24] = th;
        r[26] = 0.f;
    }
}

// compensated sums of the potential and the field
struct Sum4 {
    double s[4], c[4];
    __device__ __forceinline__ void add(const Sum4 &o) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            neumaier(s[i], c[i], o.s[i]);
            c[i] += o.c[i];
        }
    }
    // (an infinite sum has no correction)
    __device__ __forceinline__ double get(int i) const { return isfinite(s[i]) ? s[i] + c[i] : s[i]; }
};

// source j on target i in FP64, pairs at zero distance skipped
template <typename T>
__device__ __noinline__ void direct_f64(const T *__restrict__ pts, const T *__restrict__ q, int64_t i, int64_t j,
                                        Sum4 &s) {
    const double dx = (double)pts[3 * i] - (double)pts[3 * j], dy = (double)pts[3 * i + 1] - (double)pts[3 * j + 1],
                 dz = (double)pts[3 * i + 2] - (double)pts[3 * j + 2];
    const double r2 = dx * dx + dy * dy + dz * dz;
    if (r2 == 0.0) return;
    const double r = sqrt(r2), qj = (double)q[j], qr3 = qj / (r2 * r);
    neumaier(s.s[0], s.c[0], qj / r);
    neumaier(s.s[1], s.c[1], qr3 * dx);
    neumaier(s.s[2], s.c[2], qr3 * dy);
    neumaier(s.s[3], s.c[3], qr3 * dz);
}

// A, sums of positions over 2^k and charges over 2^eq, added to S
__device__ __forceinline__ void flush(const tf::Sums<float2, true> &A, int k, int eq, Sum4 &S) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int e = i ? eq - 2 * k : eq - k;
        const double m = A.M[i > 0];
        neumaier(S.s[i], S.c[i], scalbn(((double)A.a[i].x + (double)A.a[i].y) +
                                            ((((double)A.s[i].x - m) + ((double)A.s[i].y - m)) +
                                             ((double)A.c[i].x + (double)A.c[i].y)), e));
    }
}

// block (x: targets 128 x .., y: records [y len, (y + 1) len) of the slab)
template <typename T>
__global__ void __launch_bounds__(kT, 4)
k_direct_tf(const T *__restrict__ pts, const T *__restrict__ q, int64_t n, const int64_t *__restrict__ targets,
            int64_t nt, int64_t j0, int64_t j1, const DirectBox *__restrict__ box, const float4 *__restrict__ rec,
            int64_t len, bool first, Sum4 *__restrict__ partial) {
    __shared__ Sum4 red[kT];
    const int64_t t0 = (int64_t)blockIdx.x * kT;
    const P2PLane L((int)min((int64_t)kT, nt - t0), kT, threadIdx.x);
    const int64_t i = L.active ? targets[t0 + L.target] : -1;
    const bool on = i >= 0 && i < n;  // an index out of range: no access (the last pass writes NaN)
    const bool busy = __any_sync(0xffffffffu, on);
    float f[3][3] = {}, thr_i = 0.f;
    if (on) thr_i = box->grid.split((double)pts[3 * i], (double)pts[3 * i + 1], (double)pts[3 * i + 2], f);
    tf::Tri<float2> X[3];
#pragma unroll
    for (int a = 0; a < 3; a++)
        X[a] = {make_float2(f[a][0], f[a][0]), make_float2(f[a][1], f[a][1]), make_float2(f[a][2], f[a][2])};
    Sum4 S = {};
    const int64_t np = (j1 - j0 + 1) >> 1, p1 = busy ? min(np, (blockIdx.y + 1) * len) : 0;
#pragma unroll 1
    for (int64_t pp = blockIdx.y * len + L.slice; pp < p1;) {
        tf::Sums<float2, true> A(make_float2(0.f, 0.f));
        const int64_t end = min(p1, pp + kFlush * L.slices);
#pragma unroll 1
        for (int terms = 1; pp < end; pp += L.slices, terms++) {
            const float4 *r = rec + pp * kRec;
            const float4 a0 = __ldg(r), a1 = __ldg(r + 1), b0 = __ldg(r + 2), b1 = __ldg(r + 3), c0 = __ldg(r + 4),
                         c1 = __ldg(r + 5), th = __ldg(r + 6);
            const tf::Tri<float2> Y[3] = {{make_float2(a0.x, a0.y), make_float2(b0.x, b0.y), make_float2(c0.x, c0.y)},
                                          {make_float2(a0.z, a0.w), make_float2(b0.z, b0.w), make_float2(c0.z, c0.w)},
                                          {make_float2(a1.x, a1.y), make_float2(b1.x, b1.y), make_float2(c1.x, c1.y)}};
            const tf::Tri<float2> Q = {make_float2(a1.z, a1.w), make_float2(b1.z, b1.w), make_float2(c1.z, c1.w)};
            tf::PairTerms<float2> o = tf::pair_terms(X, Y, Q);
            const bool bx = o.r2.x < fmaxf(th.x, thr_i), by = o.r2.y < fmaxf(th.y, thr_i);
            if (bx || by) {
                const int64_t j = j0 + 2 * pp;
                if (bx) {
                    if (on && (j != i || isinf(th.x))) direct_f64(pts, q, i, j, S);
                    clear_x(o);
                }
                if (by) {
                    if (on && j + 1 < j1 && (j + 1 != i || isinf(th.y))) direct_f64(pts, q, i, j + 1, S);
                    clear_y(o);
                }
            }
            A.put_phi(o.phi);
            A.put_field(o.w, o.d);
            if ((terms & 31) == 0) A.settle();
        }
        A.settle();
        flush(A, box->grid.k, box->grid.eq, S);
    }
    if (L.combine(S, red, [](Sum4 &a, const Sum4 &o) { a.add(o); })) {
        Sum4 *slot = partial + blockIdx.y * nt + t0 + L.target;
        if (!first) S.add(*slot);
        *slot = S;
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_direct_finish(int64_t n, const int64_t *__restrict__ targets, int64_t nt, int64_t segs,
                const Sum4 *__restrict__ partial, T *__restrict__ pot, T *__restrict__ field) {
    // a warp per target, the lanes over the segments
    const int lane = threadIdx.x & 31;
    for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; t < nt;
         t += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        Sum4 r = {};
        for (int64_t s = lane; s < segs; s += 32) r.add(partial[s * nt + t]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            Sum4 v;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                v.s[i] = __shfl_xor_sync(0xffffffffu, r.s[i], o);
                v.c[i] = __shfl_xor_sync(0xffffffffu, r.c[i], o);
            }
            r.add(v);
        }
        if (lane) continue;
        const int64_t i = targets[t];
        const bool ok = i >= 0 && i < n;
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        pot[t] = (T)(ok ? r.get(0) : nan);
        if (field)
#pragma unroll
            for (int a = 0; a < 3; a++) field[3 * t + a] = (T)(ok ? r.get(1 + a) : nan);
    }
}

unsigned grid_for(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 8); }

}  // namespace

cudaError_t tf_setup(Plan &P) {
    const size_t n = (size_t)P.n;
    P.tf_pos = (float *)palloc(P, n * 36);
    P.tf_q = (float *)palloc(P, n * 12);
    P.tf_thr0 = (float *)palloc(P, n * 4);
    P.tf_thr = (float *)palloc(P, n * 4);
    P.tf_emax = (int *)palloc(P, 4);
    if (!P.tf_pos || !P.tf_q || !P.tf_thr0 || !P.tf_thr || !P.tf_emax) return cudaErrorMemoryAllocation;
    FMM_LAUNCH(k_tf_points, grid_for(P.n), 256, 0, P.stream, P.n, P.x, P.y, P.z, P.lo, P.hi, P.tf_pos, P.tf_thr0);
    return cudaGetLastError();
}

cudaError_t tf_p2p(Plan &P, void *pot, void *field, int dtype) {
    cudaMemsetAsync(P.tf_emax, 0, 4, P.stream);
    FMM_LAUNCH(k_tf_qmax, grid_for(P.n), 256, 0, P.stream, P.n, P.q, P.tf_emax);
    FMM_LAUNCH(k_tf_charges, grid_for(P.n), 256, 0, P.stream, P.n, P.q, P.tf_emax, P.tf_thr0, P.tf_q, P.tf_thr);
    auto go = [&](auto out, auto fld) {  // without a field array only the potential is summed
        using Out = decltype(out);
        FMM_LAUNCH((k_p2p_tf<Out, decltype(fld)::value>), (unsigned)P.p2p_nunits, kP2PTileTf, 0, P.stream, P.B, P.n, P.x, P.y,
                   P.z, P.q, P.tf_pos, P.tf_q, P.tf_thr0, P.tf_thr, P.lo, P.hi, P.tf_emax, P.begin, P.count,
                   P.ssrc[P.B], P.p2p_units, P.p2p_upart, P.p2p_nunits_dev, P.perm, P.far_phi, P.far_E,
                   P.p2p_partial, (Out *)pot, (Out *)field);
    };
    if (dtype == FMM_F64)
        field ? go(double{}, std::true_type{}) : go(double{}, std::false_type{});
    else
        field ? go(float{}, std::true_type{}) : go(float{}, std::false_type{});
    return cudaGetLastError();
}

template <typename T>
static cudaError_t direct_tf_run(const T *pts, const T *q, int64_t n, const int64_t *targets, int64_t nt, T *pot,
                                 T *field, cudaStream_t st) {
    // segments: enough blocks for about four waves of four per SM, 64 records at least
    const int64_t slab = std::min(n, kSlab), recs = (slab + 1) / 2, tiles = (nt + kT - 1) / kT;
    const int64_t want = std::max<int64_t>(1, 16 * (int64_t)sm_count() / tiles);
    const int64_t len = std::max<int64_t>(64, (recs + want - 1) / want);
    const int64_t segs = std::min<int64_t>((recs + len - 1) / len, 65535), len1 = (recs + segs - 1) / segs;
    const size_t b0 = 512, b1 = (size_t)recs * kRec * 16, b2 = (size_t)segs * nt * sizeof(Sum4);
    char *w = (char *)pool_alloc(b0 + ((b1 + 255) & ~(size_t)255) + b2, st);
    if (!w) return cudaErrorMemoryAllocation;
    DirectBox *box = (DirectBox *)w;
    float4 *rec = (float4 *)(w + b0);
    Sum4 *partial = (Sum4 *)(w + b0 + ((b1 + 255) & ~(size_t)255));
    FMM_LAUNCH(k_direct_box_init, 1, 32, 0, st, box);
    FMM_LAUNCH(k_direct_box<T>, grid_for(n), 256, 0, st, pts, q, n, box);
    for (int64_t j0 = 0; j0 < n; j0 += kSlab) {
        const int64_t j1 = std::min(n, j0 + kSlab);
        FMM_LAUNCH(k_direct_split<T>, grid_for(j1 - j0), 256, 0, st, pts, q, n, j0, j1, box, rec);
        FMM_LAUNCH(k_direct_tf<T>, dim3((unsigned)tiles, (unsigned)segs), kT, 0, st, pts, q, n, targets, nt, j0, j1,
                   box, rec, len1, j0 == 0, partial);
    }
    FMM_LAUNCH(k_direct_finish<T>, grid_for(nt * 32), 256, 0, st, n, targets, nt, segs, partial, pot, field);
    const cudaError_t e = cudaGetLastError();
    pool_free(w, st);
    return e;
}

// the exact sum; cudaErrorMemoryAllocation if its workspace cannot be had (nothing was launched then)
cudaError_t direct_tf(const void *pts, const void *q, int64_t n, int dtype, const int64_t *targets, int64_t nt,
                      void *pot, void *field, cudaStream_t st) {
    if (dtype == FMM_F64)
        return direct_tf_run((const double *)pts, (const double *)q, n, targets, nt, (double *)pot, (double *)field, st);
    return direct_tf_run((const float *)pts, (const float *)q, n, targets, nt, (float *)pot, (float *)field, st);
}

}  // namespace fmm
