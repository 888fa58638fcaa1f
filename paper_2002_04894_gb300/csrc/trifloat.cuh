// Pair interactions of double accuracy in single-precision arithmetic.
//
// GB300 retires 128 FP32 operations per clock and SM, but fewer than two FP64
// ones, so an FP64 pair (19 FP64 instructions) costs as much as ~1,400 FP32
// operations. Here a pair takes about 295: every quantity is an unevaluated
// sum of three floats (~72 bits), built from error-free transformations
// (Knuth's TwoSum, Dekker's FastTwoSum, the product's rounding error from the
// fused multiply-add). Terms of the same size are summed exactly by a
// FastTwoSum chain that starts from a constant M larger than all of them; M
// comes off exactly at the end. Every operation is an explicitly rounded
// intrinsic on packed pairs (two sources at once); signs are flipped on the
// ALU pipe.
//
// A pair whose positions are exact on the common grid has relative errors of
// at most 2^-61 (potential) and 2^-58 (field) over 1.6 million random pairs at
// distances from 1 to 1e-7 of the grid's extent (double arithmetic: 2^-51 and
// 2^-50); close pairs of rounded positions are left to FP64 (p2p_tf.cu). The
// host branch below is for tests/test_trifloat_cpu.py, which holds these bounds.
#pragma once

#ifndef __CUDACC__
#include <cmath>
#endif

namespace fmm {
namespace tf {

// ---- the arithmetic: V is float2 (device, two pairs) or float (host check)
#ifdef __CUDACC__
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 cst(float2, float c) { return make_float2(c, c); }
__device__ __forceinline__ float rsqrt1(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// by the sign bits: the ALU pipe has room, the FMA pipe has none
__device__ __forceinline__ float2 neg(float2 a) {
    return make_float2(__int_as_float(__float_as_int(a.x) ^ 0x80000000), __int_as_float(__float_as_int(a.y) ^ 0x80000000));
}
__device__ __forceinline__ float amax(float2 x) { return fmaxf(fabsf(x.x), fabsf(x.y)); }
__device__ __forceinline__ float2 rsqrt0(float2 x) { return make_float2(rsqrt1(x.x), rsqrt1(x.y)); }
#define TF_DEV __device__ __forceinline__
#else
inline float add(float a, float b) { return a + b; }
inline float mul(float a, float b) { return a * b; }
inline float fma(float a, float b, float c) { return fmaf(a, b, c); }
inline float sub(float a, float b) { return a - b; }
inline float cst(float, float c) { return c; }
inline float neg(float a) { return -a; }
inline float amax(float x) { return fabsf(x); }
inline float rsqrt0(float x) { return 1.f / sqrtf(x) * TF_RSQRT_ERR; }
#define TF_DEV inline
#endif

template <class V>
struct Tri {
    V a, b, c;  // a + b + c
};

// (By a compare and selects on the ALU pipe and a FastTwoSum instead: the near
// field of 200k points took 128.2 ms against 124.5.)
template <class V>
TF_DEV V two_sum(V a, V b, V &e) {
    const V s = add(a, b), bb = sub(s, a);
    e = add(sub(a, sub(s, bb)), sub(b, bb));
    return s;
}

// Exact sum of terms no larger than M: s holds M + their parts on the grid of
// M's last place, t the (small) parts below it.
template <class V>
struct Sum {
    V M, s, t;
    TF_DEV Sum(V m, V first) : M(m), t(cst(m, 0.f)) { put0(first, true); }
    TF_DEV void put0(V w, bool set) {
        const V n = set ? add(M, w) : add(s, w), r = add(w, sub(set ? M : s, n));
        t = set ? r : add(t, r);
        s = n;
    }
    TF_DEV void put(V w) { put0(w, false); }  // + w
    TF_DEV void take(V w) {                    // - w
        const V n = sub(s, w), r = sub(sub(s, n), w);
        t = add(t, r);
        s = n;
    }
    TF_DEV void put2(V w) {  // + 2 w
        const V two = cst(w, 2.f), n = fma(w, two, s), r = fma(w, two, sub(s, n));
        t = add(t, r);
        s = n;
    }
    TF_DEV V top() const { return sub(s, M); }
};

// d = x + y for grid positions x and (negated) y, component by component
// exact, then (h, l, t) with h the rounded sum
template <class V>
TF_DEV Tri<V> diff(const Tri<V> &x, const Tri<V> &ny) {
    const V a = add(x.a, ny.a), b = add(x.b, ny.b), c = add(x.c, ny.c);
    const V h = add(a, b), l0 = add(sub(a, h), b), l = add(l0, c);
    return {h, l, add(sub(l0, l), c)};
}

// The terms of the product of A and B below A.a B.a: w holds their sum to
// ~2^-46 of M, t the rest. nA = -A.a, nAb = -A.b; M larger than 2^-22 |A B|.
template <class V>
TF_DEV Tri<V> product(const Tri<V> &A, V nA, V nAb, const Tri<V> &B, V p, V M) {
    const V np = fma(nA, B.a, p);  // p - A.a B.a
    const V m1 = mul(A.a, B.b), n1 = fma(nA, B.b, m1), m2 = mul(A.b, B.a), n2 = fma(nAb, B.a, m2);
    Sum<V> S(M, m1);
    S.put(m2);
    S.take(np);
    V t = sub(sub(S.t, n1), n2);
    t = fma(A.a, B.c, t);
    t = fma(A.b, B.b, t);
    t = fma(A.c, B.a, t);
    return {p, S.top(), t};
}

// One pair (two in packed form) for target x, source y (coordinates negated)
// and its charge: the squared distance's leading part, q / r, W = q / r^3 and
// d = x - y (the field is W d).
template <class V>
struct PairTerms {
    V r2;  // leading part of the squared distance
    Tri<V> phi, w, d[3];
};

template <class V, bool F = true>  // F: with the field
TF_DEV PairTerms<V> pair_terms(const Tri<V> (&x)[3], const Tri<V> (&ny)[3], const Tri<V> &q) {
    PairTerms<V> o;
    const Tri<V> (&d)[3] = o.d;
#pragma unroll
    for (int i = 0; i < 3; i++) o.d[i] = diff(x[i], ny[i]);
    const V nh[3] = {neg(d[0].a), neg(d[1].a), neg(d[2].a)};
    // r2 = P + R2 + R3
    V P, R2, R3;
    {
        V p[3], np[3], u[3], nu[3];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            p[i] = mul(d[i].a, d[i].a);
            np[i] = fma(nh[i], d[i].a, p[i]);  // p - h^2
            u[i] = mul(d[i].a, d[i].b);
            nu[i] = fma(nh[i], d[i].b, u[i]);  // u - h l
        }
        V e1, e2;
        P = two_sum(two_sum(p[0], p[1], e1), p[2], e2);
        Sum<V> S(mul(P, cst(P, 0x1p-18f)), e1);
        S.put(e2);
#pragma unroll
        for (int i = 0; i < 3; i++) S.take(np[i]);
#pragma unroll
        for (int i = 0; i < 3; i++) S.put2(u[i]);
        R2 = S.top();
        V tau = mul(d[0].a, d[0].c), t = S.t;
        tau = fma(d[1].a, d[1].c, tau);
        tau = fma(d[2].a, d[2].c, tau);
#pragma unroll
        for (int i = 0; i < 3; i++) {
            tau = sub(tau, nu[i]);
            t = fma(d[i].b, d[i].b, t);
        }
        R3 = fma(tau, cst(tau, 2.f), t);
    }
    o.r2 = P;
    // The hardware's y0 ~ 1 / r and z, y0^2 rounded: with e = 1 - r2 z and
    // E = 1 - r2 y0^2, both exact to ~2^-54,
    //   1 / r = Y = y0 (1 + E / 2 + 3 E^2 / 8),  1 / r^2 = Z = z (1 + e + e^2)
    const V y0 = rsqrt0(P), n0 = neg(y0), z = mul(y0, y0), nze = fma(n0, y0, z), nz = neg(z);  // nze = z - y0^2
    Tri<V> Y, Z;
    V nf;
    {
        const V nP = neg(P), g = mul(P, z), nge = fma(nP, z, g), f1 = sub(cst(g, 1.f), g);
        const V rz = mul(R2, z), nre = fma(R3, nz, fma(R2, nz, rz));
        Sum<V> S(cst(g, 0x1p-18f), f1);
        S.put(nge);
        S.take(rz);
        if constexpr (F) {
            const V e1 = S.top(), f = mul(z, e1);
            Z = {z, f, fma(z, fma(e1, e1, add(S.t, nre)), fma(z, e1, neg(f)))};
        }
        const V pz = mul(P, nze), npe = fma(nP, nze, pz);  // E = e + r2 (z - y0^2)
        S.put(pz);
        const V t = fma(R2, nze, sub(add(S.t, nre), npe));
        const V E1 = S.top(), yh = mul(y0, cst(y0, 0.5f)), c2 = fma(mul(E1, cst(E1, 0.75f)), E1, t);
        const V f = mul(yh, E1);
        nf = neg(f);
        Y = {y0, f, fma(yh, c2, fma(yh, E1, nf))};
    }
    // q / r
    {
        const V p = mul(Y.a, q.a);
        o.phi = product(Y, n0, nf, q, p, mul(p, cst(p, 0x1p-18f)));
    }
    if constexpr (!F) return o;
    const V w0 = mul(Z.a, o.phi.a);
    o.w = product(Z, nz, neg(Z.b), o.phi, w0, mul(w0, cst(w0, 0x1p-18f)));
    return o;
}

// The running sums of a target: potential (0) and field (1..3). a takes the
// terms' leading parts by TwoSums; what is below goes to s, which runs about a
// constant M far above it and far below the terms (2^-14 of `lim`, itself 1 to 4
// times the largest term or sum so far), so that three operations add a part
// and give its rounding error; c takes those. A term's product is not rounded
// to three floats first: its parts go straight into the sums. Per addition
// ~2^-58 of the sum is lost (double arithmetic: 2^-54). `settle` after at most
// 32 terms keeps s near M. (With TwoSums for s as well and the field's products
// rounded to three floats first, ~365 operations a pair: 200k points 124.5 ms,
// 110.7 this way.) Sums of 40,000 terms: 2^-53 of the terms' absolute sum at
// worst, double arithmetic 2^-47.
template <class V, bool F>
struct Sums {
    static constexpr int N = F ? 4 : 1;
    V a[N], s[N], c[N];
    float M[2], lim[2];  // of the potential, of the field
    TF_DEV Sums(V like) {
#pragma unroll
        for (int i = 0; i < N; i++) a[i] = s[i] = c[i] = cst(like, 0.f);
        M[0] = M[1] = lim[0] = lim[1] = 0.f;
    }
    TF_DEV V put(int i, V w) {  // s += w; the rounding error
        const V n = add(s[i], w), r = add(w, sub(s[i], n));
        s[i] = n;
        return r;
    }
    // terms up to m to come in group g: sums i0 <= i < i1
    TF_DEV void fit(int g, int i0, int i1, float m) {
        if (!(m > lim[g])) return;
        lim[g] = 4.f * m;
        const float M2 = lim[g] * 0x1p-14f;
#pragma unroll
        for (int i = i0; i < i1; i++) {
            const V b = sub(s[i], cst(s[i], M[g])), n = add(cst(b, M2), b);
            c[i] = add(c[i], sub(b, sub(n, cst(b, M2))));
            s[i] = n;
        }
        M[g] = M2;
    }
    TF_DEV void put_phi(const Tri<V> &x) {
        fit(0, 0, 1, fmaxf(amax(x.a), amax(a[0])));
        V e;
        a[0] = two_sum(a[0], x.a, e);
        const V r = add(put(0, x.b), put(0, e));
        c[0] = add(c[0], add(r, x.c));
    }
    TF_DEV void put_field(const Tri<V> &W, const Tri<V> (&d)[3]) {
        const V nW = neg(W.a), nWb = neg(W.b);
        V p[3];
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            p[i] = mul(W.a, d[i].a);
            m = fmaxf(m, fmaxf(amax(p[i]), amax(a[1 + i])));
        }
        fit(1, 1, 4, m);
#pragma unroll
        for (int i = 0; i < 3; i++) {
            V e;
            a[1 + i] = two_sum(a[1 + i], p[i], e);
            const V m1 = mul(W.a, d[i].b), n1 = fma(nW, d[i].b, m1), m2 = mul(W.b, d[i].a), n2 = fma(nWb, d[i].a, m2);
            const V pe = fma(W.a, d[i].a, neg(p[i]));
            V t = add(put(1 + i, m1), put(1 + i, m2));
            t = add(t, add(put(1 + i, pe), put(1 + i, e)));
            t = sub(sub(t, n1), n2);
            t = fma(W.a, d[i].c, t);
            t = fma(W.b, d[i].b, t);
            t = fma(W.c, d[i].a, t);
            c[1 + i] = add(c[1 + i], t);
        }
    }
    TF_DEV void settle() {
#pragma unroll
        for (int i = 0; i < N; i++) {
            const V m = cst(s[i], M[i > 0]);
            V e;
            a[i] = two_sum(a[i], sub(s[i], m), e);
            s[i] = m;
            const V r = add(c[i], put(i, e)), n = add(s[i], r);
            c[i] = sub(r, sub(n, s[i]));
            s[i] = n;
        }
    }
};

}  // namespace tf
}  // namespace fmm
