// Pair interactions of double accuracy in single-precision arithmetic.
//
// GB300 retires 128 FP32 operations per clock and SM, but fewer than two FP64
// ones, so an FP64 pair (19 FP64 instructions) costs as much as ~1,400 FP32
// operations. Here a pair takes about 360: every quantity is an unevaluated
// sum of three floats (~72 bits), built from error-free transformations
// (Knuth's TwoSum, Dekker's FastTwoSum, the product's rounding error from the
// fused multiply-add). Terms of the same size are summed exactly by a
// FastTwoSum chain that starts from a constant M larger than all of them; M
// comes off exactly at the end. Every operation is an explicitly rounded
// intrinsic on packed pairs (two sources at once).
//
// A pair whose positions are exact on the common grid has relative errors of
// at most 2^-61 (potential) and 2^-58 (field) over 1.6 million random pairs at
// distances from 1 to 1e-7 of the grid's extent (double arithmetic: 2^-51 and
// 2^-50); close pairs of rounded positions are left to FP64 (p2p_tf.cu).
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
__device__ __forceinline__ float2 rsqrt0(float2 x) { return make_float2(rsqrt1(x.x), rsqrt1(x.y)); }
#define TF_DEV __device__ __forceinline__
#else
inline float add(float a, float b) { return a + b; }
inline float mul(float a, float b) { return a * b; }
inline float fma(float a, float b, float c) { return fmaf(a, b, c); }
inline float sub(float a, float b) { return a - b; }
inline float cst(float, float c) { return c; }
inline float rsqrt0(float x) { return 1.f / sqrtf(x) * TF_RSQRT_ERR; }
#define TF_DEV inline
#endif

template <class V>
struct Tri {
    V a, b, c;  // a + b + c
};

template <class V>
TF_DEV V neg(V a) { return mul(a, cst(a, -1.f)); }
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

// running sum of three-float terms: TwoSums on the first two parts
template <class V>
struct Acc {
    V a, b, c;
    TF_DEV void put(const Tri<V> &x) {
        V e1, e2, e3;
        a = two_sum(a, x.a, e1);
        b = two_sum(b, x.b, e2);
        b = two_sum(b, e1, e3);
        c = add(c, add(add(e2, e3), x.c));
    }
};

// One pair (two in packed form): the squared distance's leading part, q / r
// and q d / r^3 for target x, source y (coordinates negated) and its charge.
template <class V>
struct PairTerms {
    V r2;  // leading part of the squared distance
    Tri<V> phi, e[3];
};

template <class V, bool F = true>  // F: with the field
TF_DEV PairTerms<V> pair_terms(const Tri<V> (&x)[3], const Tri<V> (&ny)[3], const Tri<V> &q) {
    PairTerms<V> o;
    const Tri<V> d[3] = {diff(x[0], ny[0]), diff(x[1], ny[1]), diff(x[2], ny[2])};
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
    // 1 / r = Y: a Newton-like step on the hardware's y0 with the residual
    // e = 1 - r2 y0^2 exact to ~2^-54: y0 (1 + e / 2 + 3 e^2 / 8)
    const V y0 = rsqrt0(P), n0 = neg(y0), z = mul(y0, y0), nze = fma(n0, y0, z), nz = neg(z);  // nze = z - y0^2
    Tri<V> Y;
    V nf;
    {
        const V nP = neg(P), g = mul(P, z), nge = fma(nP, z, g), f1 = sub(cst(g, 1.f), g);
        const V pz = mul(P, nze), npe = fma(nP, nze, pz), rz = mul(R2, z), nre = fma(R2, nz, rz);
        Sum<V> S(cst(g, 0x1p-18f), f1);
        S.put(nge);
        S.put(pz);
        S.take(rz);
        V t = sub(add(S.t, nre), npe);
        t = fma(R2, nze, t);
        t = fma(R3, nz, t);
        const V E1 = S.top(), c1 = mul(E1, cst(E1, 0.5f)), q1 = mul(E1, cst(E1, 0.375f)),
                c2 = fma(q1, E1, mul(t, cst(t, 0.5f)));
        const V f = mul(y0, c1), nfe = fma(n0, c1, f);
        Y = {y0, f, sub(mul(y0, c2), nfe)};
        nf = neg(f);
    }
    // q / r
    {
        const V p = mul(Y.a, q.a);
        o.phi = product(Y, n0, nf, q, p, mul(p, cst(p, 0x1p-18f)));
    }
    if constexpr (!F) return o;
    // 1 / r^2 = Z
    Tri<V> Z;
    {
        const V m = mul(y0, Y.b), nm = fma(n0, Y.b, m);
        Sum<V> S(mul(z, cst(z, 0x1p-18f)), mul(m, cst(m, 2.f)));
        S.take(nze);
        V t = fma(nm, cst(nm, -2.f), S.t);
        t = fma(mul(y0, Y.c), cst(t, 2.f), t);
        t = fma(Y.b, Y.b, t);
        // z - nze = y0^2
        Z = {z, S.top(), t};
    }
    // W = q / r^3, then W d
    const V w0 = mul(Z.a, o.phi.a);
    const Tri<V> W = product(Z, nz, neg(Z.b), o.phi, w0, mul(w0, cst(w0, 0x1p-18f)));
    const V nW = neg(W.a), nWb = neg(W.b), M = mul(W.a, mul(P, mul(y0, cst(y0, 0x1p-18f))));  // 2^-18 |W| r
#pragma unroll
    for (int i = 0; i < 3; i++) o.e[i] = product(W, nW, nWb, d[i], mul(W.a, d[i].a), M);
    return o;
}

}  // namespace tf
}  // namespace fmm
