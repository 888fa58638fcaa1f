"""The three-float arithmetic of csrc/trifloat.cuh, compiled for the host, against
quadruple precision at the bounds that its header states: pair terms within 2^-61
(potential) and 2^-58 (field) at positions exact on the grid, with the reciprocal
square root off by up to 1.5e-7 as the hardware's may be; sums of 40,000 terms within
2^-53 of the terms' absolute sum, sums of 1,000 within 2^-55."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_04894_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
static float g_err = 1.f;
#define TF_RSQRT_ERR g_err
#include "trifloat.cuh"
using namespace fmm::tf;
#ifdef __SIZEOF_FLOAT128__
typedef __float128 Q;
#else
typedef long double Q;  // 128 bits on this machine
#endif
static std::mt19937_64 R(1);
static double U() { return (double)(R() >> 11) * 0x1p-53 - 0.5; }
static Q qabs(Q v) { return v < 0 ? -v : v; }
static Q qsqrt(Q v) {
    Q s = std::sqrt((double)v);
    for (int i = 0; i < 2; i++) s = (s + v / s) / 2;
    return s;
}
static double lg(Q v) { return std::log2((double)v); }
static bool split(double u, Tri<float> &t) {
    volatile double a = u + 0x1.8p28, b, c;
    const double x1 = a - 0x1.8p28, r = u - x1;
    b = r + 0x1.8p4;
    const double x2 = b - 0x1.8p4, s = r - x2;
    c = s + 0x1.8p-20;
    const double x3 = c - 0x1.8p-20;
    t = {(float)x1, (float)x2, (float)x3};
    return s == x3;
}
struct Pair {
    Tri<float> X[3], Y[3], q;
    Q phi, f[3];
    bool make(const double *x, const double *y, double charge) {
        bool ok = true;
        Q d[3], r2 = 0;
        for (int i = 0; i < 3; i++) {
            ok &= split(x[i], X[i]) & split(y[i], Y[i]);
            Y[i] = {-Y[i].a, -Y[i].b, -Y[i].c};
            d[i] = (Q)x[i] - (Q)y[i];
            r2 += d[i] * d[i];
        }
        const float a = (float)charge, b = (float)(charge - a);
        q = {a, b, (float)((charge - a) - b)};
        if (!ok || (double)r2 < 0x1p-46) return false;
        phi = (Q)charge / qsqrt(r2);
        for (int i = 0; i < 3; i++) f[i] = phi / r2 * d[i];
        g_err = 1.f + (float)(U() * 3e-7);
        return true;
    }
};
static Q val(const Tri<float> &t) { return (Q)t.a + t.b + t.c; }
static void pairs(double scale, int n) {
    Q mp = 0, mf = 0;
    int used = 0;
    for (int k = 0; k < n; k++) {
        double x[3], y[3];
        for (int i = 0; i < 3; i++) {
            x[i] = U() * .99;
            y[i] = x[i] + U() * scale;
            if (std::fabs(y[i]) > .5) y[i] = x[i] * .999;
        }
        Pair P;
        if (!P.make(x, y, U())) continue;
        used++;
        const auto o = pair_terms<float>(P.X, P.Y, P.q);
        const auto o1 = pair_terms<float, false>(P.X, P.Y, P.q);  // without the field: the same potential
        if (o1.phi.a != o.phi.a || o1.phi.b != o.phi.b || o1.phi.c != o.phi.c) mp = 1;
        Q e = qabs((val(o.phi) - P.phi) / P.phi), en = 0, nn = 0;
        if (e > mp) mp = e;
        for (int i = 0; i < 3; i++) {
            const Q d = P.f[i] - val(o.w) * val(o.d[i]);
            en += d * d;
            nn += P.f[i] * P.f[i];
        }
        e = qsqrt(en / nn);
        if (e > mf) mf = e;
    }
    std::printf("pairs %d %.2f %.2f\n", used, lg(mp), lg(mf));
}
template <bool F>
static void sums(int n, double scale, bool positive) {
    double x[3] = {U() * .5, U() * .5, U() * .5};
    Sums<float, F> A(0.f);
    Q S[4] = {}, ab[4] = {};
    for (int k = 1; k <= n; k++) {
        double y[3];
        const double s = scale < 1 ? scale * std::pow(10., 3 * U()) : 1;
        for (int i = 0; i < 3; i++) {
            y[i] = scale < 1 ? x[i] + U() * s : U();
            if (std::fabs(y[i]) > .5) y[i] = U();
        }
        Pair P;
        const double c = U();
        if (!P.make(x, y, positive ? std::fabs(c) : c)) continue;
        S[0] += P.phi, ab[0] += qabs(P.phi);
        for (int i = 0; i < 3; i++) S[1 + i] += P.f[i], ab[1 + i] += qabs(P.f[i]);
        const auto o = pair_terms<float, F>(P.X, P.Y, P.q);
        A.put_phi(o.phi);
        if constexpr (F) A.put_field(o.w, o.d);
        if ((k & 31) == 0) A.settle();
    }
    A.settle();
    Q m = 0;
    for (int i = 0; i < (F ? 4 : 1); i++) {
        const Q e = qabs((Q)A.a[i] + ((Q)A.s[i] - A.M[i > 0]) + A.c[i] - S[i]) / ab[i];
        if (e > m) m = e;
    }
    std::printf("sums %d %.2f\n", n, lg(m));
}
int main() {
    for (double s : {1., 1e-1, 1e-2, 1e-3, 1e-4, 1e-5, 2.5e-6, 3e-7}) pairs(s, 10000);
    for (double s : {1., 1e-1, 1e-3}) {
        sums<true>(40000, s, true);
        sums<true>(1000, s, true);
        sums<true>(1000, s, false);
        sums<false>(1000, s, true);
    }
}
"""


def test_three_float_arithmetic_holds_its_bounds(tmp_path):
    src, exe = tmp_path / "tf.cpp", tmp_path / "tf"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=300).stdout
    rows = [line.split() for line in out.splitlines()]
    pairs = [r for r in rows if r[0] == "pairs"]
    sums = [r for r in rows if r[0] == "sums"]
    assert len(pairs) == 8 and len(sums) == 12
    for _, used, phi, field in pairs:
        assert int(used) > 5000
        assert float(phi) <= -61 and float(field) <= -58, out
    for _, n, err in sums:
        assert float(err) <= (-53 if int(n) > 1000 else -55), out
