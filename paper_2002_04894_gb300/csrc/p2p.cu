// The exact sum of Eq. 2.1 at selected targets, and the end of the near field
// (P2P, Algorithm 4): its launch by precision form (p2p_tf.cu, mixed.cu; one
// block per work unit, a tile of a target leaf's points against a segment of
// its strong list, the far field added and the results written in input
// order) and the pass that adds the partial sums of leaves whose strong list
// was cut into segments, in segment order.
//
// Direct: p2p_tf.cu; where its workspace cannot be had, one CTA per target in
// FP64, threads striding over all sources with Neumaier-compensated partial
// sums, then a block reduction.

#include <algorithm>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

template <typename T>
__global__ void __launch_bounds__(256)
k_direct(const T *__restrict__ pts, const T *__restrict__ q, int64_t n,
         const int64_t *__restrict__ targets, T *__restrict__ pot, T *__restrict__ field) {
    __shared__ double red[4][256];
    const int64_t i = targets[blockIdx.x];
    if (i < 0 || i >= n) {  // out-of-range index: NaN outputs, no access
        if (threadIdx.x < 4) {
            const T nan = (T)__longlong_as_double(0x7ff8000000000000ll);
            if (threadIdx.x == 0)
                pot[blockIdx.x] = nan;
            else if (field)
                field[3 * blockIdx.x + threadIdx.x - 1] = nan;
        }
        return;
    }
    const double xi = (double)pts[3 * i], yi = (double)pts[3 * i + 1], zi = (double)pts[3 * i + 2];
    double s[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0};
    for (int64_t j = threadIdx.x; j < n; j += 256) {
        const double dx = xi - (double)pts[3 * j], dy = yi - (double)pts[3 * j + 1],
                     dz = zi - (double)pts[3 * j + 2];
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (r2 == 0.0) continue;
        const double r = sqrt(r2);
        const double qj = (double)q[j];
        const double qr3 = qj / (r2 * r);
        neumaier(s[0], c[0], qj / r);
        neumaier(s[1], c[1], qr3 * dx);
        neumaier(s[2], c[2], qr3 * dy);
        neumaier(s[3], c[3], qr3 * dz);
    }
    for (int a = 0; a < 4; a++) red[a][threadIdx.x] = s[a] + c[a];
    __syncthreads();
    if (threadIdx.x < 4) {
        double ss = 0.0, cc = 0.0;
        for (int j = 0; j < 256; j++) neumaier(ss, cc, red[threadIdx.x][j]);
        const double v = ss + cc;
        if (threadIdx.x == 0)
            pot[blockIdx.x] = (T)v;
        else if (field)
            field[3 * blockIdx.x + threadIdx.x - 1] = (T)v;
    }
}

// Finishes the leaves whose strong list was cut into segments: per target,
// the segments' partial sums added in segment order, then the far field;
// outputs in input order. Leaves without partial slots are skipped.
template <typename OutT, typename FarT>
__global__ void __launch_bounds__(128)
k_p2p_combine(int B, int64_t npts, const int32_t *__restrict__ begin, const int32_t *__restrict__ count,
              const int32_t *__restrict__ poff, const double4 *__restrict__ partial,
              const int32_t *__restrict__ perm, const FarT *__restrict__ far_phi, const FarT *__restrict__ far_E,
              OutT *__restrict__ pot, OutT *__restrict__ field) {
    const int64_t nl = (int64_t)1 << B;
    for (int64_t t = blockIdx.x; t < nl; t += gridDim.x) {
        const int p0 = poff[t], np = poff[t + 1] - p0;
        if (np == 0) continue;
        const int nt = count[nl - 1 + t], bt = begin[nl - 1 + t];
        const int k = np / nt;
        for (int i = threadIdx.x; i < nt; i += blockDim.x) {
            double4 s = partial[p0 + i];
            for (int j = 1; j < k; j++) {
                const double4 v = partial[p0 + j * nt + i];
                s.x += v.x;
                s.y += v.y;
                s.z += v.z;
                s.w += v.w;
            }
            const int64_t a = bt + i;
            const int64_t o = perm[a];
            pot[o] = (OutT)((double)far_phi[a] + s.x);
            if (field) {
                field[3 * o] = (OutT)((double)far_E[a] + s.y);
                field[3 * o + 1] = (OutT)((double)far_E[npts + a] + s.z);
                field[3 * o + 2] = (OutT)((double)far_E[2 * npts + a] + s.w);
            }
        }
    }
}

// batched: one block per leaf of every system that has partial slots
template <typename OutT>
__global__ void __launch_bounds__(128)
k_b_p2p_combine(const BatchSys *__restrict__ S, const int32_t *__restrict__ off, int nsys) {
    const int s = batch_sys_of(off, nsys, blockIdx.x);
    const BatchSys &y = S[s];
    const int64_t t = blockIdx.x - off[s], nl = y.nleaf;
    const int p0 = y.poff[t], np = y.poff[t + 1] - p0;
    if (np == 0) return;
    const int nt = y.count[nl - 1 + t], bt = y.begin[nl - 1 + t];
    const int k = np / nt;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) {
        double4 a = y.partial[p0 + i];
        for (int j = 1; j < k; j++) {
            const double4 v = y.partial[p0 + j * nt + i];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
        const int64_t g = bt + i;
        const int64_t o = y.perm[g];
        ((OutT *)y.pot)[o] = (OutT)((double)y.far_phi[g] + a.x);
        if (y.field) {
            ((OutT *)y.field)[3 * o] = (OutT)((double)y.far_E[g] + a.y);
            ((OutT *)y.field)[3 * o + 1] = (OutT)((double)y.far_E[y.n + g] + a.z);
            ((OutT *)y.field)[3 * o + 2] = (OutT)((double)y.far_E[2 * y.n + g] + a.w);
        }
    }
}

}  // namespace

cudaError_t eval_p2p(Plan &P, void *pot, void *field, int dtype) {
    stage_mark(P, FMM_STAGE_P2P, 0);
    if (P.prec == FMM_PREC_MIXED) {
        cudaError_t e = mixed_p2p(P, pot, field, dtype);
        stage_mark(P, FMM_STAGE_P2P, 1);
        return e;
    }
    cudaError_t e = tf_p2p(P, pot, field, dtype);
    if (e == cudaSuccess) e = p2p_combine(P, pot, field, dtype);
    stage_mark(P, FMM_STAGE_P2P, 1);
    return e;
}

cudaError_t p2p_combine(Plan &P, void *pot, void *field, int dtype) {
    if (P.p2p_nparts == 0) return cudaGetLastError();
    const unsigned grid = (unsigned)std::min<int64_t>(P.nleaf, (int64_t)sm_count() * 8);
    const bool mixed = P.prec == FMM_PREC_MIXED;
    if (mixed && dtype == FMM_F64)
        FMM_LAUNCH((k_p2p_combine<double, float>), grid, 128, 0, P.stream, P.B, P.n, P.begin, P.count, P.p2p_poff,
                   P.p2p_partial, P.perm, P.far_phi_f, P.far_E_f, (double *)pot, (double *)field);
    else if (mixed)
        FMM_LAUNCH((k_p2p_combine<float, float>), grid, 128, 0, P.stream, P.B, P.n, P.begin, P.count, P.p2p_poff,
                   P.p2p_partial, P.perm, P.far_phi_f, P.far_E_f, (float *)pot, (float *)field);
    else if (dtype == FMM_F64)
        FMM_LAUNCH((k_p2p_combine<double, double>), grid, 128, 0, P.stream, P.B, P.n, P.begin, P.count,
                   P.p2p_poff, P.p2p_partial, P.perm, P.far_phi, P.far_E, (double *)pot, (double *)field);
    else
        FMM_LAUNCH((k_p2p_combine<float, double>), grid, 128, 0, P.stream, P.B, P.n, P.begin, P.count,
                   P.p2p_poff, P.p2p_partial, P.perm, P.far_phi, P.far_E, (float *)pot, (float *)field);
    return cudaGetLastError();
}

cudaError_t direct_run(const void *points, const void *charges, int64_t n, int dtype,
                       const int64_t *targets, int64_t nt, void *pot, void *field,
                       cudaStream_t s) {
    if (nt == 0) return cudaSuccess;
    const cudaError_t e = direct_tf(points, charges, n, dtype, targets, nt, pot, field, s);
    if (e != cudaErrorMemoryAllocation) return e;
    // no workspace to be had: one block per target in FP64
    if (dtype == FMM_F64)
        FMM_LAUNCH(k_direct<double>, (unsigned)nt, 256, 0, s, (const double *)points, (const double *)charges,
                                                      n, targets, (double *)pot, (double *)field);
    else
        FMM_LAUNCH(k_direct<float>, (unsigned)nt, 256, 0, s, (const float *)points, (const float *)charges, n,
                                                     targets, (float *)pot, (float *)field);
    return cudaGetLastError();
}

cudaError_t batch_combine(const BatchSys *S, const int32_t *off, int nsys, int64_t blocks, int dtype,
                          cudaStream_t st) {
    if (blocks == 0) return cudaGetLastError();
    if (dtype == FMM_F64)
        FMM_LAUNCH(k_b_p2p_combine<double>, (unsigned)blocks, 128, 0, st, S, off, nsys);
    else
        FMM_LAUNCH(k_b_p2p_combine<float>, (unsigned)blocks, 128, 0, st, S, off, nsys);
    return cudaGetLastError();
}

}  // namespace fmm
