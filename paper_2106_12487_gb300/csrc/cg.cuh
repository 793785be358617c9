// Conjugate-gradient state, Green-operator preconditioner (Eqs. matrixP, precond)
// and block sums, shared by the vector kernels and the passes that update the
// residual.
#pragma once

#include "common.cuh"

namespace bloch {

// P_ik = sum_m A[ik][m] mono_m(q), pairs ik in (xx, yy, zz, yz, xz, xy) and
// monomials (qx^2, qy^2, qz^2, qy qz, qx qz, qx qy), from the scaled C0.
struct PrecondCoef {
    double a[6][6];
    float af[6][6];   // the same coefficients rounded once to FP32 (FP32 kernels read these:
                      // no FP64 -> FP32 conversion per voxel)
};
template <typename T> __device__ __forceinline__ T pcoef(const PrecondCoef& pc, int i, int j);
template <> __device__ __forceinline__ float pcoef<float>(const PrecondCoef& pc, int i, int j) { return pc.af[i][j]; }
template <> __device__ __forceinline__ double pcoef<double>(const PrecondCoef& pc, int i, int j) { return pc.a[i][j]; }

// Per-system CG scalars (device resident).
struct CGSys {
    double rz;       // (r, z) of the current iterate
    double rz_new;
    double rz0;      // (r, z) of the start residual
    double pAp;
    double rr;       // (r, r)
    double bb;       // (b, b) (scaled)
    double alpha;
    double beta;
    int active;
    int iters;
    int upd;         // took a step this iteration (x += alpha p is still to be applied)
    int stuck;       // cannot converge: |r|^2 in the bin where q = 0 exceeds tol^2 bb
};

// Correctly rounded reciprocal (the FP32 form uses the rounded reciprocal
// intrinsic instead of a full division).
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

// z = P^-1(q) r for one voxel (three complex components); zero where q = 0.
template <typename T>
__device__ __forceinline__ void green_apply(const PrecondCoef& pc, T qx, T qy, T qz, const cplx_t<T> r[3],
                                            cplx_t<T> z[3]) {
    const T m[6] = {qx * qx, qy * qy, qz * qz, qy * qz, qx * qz, qx * qy};
    T P[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        T s = 0;
#pragma unroll
        for (int j = 0; j < 6; ++j) s = fma(pcoef<T>(pc, i, j), m[j], s);
        P[i] = s;
    }
    const T a = P[0], bq = P[1], c = P[2], d = P[3], e = P[4], f = P[5];
    const T A = bq * c - d * d, B = a * c - e * e, Cc = a * bq - f * f;
    const T D = e * f - a * d, Ee = d * f - bq * e, F = d * e - c * f;
    const T det = a * A + f * F + e * Ee;
    if (m[0] + m[1] + m[2] == T(0) || det == T(0)) {
        z[0] = z[1] = z[2] = mk(T(0), T(0));
        return;
    }
    const T id = recip(det);
    z[0] = cscale(cadd(cadd(cscale(r[0], A), cscale(r[1], F)), cscale(r[2], Ee)), id);
    z[1] = cscale(cadd(cadd(cscale(r[0], F), cscale(r[1], B)), cscale(r[2], D)), id);
    z[2] = cscale(cadd(cadd(cscale(r[0], Ee), cscale(r[1], D)), cscale(r[2], Cc)), id);
}

// Preconditioner selection: the Green operator P^-1 computed per voxel, or a
// precomputed symmetric 3x3 table per voxel (the learned preconditioner), one
// table per group of `zgroup` consecutive systems.
struct PrecondSel {
    const float* ztab;   // nullptr: Green operator
    int zgroup;
};

template <typename T>
__device__ __forceinline__ void zsym_apply(const float* Z, const cplx_t<T> r[3], cplx_t<T> z[3]) {
    const T a = T(Z[0]), b = T(Z[1]), c = T(Z[2]), d = T(Z[3]), e = T(Z[4]), f = T(Z[5]);
    z[0] = cadd(cadd(cscale(r[0], a), cscale(r[1], f)), cscale(r[2], e));
    z[1] = cadd(cadd(cscale(r[0], f), cscale(r[1], b)), cscale(r[2], d));
    z[2] = cadd(cadd(cscale(r[0], e), cscale(r[1], d)), cscale(r[2], c));
}

template <typename T>
__device__ __forceinline__ void pre_apply(const PrecondSel& ps, const PrecondCoef& pc, int sys, unsigned v,
                                          long long V, T qx, T qy, T qz, const cplx_t<T> r[3], cplx_t<T> z[3]) {
    if (ps.ztab) zsym_apply<T>(ps.ztab + ((size_t)(sys / ps.zgroup) * V + v) * 6, r, z);
    else green_apply(pc, qx, qy, qz, r, z);
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sum of NV values; result valid in thread 0.
template <typename T, int NV>
__device__ __forceinline__ void block_sum(T (&v)[NV]) {
    __shared__ T red[NV][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) red[i][w] = v[i];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            T s = lane < nw ? red[i][lane] : T(0);
            v[i] = warp_sum(s);
        }
    }
}

// Powers of two near 1 / sqrt((r, z)) and 1 / sqrt((r, r)) of a system.  The FP32
// iteration forms its products from the direction and residual times the first,
// and (r, r) from the residual times the second, so that neither underflows nor
// overflows however small the residual gets (a power of two changes no digit; the
// sums of the start residual carry their own units, k_cg_init).  The operator of
// the plain-form baseline (fft_variant 2) forms its products unscaled.
// One scale does not do for both: a part of r that P^-1 does not see (bin 0 at
// k = 0) keeps (r, r) up while (r, z) falls by 32 digits, and its scaled square
// would leave the FP32 range.  The scalars are kept unscaled in FP64.  FP64 fields
// need no scale.
template <typename T> __device__ __forceinline__ T inv_sqrt_pow2(double v);
template <> __device__ __forceinline__ float inv_sqrt_pow2<float>(double v) {
    const int e = ((__double2hiint(v) >> 20) & 0x7ff) - 1023;
    return __int_as_float((127 + min(max(-(e >> 1), -100), 100)) << 23);
}
template <> __device__ __forceinline__ double inv_sqrt_pow2<double>(double) { return 1.0; }
template <typename T> __device__ __forceinline__ T cg_scale(const CGSys* sys, int b) {
    return inv_sqrt_pow2<T>(sys[b].rz);
}
template <typename T> __device__ __forceinline__ T cg_scale_rr(const CGSys* sys, int b) {
    return inv_sqrt_pow2<T>(sys[b].rr);
}

// What the divergence pass needs to update the residual in place of storing
// A p: r -= alpha A p, partials (r, P^-1 r) and (r, r) per CTA at
// partial[(b gridDim.x + blockIdx.x) 3].
template <typename T>
struct CgUpdate {
    cplx_t<T>* r;
    const CGSys* sys;
    double* partial;
    PrecondCoef pc;
    PrecondSel ps;
};

// Residual update at one voxel whose old residual is ro: ap = A p there times
// the system's scale sc, alpha likewise divided by it; acc += (r, z) times sc^2
// and (r, r) times sr^2 (sr = cg_scale_rr).  Callers read the residuals of several voxels before the first
// update: a load cannot pass the stores of r before it.
template <typename T>
__device__ __forceinline__ void cg_update_at(const CgUpdate<T>& cg, cplx_t<T>* rb, int b, long long V, unsigned v, T alpha,
                                             T sc, T sr, T qx, T qy, T qz, const cplx_t<T> (&ap)[3],
                                             const cplx_t<T> (&ro)[3], T (&acc)[2]) {
    cplx_t<T> rv[3], zv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        rv[c] = mk(fma(-alpha, ap[c].x, ro[c].x), fma(-alpha, ap[c].y, ro[c].y));
        rb[c * V + v] = rv[c];
        const cplx_t<T> w = sizeof(T) == 4 ? cscale(rv[c], sr) : rv[c];
        acc[1] += w.x * w.x + w.y * w.y;
        if constexpr (sizeof(T) == 4) rv[c] = cscale(rv[c], sc);
    }
    pre_apply<T>(cg.ps, cg.pc, b, v, V, qx, qy, qz, rv, zv);
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[0] += rv[c].x * zv[c].x + rv[c].y * zv[c].y;
}
template <typename T>
__device__ __forceinline__ void cg_partial_out(const CgUpdate<T>& cg, int b, T (&acc)[2]) {
    block_sum<T, 2>(acc);
    if (threadIdx.x == 0) {
        double* o = cg.partial + ((size_t)b * gridDim.x + blockIdx.x) * 3;
        o[0] = (double)acc[0];
        o[1] = (double)acc[1];
        o[2] = 0.0;
    }
}

}  // namespace bloch
