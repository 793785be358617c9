// Pointwise and reduction kernels: wave-vector tables, Green-operator
// preconditioner (Eqs. matrixP, precond), dot products and the fused PCG
// updates of Algorithm 2.  Reductions: per-thread accumulation in the field
// precision, warp shuffle, one partial per block in FP64, and a one-block
// final sum per system (deterministic, no atomics).
#pragma once

#include "cg.cuh"
#include "common.cuh"
#include "passes.cuh"

namespace bloch {

// Wave vectors of a small batch, passed as kernel arguments: no copy to the
// device precedes the operator.
constexpr int kParamWaves = 32;
struct WaveParams {
    double k[3 * kParamWaves];
};

// qtab[b][.] = ((xi + k_b) * qscale) for the x, y and z axes; k_b from kvec or,
// with kvec == nullptr, from wp.
template <typename T>
__global__ void k_qtab(const double* __restrict__ kvec, const __grid_constant__ WaveParams wp,
                       const double* __restrict__ xi, int Nx, int Ny, int Nz, int nb, double qscale,
                       T* __restrict__ qtab) {
    pdl_launch();
    const int S = Nx + Ny + Nz;
    const long long total = (long long)nb * S;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(i / S), j = (int)(i % S);
        const int ax = j < Nx ? 0 : (j < Nx + Ny ? 1 : 2);
        qtab[i] = T((xi[j] + (kvec ? kvec : wp.k)[3 * b + ax]) * qscale);
    }
}

template <typename T>
__global__ void k_scale(const cplx_t<T>* in, cplx_t<T>* out, T s, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = cscale(in[i], s);
}

// voxel index -> (x, y, z) in 32-bit unsigned arithmetic (V < 2^31 for every
// supported grid)
template <typename T>
__device__ __forceinline__ void voxel_q(const T* qb, const Geo& g, unsigned v, T& ax, T& ay, T& az) {
    const unsigned t = fdiv(v, g.dx);
    const int x = (int)(v - t * (unsigned)g.Nx);
    const unsigned z = fdiv(t, g.dy);
    const int y = (int)(t - z * (unsigned)g.Ny);
    ax = qb[x];
    ay = qb[g.Nx + y];
    az = qb[g.Nx + g.Ny + z];
}

template <typename T>
__global__ void k_precond(const cplx_t<T>* r, cplx_t<T>* z, const T* __restrict__ qtab, Geo g, PrecondCoef pc,
                          PrecondSel ps, T out_scale) {
    using C = cplx_t<T>;
    const int b = blockIdx.y;
    const T* qb = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    const C* rb = r + (size_t)b * 3 * g.V;
    C* zb = z + (size_t)b * 3 * g.V;
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < (unsigned)g.V; v += gridDim.x * blockDim.x) {
        T ax, ay, az;
        voxel_q(qb, g, v, ax, ay, az);
        C rv[3] = {rb[v], rb[g.V + v], rb[2 * g.V + v]};
        C zv[3];
        pre_apply<T>(ps, pc, b, v, g.V, ax, ay, az, rv, zv);
#pragma unroll
        for (int c = 0; c < 3; ++c) zb[c * g.V + v] = cscale(zv[c], out_scale);
    }
}

// ---------------------------------------------------------------- reductions
// partial[b][blk] = sum over the block's voxels of conj(a) b (complex)
template <typename T>
__global__ void k_dot_partial(const cplx_t<T>* a, const cplx_t<T>* bv, long long n_per, double2* partial) {
    using C = cplx_t<T>;
    const int b = blockIdx.y;
    const C* ab = a + (size_t)b * n_per;
    const C* bb = bv + (size_t)b * n_per;
    T acc[2] = {T(0), T(0)};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_per;
         i += (long long)gridDim.x * blockDim.x) {
        const C x = ab[i], y = bb[i];
        acc[0] += x.x * y.x + x.y * y.y;
        acc[1] += x.x * y.y - x.y * y.x;
    }
    block_sum<T, 2>(acc);
    if (threadIdx.x == 0) partial[(size_t)b * gridDim.x + blockIdx.x] = make_double2(acc[0], acc[1]);
}

static __global__ void k_dot_final(const double2* partial, int nblk, double2* out) {
    const int b = blockIdx.x;
    double acc[2] = {0.0, 0.0};
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
        const double2 v = partial[(size_t)b * nblk + i];
        acc[0] += v.x;
        acc[1] += v.y;
    }
    block_sum<double, 2>(acc);
    if (threadIdx.x == 0) out[b] = make_double2(acc[0], acc[1]);
}

// --------------------------------------------------------------- PCG kernels
// Sum of products of vectors whose size is not known: the sum in units of 4^e,
// 2^e a power of two that bounds the components met so far, so that the squares
// stay inside the FP32 range whatever the components are (a power of two changes
// no digit).  FP64 needs no units.  Costs 0.3 % of a solve of four iterations
// (128^3, 8 systems: 11.17 -> 11.21 ms), where a maximum found in a pass of its own
// would read the right-hand side once more.
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + min(max(e, -126), 126)) << 23); }
template <typename T, int NV> struct UnitSum;
template <int NV> struct UnitSum<float, NV> {
    float v[NV] = {};
    int e = -126;
    // the factor that brings components c to the unit of the sum, after raising it to theirs
    __device__ __forceinline__ float unit(const float2 (&c)[3]) {
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 3; ++i) m = fmaxf(m, fmaxf(fabsf(c[i].x), fabsf(c[i].y)));
        raise(min((__float_as_int(m) >> 23) - 126, 126));
        return pow2f(-e);
    }
    __device__ __forceinline__ void raise(int to) {
        if (to <= e) return;
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] *= pow2f(2 * (e - to));
        e = to;
    }
};
template <int NV> struct UnitSum<double, NV> {
    double v[NV] = {};
    __device__ __forceinline__ double unit(const double2 (&)[3]) { return 1.0; }
};

// Block sums of a and b in their values' own units, valid in thread 0
template <int NA, int NB>
__device__ __forceinline__ void unit_totals(UnitSum<float, NA>& a, UnitSum<float, NB>& b, double (&out)[NA + NB]) {
    __shared__ int top[2];
    if (threadIdx.x < 2) top[threadIdx.x] = -126;
    __syncthreads();
    const int ea = __reduce_max_sync(0xffffffffu, a.e), eb = __reduce_max_sync(0xffffffffu, b.e);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&top[0], ea);
        atomicMax(&top[1], eb);
    }
    __syncthreads();
    a.raise(top[0]);
    b.raise(top[1]);
    float v[NA + NB];
#pragma unroll
    for (int i = 0; i < NA + NB; ++i) v[i] = i < NA ? a.v[i < NA ? i : 0] : b.v[i < NA ? 0 : i - NA];
    block_sum<float, NA + NB>(v);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NA + NB; ++i) out[i] = scalbn((double)v[i], 2 * (i < NA ? a.e : b.e));
    }
}
template <int NA, int NB>
__device__ __forceinline__ void unit_totals(UnitSum<double, NA>& a, UnitSum<double, NB>& b, double (&out)[NA + NB]) {
#pragma unroll
    for (int i = 0; i < NA + NB; ++i) out[i] = i < NA ? a.v[i < NA ? i : 0] : b.v[i < NA ? 0 : i - NA];
    block_sum<double, NA + NB>(out);
}

// r = s*b - Ax (Ax may be null -> r = s*b, x = 0), p = P^-1 r;
// partials (r,z), (r,r), (s b, s b).
template <typename T>
__global__ void k_cg_init(const cplx_t<T>* bvec, const cplx_t<T>* Ax, cplx_t<T>* x, cplx_t<T>* r, cplx_t<T>* p,
                          const T* __restrict__ qtab, Geo g, PrecondCoef pc, PrecondSel ps, T s, int zero_x,
                          double* partial) {
    using C = cplx_t<T>;
    const int b = blockIdx.y;
    const size_t off = (size_t)b * 3 * g.V;
    const T* qb = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    UnitSum<T, 2> rs;   // (r, z), (r, r)
    UnitSum<T, 1> bs;   // (s b, s b)
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < (unsigned)g.V; v += gridDim.x * blockDim.x) {
        C bv[3], rv[3], zv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t i = off + c * g.V + v;
            bv[c] = cscale(bvec[i], s);
            rv[c] = Ax ? csub(bv[c], Ax[i]) : bv[c];
            if (zero_x) x[i] = mk(T(0), T(0));
            r[i] = rv[c];
        }
        T ax, ay, az;
        voxel_q(qb, g, v, ax, ay, az);
        pre_apply<T>(ps, pc, b, v, g.V, ax, ay, az, rv, zv);
        const T ub = bs.unit(bv), ur = rs.unit(rv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            p[off + c * g.V + v] = zv[c];
            const C bu = cscale(bv[c], ub), ru = cscale(rv[c], ur), zu = cscale(zv[c], ur);
            bs.v[0] += bu.x * bu.x + bu.y * bu.y;
            rs.v[0] += ru.x * zu.x + ru.y * zu.y;
            rs.v[1] += ru.x * ru.x + ru.y * ru.y;
        }
    }
    double tot[3];
    unit_totals(rs, bs, tot);
    if (threadIdx.x == 0) {
        double* o = partial + ((size_t)b * gridDim.x + blockIdx.x) * 3;
        o[0] = tot[0];
        o[1] = tot[1];
        o[2] = tot[2];
    }
}

// r -= alpha Ap; partials (r, P^-1 r), (r, r), for the plain-form baseline's
// operator (the passes update r in their divergence).  The matching x += alpha p
// is applied by k_cg_pupdate, which reads p anyway.
template <typename T>
__global__ void k_cg_update(cplx_t<T>* __restrict__ r, const cplx_t<T>* __restrict__ Ap,
                            const T* __restrict__ qtab, Geo g, PrecondCoef pc, PrecondSel ps, const CGSys* sys,
                            double* partial) {
    using C = cplx_t<T>;
    const int b = blockIdx.y;
    const size_t off = (size_t)b * 3 * g.V;
    const T* qb = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    const bool act = sys[b].active != 0;
    const T alpha = act ? T(sys[b].alpha) : T(0);
    T acc[2] = {T(0), T(0)};
    if (act) {
#pragma unroll 2
        for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < (unsigned)g.V; v += gridDim.x * blockDim.x) {
            C rv[3], zv[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const size_t i = off + c * g.V + v;
                const C av = Ap[i];
                const C ro = r[i];
                rv[c] = mk(fma(-alpha, av.x, ro.x), fma(-alpha, av.y, ro.y));
                r[i] = rv[c];
            }
            T ax, ay, az;
            voxel_q(qb, g, v, ax, ay, az);
            pre_apply<T>(ps, pc, b, v, g.V, ax, ay, az, rv, zv);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                acc[0] += rv[c].x * zv[c].x + rv[c].y * zv[c].y;
                acc[1] += rv[c].x * rv[c].x + rv[c].y * rv[c].y;
            }
        }
    }
    block_sum<T, 2>(acc);
    if (threadIdx.x == 0) {
        double* o = partial + ((size_t)b * gridDim.x + blockIdx.x) * 3;
        o[0] = acc[0];
        o[1] = acc[1];
        o[2] = 0.0;
    }
}

// For systems that took a step: x += alpha p (old p); then, if still active,
// p = P^-1 r + beta p.
template <typename T>
__global__ void k_cg_pupdate(const cplx_t<T>* r, cplx_t<T>* __restrict__ p, cplx_t<T>* __restrict__ x,
                             const T* qtab, Geo g, PrecondCoef pc, PrecondSel ps, const CGSys* sys) {
    using C = cplx_t<T>;
    const int b = blockIdx.y;
    pdl_wait();
    pdl_launch();
    if (!sys[b].upd) return;
    const bool act = sys[b].active != 0;
    const size_t off = (size_t)b * 3 * g.V;
    const T* qb = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    const T alpha = T(sys[b].alpha);
    const T beta = T(sys[b].beta);
#pragma unroll 2
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < (unsigned)g.V; v += gridDim.x * blockDim.x) {
        C pv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const size_t i = off + c * g.V + v;
            pv[c] = p[i];
            const C xv = x[i];
            x[i] = mk(fma(alpha, pv[c].x, xv.x), fma(alpha, pv[c].y, xv.y));
        }
        if (act) {
            C rv[3], zv[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) rv[c] = r[off + c * g.V + v];
            T ax, ay, az;
            voxel_q(qb, g, v, ax, ay, az);
            pre_apply<T>(ps, pc, b, v, g.V, ax, ay, az, rv, zv);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                p[off + c * g.V + v] = mk(fma(beta, pv[c].x, zv[c].x), fma(beta, pv[c].y, zv[c].y));
        }
    }
}

// Scalar recurrences of Algorithm 2, one block per system.
// After the initial residual: rz, rr, bb from the 3-wide partials; active = rr > tol^2 bb.
// A p is zero in a bin where q = xi + k is zero (k = 0, or k on the reciprocal
// lattice), so no step changes r there: a system whose residual in that bin alone
// exceeds the tolerance can never meet it (stuck).
template <typename T>
__global__ void k_cg_start(const double* partial3, int nblk, CGSys* sys, double tol2, int* n_active,
                           const cplx_t<T>* r, const T* qtab, Geo g) {
    const int b = blockIdx.x;
    __shared__ int zero[3];   // index of q = 0 along each axis
    if (threadIdx.x < 3) zero[threadIdx.x] = -1;
    __syncthreads();
    const T* qb = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    for (int i = threadIdx.x; i < g.Nx + g.Ny + g.Nz; i += blockDim.x)
        if (qb[i] == T(0)) {
            const int ax = i < g.Nx ? 0 : (i < g.Nx + g.Ny ? 1 : 2);
            zero[ax] = i - (ax > 0 ? g.Nx : 0) - (ax > 1 ? g.Ny : 0);
        }
    double acc[3] = {0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
        const double* v = partial3 + ((size_t)b * nblk + i) * 3;
        acc[0] += v[0];
        acc[1] += v[1];
        acc[2] += v[2];
    }
    block_sum<double, 3>(acc);
    if (threadIdx.x != 0) return;
    CGSys& s = sys[b];
    s.rz = s.rz0 = acc[0];
    s.rr = acc[1];
    s.bb = acc[2];
    s.iters = 0;
    s.upd = 0;
    s.active = (s.rr > tol2 * s.bb) ? 1 : 0;
    double rest = 0.0;
    if (zero[0] >= 0 && zero[1] >= 0 && zero[2] >= 0) {
        const size_t v = ((size_t)zero[2] * g.Ny + zero[1]) * g.Nx + zero[0];
        for (int c = 0; c < 3; ++c) {
            const cplx_t<T> w = r[((size_t)b * 3 + c) * g.V + v];
            rest += (double)w.x * w.x + (double)w.y * w.y;
        }
    }
    s.stuck = rest > tol2 * s.bb ? 1 : 0;
    if (s.active) atomicAdd(n_active, 1);
}

// After the stress pass: (p, A p) from its partials, alpha = rz / (p, A p).
// scaled: the sum carries the square of cg_scale (in k_cg_beta (r, z) likewise,
// and (r, r) the square of cg_scale_rr).
static __global__ void k_cg_alpha(const double2* partial2, int nblk, CGSys* sys, int scaled, int* n_active) {
    const int b = blockIdx.x;
    pdl_wait();
    pdl_launch();
    CGSys& s = sys[b];
    double acc[1] = {0.0};
    if (s.active)
        for (int i = threadIdx.x; i < nblk; i += blockDim.x) acc[0] += partial2[(size_t)b * nblk + i].x;
    block_sum<double, 1>(acc);
    if (threadIdx.x != 0) return;
    if (b == 0) *n_active = 0;   // recounted by k_cg_beta (kernels of one stream are ordered)
    const double sc = scaled ? (double)cg_scale<float>(sys, b) : 1.0;
    s.pAp = acc[0] / (sc * sc);
    s.alpha = (s.active && s.pAp > 0.0) ? s.rz / s.pAp : 0.0;
    s.upd = s.active;
}

// After the residual update: rz_new, rr; convergence test; beta = rz_new / rz.
// A system that cannot converge (stuck, k_cg_start) also ends when (r, z) has
// fallen below rz_floor of its start: the rest of r is then solved for as far as
// its digits go, and going on to the iteration cap would change nothing.  It counts
// as not converged.  Every other system goes on as long as the tolerance asks.
// The last block to finish sets the condition of the graph-resident loop
// (cond != 0): continue while a system is active and the iteration cap, which
// bounds every launch, is not reached.  *ticket counts finished blocks and is
// left at zero.
static __global__ void k_cg_beta(const double* partial3, int nblk, CGSys* sys, double tol2, double rz_floor, int scaled,
                                 int* n_active, int* ticket, int cond, cudaGraphConditionalHandle h, int* iter, int max_iter) {
    const int b = blockIdx.x;
    pdl_wait();
    pdl_launch();
    CGSys& s = sys[b];
    double acc[2] = {0.0, 0.0};
    const int active = s.active;
    if (active)
        for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
            const double* v = partial3 + ((size_t)b * nblk + i) * 3;
            acc[0] += v[0];
            acc[1] += v[1];
        }
    block_sum<double, 2>(acc);
    if (threadIdx.x != 0) return;
    if (active) {
        const double sc = scaled ? (double)cg_scale<float>(sys, b) : 1.0;
        const double sr = scaled ? (double)cg_scale_rr<float>(sys, b) : 1.0;   // of the old (r, r)
        s.iters += 1;
        s.rz_new = acc[0] / (sc * sc);
        s.rr = acc[1] / (sr * sr);
        if (!(s.rr > tol2 * s.bb) || !(s.rz_new > (s.stuck ? rz_floor * s.rz0 : 0.0))) {
            s.active = 0;
        } else {
            s.beta = s.rz_new / s.rz;
            s.rz = s.rz_new;
            atomicAdd(n_active, 1);
        }
    }
    if (!cond) return;
    __threadfence();
    if (atomicAdd(ticket, 1) == (int)gridDim.x - 1) {
        *ticket = 0;
        __threadfence();
        const int i = ++(*iter);
        cudaGraphSetConditional(h, (*(volatile int*)n_active > 0 && i < max_iter) ? 1u : 0u);
    }
}

// Device tally of PCG runs enqueued without host synchronisation:
// tally[0] += sum of iterations, tally[1] += systems that missed tol,
// tally[2] += systems with a non-finite residual, tally[3] += loop
// iterations executed (*iter, the graph's iteration counter).
static __global__ void k_cg_tally(const CGSys* __restrict__ sys, int nb, double tol2, const int* __restrict__ iter,
                                  long long* __restrict__ tally) {
    long long it = 0, miss = 0, bad = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        it += sys[b].iters;
        const double rr = sys[b].rr, bb = sys[b].bb;
        if (!isfinite(rr) || !isfinite(bb)) ++bad;
        else if (rr > tol2 * bb) ++miss;
    }
    for (int o = 16; o > 0; o >>= 1) {
        it += __shfl_xor_sync(0xffffffffu, it, o);
        miss += __shfl_xor_sync(0xffffffffu, miss, o);
        bad += __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if (threadIdx.x == 0) {
        tally[0] += it;
        tally[1] += miss;
        tally[2] += bad;
        tally[3] += *iter;
    }
}

}  // namespace bloch
