// Properties of computed bands: group velocity (Section 5.1, Eq. c_group)
// by the Hellmann-Feynman identity, and real-space eigenvector fields with
// their strain (Section 5.2, Eq. rotate_eigenvector).
//
// For an eigenpair A_k u = lambda M u (M independent of k):
//   d lambda / d k_m = u^H (dA_k/dk_m) u / u^H M u,
// and from the component form of Eq. (hatA), with q = xi + k, dq_j/dk_m = delta_jm,
// the stress field sigma = C(x) : F^-1(sym q (x) U) and S = F{sigma}:
//   u^H A_k u          = sum_xi conj(U_i) q_j S_ij,
//   u^H (dA_k/dk_m) u  = 2 Re sum_xi conj(U_i) S_im      (major symmetry of C).
// So one pass chain -- the K-apply's passes 1-4 and a forward z transform of
// the six stress components -- and one reduction give lambda (the Rayleigh
// quotient) and its gradient; d omega/d k = (d lambda/d k) / (2 omega).
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <vector>

#include "internal.h"

namespace bloch {

constexpr int kDkVals = 5;   // Re d_x, Re d_y, Re d_z, Re a, u^H M~ u

// Sum of products of one thread.  For FP32 values a pair hi + lo: the rounding
// error of a product is one fused multiply-add, that of an addition Knuth's
// two-sum, and both go to lo, so the products are exact and the sum carries about
// 48 bits.  FP64 values are added plainly.  GB300 runs FP64 at 1/64 of its FP32
// rate: with FP64 products and sums of FP32 values this pass took ten times its
// memory time.  Exact products cost 1.4 % of the property calls over rounded ones
// (128^3, 10 vectors: 4.21 -> 4.27 ms); the phase is then that of the FP32 values
// to 1e-15 (3e-9 from real-space FP32 fields in FP64 sums, 1e-9 with rounded
// products).
template <typename T> struct Sum;
template <> struct Sum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v, float err) {
        const dfloat s = df_two_sum(hi, v);
        hi = s.hi;
        lo = __fadd_rn(lo, __fadd_rn(s.lo, err));
    }
    __device__ __forceinline__ void mul(float a, float b) {   // += a b
        const float p = __fmul_rn(a, b);
        add(p, __fmaf_rn(a, b, -p));
    }
    __device__ __forceinline__ void mul(float a, const Sum& b) {   // += a b
        mul(a, b.hi);
        lo = __fmaf_rn(a, b.lo, lo);
    }
    __device__ __forceinline__ void add(const Sum& b) { add(b.hi, b.lo); }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
template <> struct Sum<double> {
    double s = 0.0;
    __device__ __forceinline__ void mul(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ void mul(double a, const Sum& b) { s = fma(a, b.s, s); }
    __device__ __forceinline__ void add(const Sum& b) { s += b.s; }
    __device__ __forceinline__ double value() const { return s; }
};

// Largest |component| of each FP32 vector (as bits, which order like the
// values), so that the sums below can scale it to O(1): products of vectors of
// any normalisation then stay inside the FP32 range.  Only ratios of the sums
// are used, so the power of two drops out.  mx zeroed by the caller.
static __global__ void k_absmax(const float2* __restrict__ U, long long n_per, unsigned* __restrict__ mx) {
    const float2* u = U + (size_t)blockIdx.y * n_per;
    float m = 0.f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_per;
         i += (long long)gridDim.x * blockDim.x)
        m = fmaxf(m, fmaxf(fabsf(u[i].x), fabsf(u[i].y)));
    unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0 && b) atomicMax(mx + blockIdx.y, b);
}
template <typename T> __device__ __forceinline__ T unit_scale(const unsigned* mx, int b);
template <> __device__ __forceinline__ float unit_scale<float>(const unsigned* mx, int b) {
    const int e = min(max((int)(mx[b] >> 23), 8), 246) - 127;
    return __uint_as_float((unsigned)(127 - e) << 23);   // 2^-e
}
template <> __device__ __forceinline__ double unit_scale<double>(const unsigned*, int) { return 1.0; }

// enqueues the maxima of nb vectors into mx (FP32; nothing to do in FP64)
template <typename T>
static bloch_status launch_absmax(bloch_plan* pl, int nb, const cplx_t<T>* u, unsigned* mx) {
    if constexpr (std::is_same<T, float>::value) {
        const long long n3 = 3 * pl->V;
        BLOCH_CUDA_CHECK_RET(cudaMemsetAsync(mx, 0, sizeof(unsigned) * nb, pl->stream));
        ++pl->launches;
        k_absmax<<<dim3((unsigned)std::max(1LL, std::min<long long>((n3 + 1023) / 1024, 512)), nb), 256, 0,
                   pl->stream>>>(u, n3, mx);
    }
    return BLOCH_OK;
}

// Per system b = blockIdx.y, per block: partial sums over Fourier voxels of
//   Re d_m = Re sum_i conj(U_i) S_im,  Re a = sum_m q_m Re d_m (per voxel),
//   mu = Re sum conj(U) (M~ U)
// with M~ U = MU (non-uniform density) or rho_s U.  Products and sums of a thread
// as Sum<T>, FP64 across threads.
template <typename T>
__global__ void k_dk_partial(const cplx_t<T>* __restrict__ U, const cplx_t<T>* __restrict__ S,
                             const cplx_t<T>* __restrict__ MU, double rho_s, const T* __restrict__ qtab, Geo g,
                             const unsigned* __restrict__ mx, double* __restrict__ partial) {
    using C = cplx_t<T>;
    const int b = blockIdx.y;
    const T sc = unit_scale<T>(mx, b);
    const C* ub = U + (size_t)b * 3 * g.V;
    const C* sb = S + (size_t)b * 6 * g.V;
    const C* mb = MU ? MU + (size_t)b * 3 * g.V : nullptr;
    const T* qb = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    // Voigt index of S_im: rows i = x, y, z; columns m = x, y, z
    const int vo[3][3] = {{0, 5, 4}, {5, 1, 3}, {4, 3, 2}};
    Sum<T> acc[kDkVals];
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < (unsigned)g.V; v += gridDim.x * blockDim.x) {
        T q[3];
        voxel_q(qb, g, v, q[0], q[1], q[2]);
        C u[3], s[6];
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = cscale(ub[(size_t)c * g.V + v], sc);
#pragma unroll
        for (int c = 0; c < 6; ++c) s[c] = cscale(sb[(size_t)c * g.V + v], sc);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            Sum<T> d;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const C sv = s[vo[i][m]];
                d.mul(u[i].x, sv.x);
                d.mul(u[i].y, sv.y);
            }
            acc[m].add(d);
            acc[3].mul(q[m], d);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const C mv = mb ? cscale(mb[(size_t)i * g.V + v], sc) : u[i];
            acc[4].mul(u[i].x, mv.x);
            acc[4].mul(u[i].y, mv.y);
        }
    }
    double tot[kDkVals];
#pragma unroll
    for (int i = 0; i < kDkVals; ++i) tot[i] = acc[i].value();
    if (!mb) tot[4] *= rho_s;
    block_sum<double, kDkVals>(tot);
    if (threadIdx.x == 0) {
        double* o = partial + ((size_t)b * gridDim.x + blockIdx.x) * kDkVals;
#pragma unroll
        for (int i = 0; i < kDkVals; ++i) o[i] = tot[i];
        // the pass error word rides behind the partials: the host reads it in the same copy
        if (b == 0 && blockIdx.x == 0) partial[(size_t)gridDim.y * gridDim.x * kDkVals] = *g.err ? 1.0 : 0.0;
    }
}

template <typename T>
static bloch_status group_velocity_impl(bloch_plan* pl, int nb, const double* k, const cplx_t<T>* u,
                                        double* omega_out, double* c_out) {
    bloch_status st = ensure_cg<T>(pl, nb);
    if (st != BLOCH_OK) return st;
    if ((st = set_k<T>(pl, nb, k)) != BLOCH_OK) return st;
    Workspace<T>& w = ws_of<T>(pl);
    // M u first: the mass operator's passes use the same workspace E that
    // then holds the stress field
    const cplx_t<T>* MU = nullptr;
    if (!pl->uniform_rho) {
        launch_M<T>(pl, nb, u, w.Ap, T(1));
        MU = w.Ap;
    }
    launch_K_stress<T>(pl, nb, u);
    const int nblk = (int)std::max(1LL, std::min<long long>((pl->V + 255) / 256, 512));
    const size_t nval = (size_t)nb * nblk * kDkVals;
    double* d_part = nullptr;
    if ((st = plan_solver_buf(pl, 2, 0, (nval + 1) * sizeof(double) + nb * sizeof(unsigned), (void**)&d_part)) != BLOCH_OK)
        return st;
    unsigned* d_mx = (unsigned*)(d_part + nval + 1);
    if ((st = launch_absmax<T>(pl, nb, u, d_mx)) != BLOCH_OK) return st;
    ++pl->launches;
    k_dk_partial<T><<<dim3(nblk, nb), 256, 0, pl->stream>>>(u, w.E, MU, pl->uniform_rho ? pl->rho_uniform_scaled : 1.0,
                                                            w.qtab, geo_of<T>(pl), d_mx, d_part);
    BLOCH_CUDA_CHECK_RET(cudaGetLastError());
    std::vector<double> h(nval + 1);
    BLOCH_CUDA_CHECK_RET(
        cudaMemcpyAsync(h.data(), d_part, h.size() * sizeof(double), cudaMemcpyDeviceToHost, pl->stream));
    BLOCH_CUDA_CHECK_RET(cudaStreamSynchronize(pl->stream));
    if (h[nval] != 0.0 && (st = check_pass_err(pl)) != BLOCH_OK) return st;
    for (int b = 0; b < nb; ++b) {
        double s[kDkVals] = {0};
        for (int j = 0; j < nblk; ++j)
            for (int i = 0; i < kDkVals; ++i) s[i] += h[((size_t)b * nblk + j) * kDkVals + i];
        const double uMu = pl->rho_ref * s[4];   // u^H M u (SI)
        if (!(uMu > 0.0)) return set_error(BLOCH_EINVAL, "a vector is zero (u^H M u = 0)");
        const double lam = pl->Kscale * s[3] / uMu;
        const double om = lam > 0.0 ? std::sqrt(lam) : 0.0;
        if (omega_out) omega_out[b] = om;
        for (int m = 0; m < 3; ++m) {
            const double dlam = pl->Kscale * pl->qscale * 2.0 * s[m] / uMu;
            c_out[(size_t)b * 3 + m] = om > 0.0 ? dlam / (2.0 * om) : 0.0;
        }
    }
    return BLOCH_OK;
}

// ------------------------------------------------ real-space eigenvectors
// Eq. (rotate_eigenvector): U(x) = e^{-i phi} F^-1(U^).  The paper takes phi
// as the one phase shared by every point of the field; phi = arg(s)/2 with
// s = sum_x sum_i U_i(x)^2 is that phase (mod pi) whenever the field has a
// single phase, and otherwise the single phase that maximises
// ||Re(e^{-i phi} U)|| (least squares).

// partial[b][blk] = sum over the block's Fourier voxels m of sum_i U_i(m) U_i(-m)
// = V sum_x sum_i (F^-1 U_i)(x)^2 (indices modulo the grid): the phase is
// known before the inverse transforms, whose last pass then applies it.
template <typename T>
__global__ void k_sq_partial(const cplx_t<T>* __restrict__ U, Geo g, const unsigned* __restrict__ mx,
                             double2* __restrict__ partial) {
    const int b = blockIdx.y;
    const T sc = unit_scale<T>(mx, b);
    const cplx_t<T>* ub = U + (size_t)b * 3 * g.V;
    Sum<T> acc[2];
    for (unsigned v = blockIdx.x * blockDim.x + threadIdx.x; v < (unsigned)g.V; v += gridDim.x * blockDim.x) {
        const unsigned t = fdiv(v, g.dx);
        const int x = (int)(v - t * (unsigned)g.Nx);
        const int z = (int)fdiv(t, g.dy), y = (int)t - z * g.Ny;
        const unsigned w = ((unsigned)(z ? g.Nz - z : 0) * g.Ny + (y ? g.Ny - y : 0)) * (unsigned)g.Nx +
                           (unsigned)(x ? g.Nx - x : 0);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cplx_t<T> a = cscale(ub[(size_t)c * g.V + v], sc), m = cscale(ub[(size_t)c * g.V + w], sc);
            acc[0].mul(a.x, m.x);
            acc[0].mul(-a.y, m.y);
            acc[1].mul(a.x, m.y);
            acc[1].mul(a.y, m.x);
        }
    }
    double tot[2] = {acc[0].value(), acc[1].value()};
    block_sum<double, 2>(tot);
    if (threadIdx.x == 0) partial[(size_t)b * gridDim.x + blockIdx.x] = make_double2(tot[0], tot[1]);
}

template <typename T>
static bloch_status eigvec_real_impl(bloch_plan* pl, int nb, const cplx_t<T>* uh, cplx_t<T>* ur, cplx_t<T>* eps,
                                     double* phi_out) {
    bloch_status st = ensure_ws<T>(pl, nb);
    if (st != BLOCH_OK) return st;
    const int nblk = (int)std::max(1LL, std::min<long long>((pl->V + 255) / 256, 512));
    double2* d_part = nullptr;
    if ((st = plan_solver_buf(pl, 2, 1, sizeof(double2) * ((size_t)nb * nblk + 2 * nb) + nb * sizeof(unsigned),
                              (void**)&d_part)) != BLOCH_OK)
        return st;
    double2* d_ph = d_part + (size_t)nb * nblk;   // e^{-i phi}, then i e^{-i phi}
    unsigned* d_mx = (unsigned*)(d_ph + 2 * (size_t)nb);
    if ((st = launch_absmax<T>(pl, nb, uh, d_mx)) != BLOCH_OK) return st;
    ++pl->launches;
    k_sq_partial<T><<<dim3(nblk, nb), 256, 0, pl->stream>>>(uh, geo_of<T>(pl), d_mx, d_part);
    BLOCH_CUDA_CHECK_RET(cudaGetLastError());
    std::vector<double2> h((size_t)nb * nblk);
    BLOCH_CUDA_CHECK_RET(
        cudaMemcpyAsync(h.data(), d_part, sizeof(double2) * h.size(), cudaMemcpyDeviceToHost, pl->stream));
    BLOCH_CUDA_CHECK_RET(cudaStreamSynchronize(pl->stream));
    std::vector<double2> ph(2 * (size_t)nb);
    for (int b = 0; b < nb; ++b) {
        double re = 0.0, im = 0.0;
        for (int j = 0; j < nblk; ++j) {
            re += h[(size_t)b * nblk + j].x;
            im += h[(size_t)b * nblk + j].y;
        }
        const double phi = 0.5 * std::atan2(im, re);
        if (phi_out) phi_out[b] = phi;
        ph[b] = make_double2(std::cos(phi), -std::sin(phi));
        ph[nb + b] = make_double2(std::sin(phi), std::cos(phi));
    }
    BLOCH_CUDA_CHECK_RET(
        cudaMemcpyAsync(d_ph, ph.data(), sizeof(double2) * ph.size(), cudaMemcpyHostToDevice, pl->stream));
    launch_fft3<T, +1>(pl, nb, uh, ur, T(1.0 / (double)pl->V), d_ph);       // F^-1 (numpy normalisation)
    if (eps) {
        std::vector<double> zero((size_t)nb * 3, 0.0);
        if ((st = set_k<T>(pl, nb, zero.data())) != BLOCH_OK) return st;
        launch_strain_real<T>(pl, nb, uh, eps, T(1.0 / (pl->qscale * (double)pl->V)), d_ph + nb);
    }
    BLOCH_CUDA_CHECK_RET(cudaGetLastError());
    return check_pass_err(pl);   // synchronises
}

}  // namespace bloch

using namespace bloch;

extern "C" bloch_status bloch_eigvec_real(bloch_plan* pl, int32_t nb, int32_t precision, const void* u_hat,
                                          void* u_real, void* strain, double* phi_out) {
    if (!pl) return set_error(BLOCH_EINVAL, "plan is NULL");
    if (nb < 1 || 2 * nb > 65535 / 3) return set_error(BLOCH_EINVAL, "nb must be in [1, 10922]");
    if (precision != BLOCH_FP32 && precision != BLOCH_FP64)
        return set_error(BLOCH_EINVAL, "precision must be BLOCH_FP32 or BLOCH_FP64");
    if (!u_hat || !u_real) return set_error(BLOCH_EINVAL, "NULL argument");
    if (u_hat == u_real || u_hat == strain) return set_error(BLOCH_EINVAL, "outputs may not alias u_hat");
    if (precision == BLOCH_FP32)
        return eigvec_real_impl<float>(pl, nb, (const float2*)u_hat, (float2*)u_real, (float2*)strain, phi_out);
    return eigvec_real_impl<double>(pl, nb, (const double2*)u_hat, (double2*)u_real, (double2*)strain, phi_out);
}

extern "C" bloch_status bloch_group_velocity(bloch_plan* pl, int32_t nb, const double* k, int32_t precision,
                                             const void* u, double* omega_out, double* c_out) {
    if (!pl) return set_error(BLOCH_EINVAL, "plan is NULL");
    if (nb < 1 || nb > 65535 / 6) return set_error(BLOCH_EINVAL, "nb must be in [1, 10922]");
    if (precision != BLOCH_FP32 && precision != BLOCH_FP64)
        return set_error(BLOCH_EINVAL, "precision must be BLOCH_FP32 or BLOCH_FP64");
    if (!k || !u || !c_out) return set_error(BLOCH_EINVAL, "NULL argument");
    bloch_status st;
    if (precision == BLOCH_FP32)
        st = group_velocity_impl<float>(pl, nb, k, (const float2*)u, omega_out, c_out);
    else
        st = group_velocity_impl<double>(pl, nb, k, (const double2*)u, omega_out, c_out);
    if (st != BLOCH_OK) return st;
    BLOCH_CUDA_CHECK_RET(cudaGetLastError());
    return BLOCH_OK;
}
