// Mixed-radix FFT passes of the Bloch stiffness and mass operators: any axis
// length up to 512 with prime factors in {2,3,5,7}, in FP32, FP64 and
// float-float.
//
// Stiffness operator A_k (Eq. hatA, component form), Fourier basis in and out,
// five HBM passes with the pointwise work fused into the FFT passes:
//   pass 1  z: inverse FFTs a_k, b_k of U_k and q_z U_k along z, strains
//            gamma_c in Voigt order (engineering shear)          3c in, 6c out
//   pass 2  y: inverse FFT along y, 6 components in place      6c in, 6c out
//   pass 3  x: inverse FFT along x, sigma = C_g(x) gamma / V,
//            forward FFT along x, in place                      6c + id in, 6c out
//   pass 4  y: forward FFT along y, in place                    6c in, 6c out
//   pass 5  z: forward FFT along z, divergence
//            out_i = sum_j q_j sigma_ij                         6c in, 3c out
// with q = xi + k.  The factor 1/V of F^-1 and the unit scaling are folded
// into the per-grain stiffness table.  Mass operator with non-uniform rho: the
// same chain on the three displacement components with rho_g(x)/V in pass 3.
//
// A pencil of length N = r1 r2 r3 is transformed in place in shared memory by
// decimation in frequency, each thread owning one radix-R butterfly in
// registers at a time.  With the input index n = n1 r2 r3 + n2 r3 + n3:
//   stage 1  DFT over n1 -> k1, times w_N^(k1 (n2 r3 + n3))
//   stage 2  DFT over n2 -> k2, times w_(r2 r3)^(k2 n3)        (r2 > 1 only)
//   stage 3  DFT over n3 -> k3
// leaves output k = k1 + r1 k2 + r1 r2 k3 in the slot of (k1, k2, k3).  The
// digit-reversed order costs nothing: the z and y passes write whole rows of
// neighbouring pencils for each k, and the x pass applies the stress in that
// order and undoes it with the mirrored (decimation in time) stages.  The
// first stage loads its inputs straight from HBM into registers and the last
// stage or the pointwise epilogue stores to HBM, so a component makes one
// shared-memory round trip per stage and needs one buffer.  Tasks of all
// components of a tile are spread over the CTA, so small tiles still fill its
// threads; registers stay below the launch bounds (kPassCtas).
//
// K-apply before and after this form replaced two-buffer Stockham tiles (copied in,
// between the buffers per stage and out; odd radices with run-time sines):
//   120 x 100 x 84, FP32, 6 systems   14.28 -> 0.67 ms
//   256^3, FP32, 2 systems            14.26 -> 3.75 ms
//   64^3, FP64, 4 systems              1.73 -> 1.50 ms (bound by FP64 issue)
//   128^3, float-float, 4 systems      7.92 -> 4.61 ms (bound by FP32 issue)
#pragma once

#include "cg.cuh"
#include "common.cuh"
#include "fft.cuh"

namespace bloch {

struct Geo {
    int Nx, Ny, Nz;
    long long V;
    AxisPlan ax[3];
    FastDiv dx, dy;   // division by Nx and by Ny
    // PCG convergence mask: system b is skipped when skip[b * skip_stride] == 0
    // (nullptr: every system runs); blockIdx.y / skip_ncomp is the system of a
    // per-component pass.
    const int* skip = nullptr;
    int skip_stride = 1;
    int skip_ncomp = 1;
    // plan error word: a pass whose staging wait runs out sets it (nullptr: none)
    int* err = nullptr;
};

__device__ __forceinline__ bool sys_idle(const Geo& g, int b) {
    return g.skip != nullptr && g.skip[(size_t)b * g.skip_stride] == 0;
}

// Stiffness table of a grain.  FP32: the packed upper triangle (21 values,
// sym6), padded to 24 so that six 16-byte loads bring it (120 x 100 x 84 x 6:
// 747 -> 735 us against single loads).  Wider types: the full 6 x 6
// table, read in 16-byte pairs.
__host__ __device__ constexpr int sym6(int i, int j) {
    return i <= j ? i * 6 - i * (i - 1) / 2 + (j - i) : j * 6 - j * (j - 1) / 2 + (i - j);
}
template <typename T> constexpr int kCtabRow = sizeof(T) == 4 ? 24 : 36;

// sigma = C_g gamma at one point
template <typename T, typename C>
__device__ __forceinline__ void stress_of(const C (&gam)[6], C (&sig)[6], const T* __restrict__ Cg) {
    if constexpr (std::is_same<T, float>::value) {
        float c[24];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(Cg) + k);
            c[4 * k] = v.x;
            c[4 * k + 1] = v.y;
            c[4 * k + 2] = v.z;
            c[4 * k + 3] = v.w;
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) sig[i] = cscale(gam[i], c[sym6(i, i)]);
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int j = i + 1; j < 6; ++j) {
                const float cij = c[sym6(i, j)];
                sig[i] = mk(fma(cij, gam[j].x, sig[i].x), fma(cij, gam[j].y, sig[i].y));
                sig[j] = mk(fma(cij, gam[i].x, sig[j].x), fma(cij, gam[i].y, sig[j].y));
            }
    } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            T sr = 0, si = 0;
#pragma unroll
            for (int j = 0; j < 6; j += 2) {
                T c0, c1;
                ldg_pair(Cg + i * 6 + j, c0, c1);
                sr = fma(c0, gam[j].x, sr);
                si = fma(c0, gam[j].y, si);
                sr = fma(c1, gam[j + 1].x, sr);
                si = fma(c1, gam[j + 1].y, si);
            }
            sig[i] = mk(sr, si);
        }
    }
}

__host__ __device__ __forceinline__ int pad_even(int n) { return (n + 1) & ~1; }

// Rows of the x passes keep one spare element after every r3 slots when r3 is
// even: the last stage's threads then step by an odd number of elements and
// meet no bank conflicts.  xgroup(a) is the length of such a group, xrow(a)
// that of a row (odd, so that rows are spread too).
__host__ __device__ __forceinline__ int xgroup(const AxisPlan& a) { return a.r3 + ((a.r3 & 1) ^ 1); }
__host__ __device__ __forceinline__ int xrow(const AxisPlan& a) { return (a.r1 * a.r2 * xgroup(a)) | 1; }

// CTAs per SM the pass kernels leave registers for.  FP32 kernels come in two
// forms: with radices up to 12 four CTAs share an SM (64 registers), with the
// wide ones (14 to 16, which would spill) three.  120 x 100 x 84, 6 systems:
// 735 us with three, 680 with four; 256^3 (16 x 16): 3.79 ms with three, 4.27
// with four.
template <typename T, bool WIDE> constexpr int kPassCtas = sizeof(T) != 4 ? 2 : WIDE ? 3 : 4;
// the wide z passes' six-buffer tiles admit two CTAs anyway (256^3: 3.99 ms with
// registers for three, which spill, 3.78 with two)
template <typename T, bool WIDE> constexpr int kPassCtasZ = sizeof(T) != 4 || WIDE ? 2 : 4;

// f(std::integral_constant<int, R>) for the run-time radix R.  Float-float
// leaves out the radices whose code is longest for what they save (compile time).
template <typename T, bool WIDE, typename F>
__device__ __forceinline__ void with_radix(int R, F&& f) {
    switch (R) {
#define BLOCH_RADIX(r) \
    case r: f(std::integral_constant<int, r>{}); break;
        BLOCH_RADIX(1) BLOCH_RADIX(2) BLOCH_RADIX(3) BLOCH_RADIX(4) BLOCH_RADIX(5) BLOCH_RADIX(6) BLOCH_RADIX(7)
        BLOCH_RADIX(8) BLOCH_RADIX(9) BLOCH_RADIX(10)
        default: break;
    }
    if constexpr (!std::is_same<T, dfloat>::value) {
        if (R == 12) f(std::integral_constant<int, 12>{});
    }
    if constexpr (WIDE) {
        switch (R) {
            BLOCH_RADIX(15) BLOCH_RADIX(16)
            default: break;
        }
        if constexpr (!std::is_same<T, dfloat>::value) {
            if (R == 14) f(std::integral_constant<int, 14>{});
        }
    }
}
// Middle radices that a schedule chooses: 4 occurs in float-float only (84 = 3 4 7,
// 7 x 12 in the types that have a 12).
template <typename T, typename F>
__device__ __forceinline__ void with_mid_radix(int R, F&& f) {
    switch (R) {
        BLOCH_RADIX(3) BLOCH_RADIX(5) BLOCH_RADIX(6) BLOCH_RADIX(7) BLOCH_RADIX(8)
        default: break;
    }
    if constexpr (std::is_same<T, dfloat>::value) {
        switch (R) {
            BLOCH_RADIX(4)
#undef BLOCH_RADIX
            default: break;
        }
    }
}

template <typename C> using real_t = decltype(C::x);

// Twiddle table of an axis, in the order the stages read it: w_N^(r j) at
// r (N / r1) + j for the first stage's butterflies j < N / r1, then, with a
// middle stage, w_(r2 r3)^(r n3) at N + r r3 + n3.  Neighbouring threads of the
// x passes take neighbouring j: the natural order w_N^t, read at r j, meets up to
// r-way bank conflicts (worth about 1 % of 120 x 100 x 84 and 4 % of 256^3).
__host__ __device__ __forceinline__ int twtab_len(const AxisPlan& a) { return a.N + (a.r2 > 1 ? a.r2 * a.r3 : 0); }

template <int DIR, typename C>
__device__ __forceinline__ C twiddled(C v, C w) {
    if (DIR > 0) w.y = -w.y;
    return cmul(v, w);
}

// slot of output index k: (k1, k2, k3) with k = k1 + r1 k2 + r1 r2 k3
__device__ __forceinline__ int slot_of(int k, const AxisPlan& a) {
    const int t = (int)fdiv((unsigned)k, a.d1);
    const int k1 = k - t * a.r1;
    const int k3 = (int)fdiv((unsigned)t, a.d2);
    return (k1 * a.r2 + (t - k3 * a.r2)) * a.r3 + k3;
}

// ------------------------------------------------ stages on pencil-fast tiles
// Element (buffer c, slot n, pencil p) at c NP + (n << lp) + p, NP = N << lp.

// middle stage (decimation in frequency) of nbuf buffers, in place
template <int DIR, typename C>
__device__ __forceinline__ void pf_mid(C* buf, int nbuf, const AxisPlan& a, int lp, const C* tw, int tid, int nthr) {
    const int P1 = (1 << lp) - 1, NP = a.N << lp;
    with_mid_radix<real_t<C>>(a.r2, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int per = (a.N / R) << lp, r3 = a.r3;
        for (int t = tid; t < nbuf * per; t += nthr) {
            const int c = t / per, u = t - c * per;
            const int j = u >> lp, k1 = (int)fdiv((unsigned)j, a.d3), n3 = j - k1 * r3;
            C* s = buf + c * NP + ((k1 * R * r3 + n3) << lp) + (u & P1);
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = s[(r * r3) << lp];
            RegDFT<R, DIR, C>::run(v);
            s[0] = v[0];
#pragma unroll
            for (int r = 1; r < R; ++r) s[(r * r3) << lp] = twiddled<DIR>(v[r], tw[a.N + r * a.r3 + n3]);
        }
    });
}

// last stage of nbuf buffers, in place
template <int DIR, bool WIDE, typename C>
__device__ __forceinline__ void pf_last(C* buf, int nbuf, const AxisPlan& a, int lp, int tid, int nthr) {
    const int P1 = (1 << lp) - 1;
    with_radix<real_t<C>, WIDE>(a.r3, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        if constexpr (R > 1) {
            // the buffers are contiguous and N is a multiple of R: one run of butterflies over all of them
            const int total = (nbuf * (a.N / R)) << lp;
            for (int t = tid; t < total; t += nthr) {
                C* s = buf + (((t >> lp) * R) << lp) + (t & P1);
                C v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = s[r << lp];
                RegDFT<R, DIR, C>::run(v);
#pragma unroll
                for (int r = 0; r < R; ++r) s[r << lp] = v[r];
            }
        }
    });
}

// ---------------------------------------------------------------- pass 1
// P = 1 << lp neighbouring pencils per CTA; blockIdx.y = system.  Buffers
// a_x, b_x, a_y, b_y, a_z, b_z; with them the six Voigt strains are
//   g_xx = q_x a_x, g_yy = q_y a_y, g_zz = b_z, g_yz = q_y a_z + b_y,
//   g_xz = q_x a_z + b_x, g_xy = q_y a_x + q_x a_y
// (q_x and q_y are constant on a z pencil).
template <typename T, bool WIDE>
__global__ void __launch_bounds__(256, kPassCtasZ<T, WIDE>)
    k_pass_z_strain(const cplx_t<T>* U, cplx_t<T>* __restrict__ E, const T* qtab, const cplx_t<T>* __restrict__ twz,
                    Geo g, int lp, const CGSys* sys) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const AxisPlan& a = g.ax[2];
    const int N = a.N, NP = N << lp, P1 = (1 << lp) - 1;
    C* tw = reinterpret_cast<C*>(smem_raw);
    const int ntw = twtab_len(a);
    C* buf = tw + pad_even(ntw);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int b = blockIdx.y;
    const unsigned plane = (unsigned)g.Nx * (unsigned)g.Ny;
    const unsigned pi0 = blockIdx.x << lp;
    const int np = (int)min((unsigned)P1 + 1u, plane - pi0);
    const C* Ub = U + (size_t)b * 3 * g.V;
    C* Eb = E + (size_t)b * 6 * g.V;
    const T* qx = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    const T* qy = qx + g.Nx;
    const T* qz = qy + g.Ny;
    // FP32 conjugate gradients: every strain is linear in q, so scaling q scales them all
    T sc = T(1);
    auto qs = [&](T q) {
        if constexpr (sizeof(T) == 4) return q * sc;
        else return q;
    };
    for (int i = tid; i < ntw; i += nthr) tw[i] = twz[i];
    pdl_wait();
    pdl_launch();
    if (sys_idle(g, b)) return;
    if constexpr (sizeof(T) == 4) {
        if (sys) sc = cg_scale<T>(sys, b);
    }
    __syncthreads();
    with_radix<real_t<C>, WIDE>(a.r1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = N / R, per = M << lp;
        for (int t = tid; t < 3 * per; t += nthr) {
            const int c = t / per, u = t - c * per;
            const int p = u & P1, j = u >> lp;
            const bool ok = p < np;
            const C* src = Ub + (size_t)c * g.V + pi0 + (ok ? p : 0) + (size_t)j * plane;
            C* s = buf + 2 * c * NP + u;
            // the scaled transform reads its inputs again (from L1) where the
            // registers cannot hold both; 32-bit indices into the q table (with
            // 64-bit addresses the wide form spills: 256^3 3.84 against 3.75 ms)
            constexpr bool keep = sizeof(T) == 4 && R <= 8;
            C v[R];
            if constexpr (keep) {
                C w[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    v[r] = src[(unsigned)(r * M) * plane];
                    w[r] = cscale(v[r], qs(qz[(unsigned)(r * M + j)]));
                }
                RegDFT<R, +1, C>::run(v);
                RegDFT<R, +1, C>::run(w);
                s[0] = v[0];
                s[NP] = w[0];
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const C f = tw[r * M + j];
                    s[(r * M) << lp] = twiddled<+1>(v[r], f);
                    s[NP + ((r * M) << lp)] = twiddled<+1>(w[r], f);
                }
            } else {
#pragma unroll 1
                for (int h = 0; h < 2; ++h, s += NP) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        v[r] = src[(unsigned)(r * M) * plane];
                        if (h) v[r] = cscale(v[r], qs(qz[(unsigned)(r * M + j)]));
                    }
                    RegDFT<R, +1, C>::run(v);
                    s[0] = v[0];
#pragma unroll
                    for (int r = 1; r < R; ++r) s[(r * M) << lp] = twiddled<+1>(v[r], tw[r * M + j]);
                }
            }
        }
    });
    __syncthreads();
    if (a.r2 > 1) {
        pf_mid<+1>(buf, 6, a, lp, tw, tid, nthr);
        __syncthreads();
    }
    pf_last<+1, WIDE>(buf, 6, a, lp, tid, nthr);
    __syncthreads();
    for (int t = tid; t < NP; t += nthr) {
        const int p = t & P1, k = t >> lp;
        if (p >= np) continue;
        const C* s = buf + (slot_of(k, a) << lp) + p;
        const unsigned pi = pi0 + p, y = fdiv(pi, g.dx);
        const T ax = qs(qx[pi - y * (unsigned)g.Nx]), ay = qs(qy[y]);
        const C a0 = s[0], b0 = s[NP], a1 = s[2 * NP], b1 = s[3 * NP], a2 = s[4 * NP], b2 = s[5 * NP];
        C* d = Eb + (size_t)k * plane + pi;
        d[0] = cscale(a0, ax);
        d[g.V] = cscale(a1, ay);
        d[2 * g.V] = b2;
        d[3 * g.V] = cadd(cscale(a2, ay), b1);
        d[4 * g.V] = cadd(cscale(a2, ax), b0);
        d[5 * g.V] = cadd(cscale(a0, ay), cscale(a1, ax));
    }
}

// ------------------------------------------------- plain FFT pass along y or z
// blockIdx.y enumerates (batch, component) pairs: offset blockIdx.y * V.
template <typename T, int DIR, int AXIS, bool WIDE>
__global__ void __launch_bounds__(256, kPassCtas<T, WIDE>)
    k_pass_axis(const cplx_t<T>* in, cplx_t<T>* out, const cplx_t<T>* __restrict__ twa, Geo g, int lp, T out_scale) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const AxisPlan& a = g.ax[AXIS];
    const int N = a.N, P1 = (1 << lp) - 1;
    C* tw = reinterpret_cast<C*>(smem_raw);
    const int ntw = twtab_len(a);
    C* buf = tw + pad_even(ntw);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const unsigned nx = (unsigned)g.Nx, plane = nx * (unsigned)g.Ny;
    const unsigned step = AXIS == 1 ? nx : plane;     // between the elements of a pencil
    const unsigned npen = AXIS == 1 ? nx * (unsigned)g.Nz : plane;
    const unsigned pi0 = blockIdx.x << lp;
    const C* src = in + (size_t)blockIdx.y * g.V;
    C* dst = out + (size_t)blockIdx.y * g.V;
    // first element of pencil pi
    auto base = [&](unsigned pi) -> size_t {
        if (AXIS == 2) return pi;
        const unsigned z = fdiv(pi, g.dx);
        return (size_t)z * plane + (pi - z * nx);
    };
    for (int i = tid; i < ntw; i += nthr) tw[i] = twa[i];
    pdl_wait();
    pdl_launch();
    if (sys_idle(g, (int)blockIdx.y / g.skip_ncomp)) return;
    __syncthreads();
    with_radix<real_t<C>, WIDE>(a.r1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = N / R;
        for (int t = tid; t < (M << lp); t += nthr) {
            const unsigned pi = min(pi0 + (t & P1), npen - 1);
            const int j = t >> lp;
            const C* s = src + base(pi) + (size_t)j * step;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = s[(unsigned)(r * M) * step];
            RegDFT<R, DIR, C>::run(v);
            buf[t] = v[0];
#pragma unroll
            for (int r = 1; r < R; ++r) buf[((r * M) << lp) + t] = twiddled<DIR>(v[r], tw[r * M + j]);
        }
    });
    __syncthreads();
    if (a.r2 > 1) {
        pf_mid<DIR>(buf, 1, a, lp, tw, tid, nthr);
        __syncthreads();
    }
    with_radix<real_t<C>, WIDE>(a.r3, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = N / R;
        for (int t = tid; t < (M << lp); t += nthr) {
            const unsigned pi = pi0 + (t & P1);
            if (pi >= npen) continue;
            const int k = t >> lp;                    // k1 + r1 k2
            const int k2 = (int)fdiv((unsigned)k, a.d1), k1 = k - k2 * a.r1;
            const C* s = buf + (((k1 * a.r2 + k2) * R) << lp) + (t & P1);
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = s[r << lp];
            RegDFT<R, DIR, C>::run(v);
            C* d = dst + base(pi) + (size_t)k * step;
#pragma unroll
            for (int r = 0; r < R; ++r) d[(unsigned)(r * M) * step] = cscale(v[r], out_scale);
        }
    });
}

// ---------------------------------------------------------------- pass 5
// With CG the divergence A p is not stored: the residual of the conjugate
// gradients is updated with it in place (CgUpdate).
template <typename T, bool WIDE, bool CG>
__global__ void __launch_bounds__(256, kPassCtasZ<T, WIDE>)
    k_pass_z_div(const cplx_t<T>* E, cplx_t<T>* __restrict__ out, const T* qtab, const cplx_t<T>* __restrict__ twz,
                 Geo g, int lp, T out_scale,
                 const __grid_constant__ std::conditional_t<CG, CgUpdate<T>, int> cg) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const AxisPlan& a = g.ax[2];
    const int N = a.N, NP = N << lp, P1 = (1 << lp) - 1;
    C* tw = reinterpret_cast<C*>(smem_raw);
    const int ntw = twtab_len(a);
    C* buf = tw + pad_even(ntw);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int b = blockIdx.y;
    const unsigned plane = (unsigned)g.Nx * (unsigned)g.Ny;
    const unsigned pi0 = blockIdx.x << lp;
    const int np = (int)min((unsigned)P1 + 1u, plane - pi0);
    const C* Eb = E + (size_t)b * 6 * g.V;
    C* ob;
    T alpha = T(0), sc = T(1), sr = T(1), acc[2] = {T(0), T(0)};
    if constexpr (CG) {
        ob = cg.r + (size_t)b * 3 * g.V;
    } else {
        ob = out + (size_t)b * 3 * g.V;
    }
    const T* qx = qtab + (size_t)b * (g.Nx + g.Ny + g.Nz);
    const T* qy = qx + g.Nx;
    const T* qz = qy + g.Ny;
    for (int i = tid; i < ntw; i += nthr) tw[i] = twz[i];
    pdl_wait();
    pdl_launch();
    if (sys_idle(g, b)) return;
    if constexpr (CG) {
        sc = cg_scale<T>(cg.sys, b);
        sr = cg_scale_rr<T>(cg.sys, b);
        alpha = T(cg.sys[b].alpha / (double)sc);
    }
    __syncthreads();
    with_radix<real_t<C>, WIDE>(a.r1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = N / R, per = M << lp;
        for (int t = tid; t < 6 * per; t += nthr) {
            const int c = t / per, u = t - c * per;
            const int p = min(u & P1, np - 1), j = u >> lp;
            const C* src = Eb + (size_t)c * g.V + pi0 + p + (size_t)j * plane;
            C* s = buf + c * NP + u;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = src[(unsigned)(r * M) * plane];
            RegDFT<R, -1, C>::run(v);
            s[0] = v[0];
#pragma unroll
            for (int r = 1; r < R; ++r) s[(r * M) << lp] = twiddled<-1>(v[r], tw[r * M + j]);
        }
    });
    __syncthreads();
    if (a.r2 > 1) {
        pf_mid<-1>(buf, 6, a, lp, tw, tid, nthr);
        __syncthreads();
    }
    pf_last<-1, WIDE>(buf, 6, a, lp, tid, nthr);
    __syncthreads();
    constexpr int U = CG ? 4 : 1;   // voxels whose residuals are in flight together
    for (int t0 = tid; t0 < NP; t0 += U * nthr) {
        C ro[U][3];
        if constexpr (CG) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int t = t0 + u * nthr, p = t & P1, k = t >> lp;
                if (t < NP && p < np) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) ro[u][i] = ob[(size_t)i * g.V + (size_t)k * plane + pi0 + p];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int t = t0 + u * nthr, p = t & P1, k = t >> lp;
            if (t >= NP || p >= np) continue;
            const C* s = buf + (slot_of(k, a) << lp) + p;
            const unsigned pi = pi0 + p, y = fdiv(pi, g.dx);
            const T ax = qx[pi - y * (unsigned)g.Nx], ay = qy[y], az = qz[k];
            const C s0 = s[0], s1 = s[NP], s2 = s[2 * NP], s3 = s[3 * NP], s4 = s[4 * NP], s5 = s[5 * NP];
            const C o[3] = {cadd(cadd(cscale(s0, ax), cscale(s4, az)), cscale(s5, ay)),
                            cadd(cadd(cscale(s1, ay), cscale(s3, az)), cscale(s5, ax)),
                            cadd(cadd(cscale(s2, az), cscale(s3, ay)), cscale(s4, ax))};
            if constexpr (CG) {
                cg_update_at<T>(cg, ob, b, g.V, (unsigned)k * plane + pi, alpha, sc, sr, ax, ay, az, o, ro[u], acc);
            } else {
                C* d = ob + (size_t)k * plane + pi;
                d[0] = cscale(o[0], out_scale);
                d[g.V] = cscale(o[1], out_scale);
                d[2 * g.V] = cscale(o[2], out_scale);
            }
        }
    }
    if constexpr (CG) cg_partial_out<T>(cg, b, acc);
}

// ------------------------------------------------ stages on rows along x
// Element (component c, row p, slot n) at (c P + p) xrow + (n / r3) xgroup + n mod r3.

// stage 1 (decimation in frequency) of ncomp components of P rows, from HBM
template <int DIR, bool WIDE, typename C>
__device__ __forceinline__ void lf_first(const C* Wb, long long V, C* buf, int ncomp, const AxisPlan& a, int P, int nr,
                                         unsigned r0, const C* tw, int tid, int nthr) {
    const int ld = xrow(a), gr = xgroup(a);
    with_radix<real_t<C>, WIDE>(a.r1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = a.N / R, Mg = a.r2 * gr;
        for (int t = tid; t < ncomp * P * M; t += nthr) {
            const int cp = (int)fdiv((unsigned)t, a.m1), j = t - cp * M;
            const int c = cp / P, p = min(cp - c * P, nr - 1);
            const C* src = Wb + (size_t)c * V + (size_t)(r0 + p) * a.N + j;
            C* s = buf + cp * ld + j + (int)fdiv((unsigned)j, a.d3) * (gr - a.r3);
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = src[r * M];
            RegDFT<R, DIR, C>::run(v);
            s[0] = v[0];
#pragma unroll
            for (int r = 1; r < R; ++r) s[r * Mg] = twiddled<DIR>(v[r], tw[r * M + j]);
        }
    });
}

// middle stage: FREQ decimation in frequency (twiddles after), else in time (before)
template <int DIR, bool FREQ, typename C>
__device__ __forceinline__ void lf_mid(C* buf, int nrows, const AxisPlan& a, const C* tw, int tid, int nthr) {
    const int ld = xrow(a), gr = xgroup(a);
    with_mid_radix<real_t<C>>(a.r2, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = a.N / R;
        for (int t = tid; t < nrows * M; t += nthr) {
            const int cp = (int)fdiv((unsigned)t, a.m2), j = t - cp * M;
            const int k1 = (int)fdiv((unsigned)j, a.d3), n3 = j - k1 * a.r3;
            C* s = buf + cp * ld + k1 * R * gr + n3;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r] = s[r * gr];
                if (!FREQ && r > 0) v[r] = twiddled<DIR>(v[r], tw[a.N + r * a.r3 + n3]);
            }
            RegDFT<R, DIR, C>::run(v);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (FREQ && r > 0) v[r] = twiddled<DIR>(v[r], tw[a.N + r * a.r3 + n3]);
                s[r * gr] = v[r];
            }
        }
    });
}

// butterflies over the last digit, in place: the last stage of the inverse
// and the first of the mirrored forward transform
template <int DIR, bool WIDE, typename C>
__device__ __forceinline__ void lf_last(C* buf, int nrows, const AxisPlan& a, int tid, int nthr) {
    const int ld = xrow(a), gr = xgroup(a);
    with_radix<real_t<C>, WIDE>(a.r3, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        if constexpr (R > 1) {
            const int M = a.N / R;
            for (int t = tid; t < nrows * M; t += nthr) {
                const int cp = (int)fdiv((unsigned)t, a.m3);
                C* s = buf + cp * ld + (t - cp * M) * gr;
                C v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = s[r];
                RegDFT<R, DIR, C>::run(v);
#pragma unroll
                for (int r = 0; r < R; ++r) s[r] = v[r];
            }
        }
    });
}

// last stage of the mirrored forward transform, to HBM
template <int DIR, bool WIDE, typename C>
__device__ __forceinline__ void lf_store(C* Wb, long long V, const C* buf, int ncomp, const AxisPlan& a, int P, int nr,
                                         unsigned r0, const C* tw, int tid, int nthr) {
    const int ld = xrow(a), gr = xgroup(a);
    with_radix<real_t<C>, WIDE>(a.r1, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int M = a.N / R, Mg = a.r2 * gr;
        for (int t = tid; t < ncomp * P * M; t += nthr) {
            const int cp = (int)fdiv((unsigned)t, a.m1), j = t - cp * M;
            const int c = cp / P, p = cp - c * P;
            if (p >= nr) continue;
            const C* s = buf + cp * ld + j + (int)fdiv((unsigned)j, a.d3) * (gr - a.r3);
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                v[r] = s[r * Mg];
                if (r > 0) v[r] = twiddled<DIR>(v[r], tw[r * M + j]);
            }
            RegDFT<R, DIR, C>::run(v);
            C* d = Wb + (size_t)c * V + (size_t)(r0 + p) * a.N + j;
#pragma unroll
            for (int r = 0; r < R; ++r) d[r * M] = v[r];
        }
    });
}

// sigma = C_g gamma in place on the six components s[c cs]; with want adds conj(gamma) sigma
template <typename T, typename C>
__device__ __forceinline__ void stress_smem(C* s, int cs, const T* __restrict__ Cg, bool want, T& energy) {
    C gam[6], sig[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) gam[c] = s[c * cs];
    stress_of<T>(gam, sig, Cg);
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i * cs] = sig[i];
    if constexpr (!std::is_same<T, dfloat>::value) {
        if (want) {
#pragma unroll
            for (int i = 0; i < 6; ++i) energy = fma(gam[i].x, sig[i].x, fma(gam[i].y, sig[i].y, energy));
        }
    }
}

// CTA sum of the threads' energies (field precision within a warp, FP64 across)
template <typename T>
__device__ __forceinline__ void energy_out(T e, double2* dst) {
    if constexpr (!std::is_same<T, dfloat>::value) {
        __shared__ double red[32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (double)e;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += red[w];
            *dst = make_double2(t, 0.0);
        }
    }
}

// Row pass along x on P rows per CTA (blockIdx.y = system): inverse FFT,
// pointwise product in real space, forward FFT, in place.
//   NC = 6: strains to stresses with the per-grain table (pass 3)
//   NC = 3: displacements times the per-grain scalar table (mass operator)
// The pointwise step walks a row in real-space order, so a warp meets one or
// two grains and reads their tables once; the odd length of the slot groups
// keeps its strided slots free of bank conflicts.  With dpart
// (NC = 6) the CTA writes its share of the strain energy sum conj(gamma) sigma
// = (u, A_k u) to dpart[b gridDim.x + blockIdx.x] (as k_fpass_x_stress).
template <typename T, int NC, bool WIDE>
__global__ void __launch_bounds__(256, kPassCtas<T, WIDE>)
    k_pass_x_grain(cplx_t<T>* W, const int32_t* __restrict__ ids, const T* __restrict__ tab,
                   const cplx_t<T>* __restrict__ twx, Geo g, int P, double2* __restrict__ dpart) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const AxisPlan& a = g.ax[0];
    const int N = a.N, ld = xrow(a), gr = xgroup(a);
    T energy = T(0);
    C* tw = reinterpret_cast<C*>(smem_raw);
    const int ntw = twtab_len(a);
    C* buf = tw + pad_even(ntw);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int b = blockIdx.y;
    const unsigned rows = (unsigned)g.Ny * (unsigned)g.Nz;
    const unsigned r0 = blockIdx.x * (unsigned)P;
    const int nr = (int)min((unsigned)P, rows - r0);
    C* Wb = W + (size_t)b * NC * g.V;
    for (int i = tid; i < ntw; i += nthr) tw[i] = twx[i];
    pdl_wait();
    pdl_launch();
    if (sys_idle(g, b)) return;
    __syncthreads();
    lf_first<+1, WIDE>(Wb, g.V, buf, NC, a, P, nr, r0, tw, tid, nthr);
    __syncthreads();
    if (a.r2 > 1) {
        lf_mid<+1, true>(buf, NC * P, a, tw, tid, nthr);
        __syncthreads();
    }
    lf_last<+1, WIDE>(buf, NC * P, a, tid, nthr);
    __syncthreads();
    for (int t = tid; t < nr * N; t += nthr) {
        const int p = (int)fdiv((unsigned)t, g.dx), k = t - p * N;
        const int gid = ids[(size_t)(r0 + p) * N + k];
        const int q = (int)fdiv((unsigned)k, a.d1), k3 = (int)fdiv((unsigned)q, a.d2);
        C* s = buf + p * ld + ((k - q * a.r1) * a.r2 + (q - k3 * a.r2)) * gr + k3;   // slot (k1, k2, k3)
        const int cs = P * ld;
        if constexpr (NC == 6) {
            stress_smem<T>(s, cs, tab + (size_t)gid * kCtabRow<T>, dpart != nullptr, energy);
        } else {
            const T r = ldg_t(tab + gid);
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c * cs] = cscale(s[c * cs], r);
        }
    }
    if (NC == 6 && dpart) energy_out(energy, dpart + (size_t)b * gridDim.x + blockIdx.x);
    __syncthreads();
    lf_last<-1, WIDE>(buf, NC * P, a, tid, nthr);
    __syncthreads();
    if (a.r2 > 1) {
        lf_mid<-1, false>(buf, NC * P, a, tw, tid, nthr);
        __syncthreads();
    }
    lf_store<-1, WIDE>(Wb, g.V, buf, NC, a, P, nr, r0, tw, tid, nthr);
}

// ------------------------------------------- plain transform along x
// 1D FFT (DIR -1 forward, +1 inverse, unnormalised) of the three components
// of nb fields along x, in place, times out_scale; rows are contiguous, P
// rows per CTA, blockIdx.y = field.  With ph the fields of system b (`per`
// fields each) are also multiplied by the complex factor ph[b], and the second
// of two fields by 1/2 (the shears of a strain field: engineering to tensor).
template <typename T, int DIR, bool WIDE>
__global__ void __launch_bounds__(256, kPassCtas<T, WIDE>)
    k_pass_x(cplx_t<T>* W, const cplx_t<T>* __restrict__ twx, Geo g, int P, T out_scale,
             const double2* ph, int per) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const AxisPlan& a = g.ax[0];
    const int N = a.N, ld = xrow(a), gr = xgroup(a);
    C* tw = reinterpret_cast<C*>(smem_raw);
    const int ntw = twtab_len(a);
    C* buf = tw + pad_even(ntw);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int b = blockIdx.y;
    const unsigned rows = (unsigned)g.Ny * (unsigned)g.Nz;
    const unsigned r0 = blockIdx.x * (unsigned)P;
    const int nr = (int)min((unsigned)P, rows - r0);
    C* Wb = W + (size_t)b * 3 * g.V;
    for (int i = tid; i < ntw; i += nthr) tw[i] = twx[i];
    pdl_wait();
    pdl_launch();
    if (sys_idle(g, b)) return;
    __syncthreads();
    lf_first<DIR, WIDE>(Wb, g.V, buf, 3, a, P, nr, r0, tw, tid, nthr);
    __syncthreads();
    if (a.r2 > 1) {
        lf_mid<DIR, true>(buf, 3 * P, a, tw, tid, nthr);
        __syncthreads();
    }
    lf_last<DIR, WIDE>(buf, 3 * P, a, tid, nthr);
    __syncthreads();
    if (per == 2 && (b & 1)) out_scale = out_scale * T(0.5);
    const C f = ph ? mk(T(ph[b / per].x) * out_scale, T(ph[b / per].y) * out_scale) : mk(out_scale, T(0));
    for (int t = tid; t < 3 * P * N; t += nthr) {
        const int cp = (int)fdiv((unsigned)t, g.dx), k = t - cp * N;
        const int c = cp / P, p = cp - c * P;
        if (p >= nr) continue;
        const int s = slot_of(k, a);
        const C v = buf[cp * ld + s + (int)fdiv((unsigned)s, a.d3) * (gr - a.r3)];
        Wb[(size_t)c * g.V + (size_t)(r0 + p) * N + k] = ph ? cmul(v, f) : cscale(v, out_scale);
    }
}

}  // namespace bloch
