// Launchers of the mixed-radix passes (passes.cuh), one translation unit per
// field type.
#pragma once

#include <algorithm>

#include "internal.h"

namespace bloch {

template <typename T> static inline const cplx_t<T>* pass_tw(const bloch_plan* pl, int axis);
template <> inline const float2* pass_tw<float>(const bloch_plan* pl, int axis) { return pl->d_mtf[axis]; }
template <> inline const double2* pass_tw<double>(const bloch_plan* pl, int axis) { return pl->d_mtd[axis]; }
template <> inline const dfloat2* pass_tw<dfloat>(const bloch_plan* pl, int axis) { return pl->d_mtx[axis]; }
template <typename T> static inline const T* pass_ctab(const bloch_plan* pl);
template <> inline const float* pass_ctab<float>(const bloch_plan* pl) { return pl->d_Cpf; }
template <> inline const double* pass_ctab<double>(const bloch_plan* pl) { return pl->d_Cd; }
template <> inline const dfloat* pass_ctab<dfloat>(const bloch_plan* pl) { return pl->d_Cx; }
template <typename T> static inline const T* pass_rtab(const bloch_plan* pl);
template <> inline const float* pass_rtab<float>(const bloch_plan* pl) { return pl->d_rf; }
template <> inline const double* pass_rtab<double>(const bloch_plan* pl) { return pl->d_rd; }
template <> inline const dfloat* pass_rtab<dfloat>(const bloch_plan* pl) { return pl->d_rx; }

static inline dim3 pass_grid(long long npen, int lp, int ny) {
    return dim3((unsigned)((npen + (1LL << lp) - 1) >> lp), (unsigned)ny);
}

// whether the schedule of an axis needs the wide-radix kernels (always, but in FP32)
template <typename T>
static inline bool pass_wide(const bloch_plan* pl, int axis) {
    const AxisPlan& a = geo_of<T>(pl).ax[axis];
    return sizeof(T) != 4 || a.r1 > 12 || a.r3 > 12;
}
// f(WIDE) with WIDE a compile-time constant; one form only for the wider types
template <typename T, typename F>
static inline void with_width(const bloch_plan* pl, int axis, F&& f) {
    if constexpr (sizeof(T) == 4) {
        if (!pass_wide<T>(pl, axis)) {
            f(std::false_type{});
            return;
        }
    }
    f(std::true_type{});
}

template <typename T>
void pass_z_strain(bloch_plan* pl, int nb, const cplx_t<T>* u, cplx_t<T>* E, const T* qtab, const CGSys* sys) {
    const PassTile t = pass_tile<T>(pl, PASS_Z6, nb);
    ++pl->launches;
    with_width<T>(pl, 2, [&](auto w) {
        launch_pdl(k_pass_z_strain<T, decltype(w)::value>, pass_grid((long long)pl->Nx * pl->Ny, t.lp, nb), t.nthr,
                   t.smem, pl->stream,
                u, E, qtab, pass_tw<T>(pl, 2), geo_of<T>(pl), t.lp, sys);
    });
}

template <typename T>
void pass_axis(bloch_plan* pl, int axis, int dir, int nfields, const cplx_t<T>* in, cplx_t<T>* out, T out_scale) {
    const PassTile t = pass_tile<T>(pl, axis == 1 ? PASS_Y1 : PASS_Z1, nfields);
    const dim3 gr = pass_grid((long long)pl->Nx * (axis == 1 ? pl->Nz : pl->Ny), t.lp, nfields);
    const Geo& g = geo_of<T>(pl);
    const cplx_t<T>* tw = pass_tw<T>(pl, axis);
    ++pl->launches;
    with_width<T>(pl, axis, [&](auto w) {
        constexpr bool W = decltype(w)::value;
        if (axis == 1 && dir > 0)
            launch_pdl(k_pass_axis<T, +1, 1, W>, gr, t.nthr, t.smem, pl->stream, in, out, tw, g, t.lp, out_scale);
        else if (axis == 1)
            launch_pdl(k_pass_axis<T, -1, 1, W>, gr, t.nthr, t.smem, pl->stream, in, out, tw, g, t.lp, out_scale);
        else if (dir > 0)
            launch_pdl(k_pass_axis<T, +1, 2, W>, gr, t.nthr, t.smem, pl->stream, in, out, tw, g, t.lp, out_scale);
        else
            launch_pdl(k_pass_axis<T, -1, 2, W>, gr, t.nthr, t.smem, pl->stream, in, out, tw, g, t.lp, out_scale);
    });
}

template <typename T>
int pass_x_stress(bloch_plan* pl, int nb, cplx_t<T>* E, double2* dpart) {
    const PassTile t = pass_tile<T>(pl, PASS_X6, nb);
    const dim3 gr = pass_grid((long long)pl->Ny * pl->Nz, t.lp, nb);
    ++pl->launches;
    with_width<T>(pl, 0, [&](auto w) {
        launch_pdl(k_pass_x_grain<T, 6, decltype(w)::value>, gr, t.nthr, t.smem, pl->stream,
            E, pl->d_ids, pass_ctab<T>(pl), pass_tw<T>(pl, 0), geo_of<T>(pl), 1 << t.lp, dpart);
    });
    return (int)gr.x;
}

template <typename T>
void pass_x_rho(bloch_plan* pl, int nb, cplx_t<T>* W) {
    const PassTile t = pass_tile<T>(pl, PASS_X3, nb);
    ++pl->launches;
    with_width<T>(pl, 0, [&](auto w) {
        launch_pdl(k_pass_x_grain<T, 3, decltype(w)::value>, pass_grid((long long)pl->Ny * pl->Nz, t.lp, nb),
                   t.nthr, t.smem, pl->stream,
                W, pl->d_ids, pass_rtab<T>(pl), pass_tw<T>(pl, 0), geo_of<T>(pl), 1 << t.lp, nullptr);
    });
}

template <typename T>
void pass_x(bloch_plan* pl, int dir, int nb, cplx_t<T>* W, T out_scale, const double2* ph, int per) {
    const PassTile t = pass_tile<T>(pl, PASS_X3, nb);
    const dim3 gr = pass_grid((long long)pl->Ny * pl->Nz, t.lp, nb);
    const cplx_t<T>* tw = pass_tw<T>(pl, 0);
    const Geo& g = geo_of<T>(pl);
    ++pl->launches;
    with_width<T>(pl, 0, [&](auto w) {
        constexpr bool WD = decltype(w)::value;
        if (dir > 0)
            launch_pdl(k_pass_x<T, +1, WD>, gr, t.nthr, t.smem, pl->stream, W, tw, g, 1 << t.lp, out_scale, ph, per);
        else
            launch_pdl(k_pass_x<T, -1, WD>, gr, t.nthr, t.smem, pl->stream, W, tw, g, 1 << t.lp, out_scale, ph, per);
    });
}

template <typename T>
int pass_z_div(bloch_plan* pl, int nb, const cplx_t<T>* E, cplx_t<T>* out, const T* qtab, T out_scale,
               const CgUpdate<T>* cg) {
    const PassTile t = pass_tile<T>(pl, PASS_Z6, nb);
    const dim3 gr = pass_grid((long long)pl->Nx * pl->Ny, t.lp, nb);
    ++pl->launches;
    with_width<T>(pl, 2, [&](auto w) {
        constexpr bool W = decltype(w)::value;
        if constexpr (!std::is_same<T, dfloat>::value) {
            if (cg) {
                launch_pdl(k_pass_z_div<T, W, true>, gr, t.nthr, t.smem, pl->stream, E, nullptr, qtab,
                           pass_tw<T>(pl, 2),
                                                                             geo_of<T>(pl), t.lp, out_scale, *cg);
                return;
            }
        }
        launch_pdl(k_pass_z_div<T, W, false>, gr, t.nthr, t.smem, pl->stream, E, out, qtab, pass_tw<T>(pl, 2),
                   geo_of<T>(pl), t.lp, out_scale, 0);
    });
    return (int)gr.x;
}

// shared-memory limits of both forms
template <typename T, typename F>
static cudaError_t each_width(F&& f) {
    cudaError_t e = f(std::true_type{});
    if constexpr (sizeof(T) == 4) {
        if (e == cudaSuccess) e = f(std::false_type{});
    }
    return e;
}
template <typename T>
cudaError_t pass_attrs_z() {
    return each_width<T>([](auto w) {
        constexpr bool W = decltype(w)::value;
        cudaError_t e = allow_max_dyn_smem(k_pass_z_strain<T, W>);
        if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_z_div<T, W, false>);
        if constexpr (!std::is_same<T, dfloat>::value) {
            if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_z_div<T, W, true>);
        }
        return e;
    });
}
template <typename T>
cudaError_t pass_attrs_axis() {
    return each_width<T>([](auto w) {
        constexpr bool W = decltype(w)::value;
        cudaError_t e = allow_max_dyn_smem(k_pass_axis<T, +1, 1, W>);
        if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_axis<T, -1, 1, W>);
        if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_axis<T, +1, 2, W>);
        return e == cudaSuccess ? allow_max_dyn_smem(k_pass_axis<T, -1, 2, W>) : e;
    });
}
template <typename T>
cudaError_t pass_attrs_x() {
    return each_width<T>([](auto w) {
        constexpr bool W = decltype(w)::value;
        cudaError_t e = allow_max_dyn_smem(k_pass_x_grain<T, 6, W>);
        if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_x_grain<T, 3, W>);
        if constexpr (!std::is_same<T, dfloat>::value) {
            if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_x<T, +1, W>);
            if (e == cudaSuccess) e = allow_max_dyn_smem(k_pass_x<T, -1, W>);
        }
        return e;
    });
}

#define BLOCH_INST_PASSES_Z(T)                                                                            \
    template void pass_z_strain<T>(bloch_plan*, int, const cplx_t<T>*, cplx_t<T>*, const T*, const CGSys*); \
    template int pass_z_div<T>(bloch_plan*, int, const cplx_t<T>*, cplx_t<T>*, const T*, T,               \
                               const CgUpdate<T>*);                                                      \
    template cudaError_t pass_attrs_z<T>();
#define BLOCH_INST_PASSES_AXIS(T)                                                                         \
    template void pass_axis<T>(bloch_plan*, int, int, int, const cplx_t<T>*, cplx_t<T>*, T);              \
    template cudaError_t pass_attrs_axis<T>();
#define BLOCH_INST_PASSES_X(T)                                                                            \
    template int pass_x_stress<T>(bloch_plan*, int, cplx_t<T>*, double2*);                                \
    template void pass_x_rho<T>(bloch_plan*, int, cplx_t<T>*);                                            \
    template cudaError_t pass_attrs_x<T>();

}  // namespace bloch
