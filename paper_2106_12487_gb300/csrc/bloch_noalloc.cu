// Allocation-free variant of the stiffness operator apply.
//
// bloch_apply_K runs its FFT passes through a plan-owned scratch buffer that
// grows with cudaMalloc the first time a larger batch is seen.  Callers that
// may not allocate device memory at the point of the call (services with a
// fixed device-memory budget, code embedded in a framework that owns the
// allocator, real-time loops in which an allocator call may stall the
// device) use bloch_apply_K_noalloc
// instead: its scratch is one file-scope device array of fixed size.  The
// array is placed on a device when this file's module is loaded there --
// with CUDA's lazy module loading, at the first call of the entry point on
// that device -- and held until the process exits.  The operator, its kernels
// (the same pass kernels and launch shapes) and its results are those of
// bloch_apply_K in FP32.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "internal.h"

namespace bloch {

// Scratch layout inside the one static array: the six-component FFT-pass
// intermediates (6 x V x nb float2) first, then the per-system q tables
// ((Nx+Ny+Nz) x nb float) and the wave vectors (3 x nb double).
constexpr size_t kNoAllocPassBytes = (size_t)96 << 20;   // 96 MiB: nb*V <= 2^21 (one 128^3 system)
constexpr size_t kNoAllocTableBytes = (size_t)1 << 20;   // 1 MiB for q tables and wave vectors
constexpr size_t kNoAllocBytes = kNoAllocPassBytes + kNoAllocTableBytes;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Set-up, once per device (with that device current): the device address of
// the scratch array (the pass kernels' attributes are the plan's).
constexpr int kMaxDevices = 64;
static void* g_noalloc_ptr[kMaxDevices] = {nullptr};
static std::mutex g_noalloc_mu;

static bloch_status noalloc_scratch(void** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_cuda_error(e, "cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) return set_error(BLOCH_EUNSUPPORTED, "device index above 63");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return set_cuda_error(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return BLOCH_OK;
}

}  // namespace bloch

using namespace bloch;

extern "C" bloch_status bloch_apply_K_noalloc(bloch_plan* pl, int32_t nb, const double* k, const void* u, void* Ku) {
    if (!pl) return set_error(BLOCH_EINVAL, "plan is NULL");
    if (!k || !u || !Ku) return set_error(BLOCH_EINVAL, "NULL argument");
    if (u == Ku) return set_error(BLOCH_EINVAL, "Ku may not alias u");
    // the y passes launch 6 * nb CTA rows (gridDim.y <= 65535), as in bloch_apply_K
    if (nb < 1 || nb > 65535 / 6) return set_error(BLOCH_EINVAL, "nb must be in [1, 10922]");
    if (!pl->fast) return set_error(BLOCH_EUNSUPPORTED, "bloch_apply_K_noalloc runs the default FFT variant only");
    const size_t pass_bytes = (size_t)6 * (size_t)pl->V * (size_t)nb * sizeof(float2);
    if (pass_bytes > kNoAllocPassBytes)
        return set_error(BLOCH_EINVAL, "bloch_apply_K_noalloc: nb * V = " + std::to_string((long long)nb * pl->V) +
                                           " exceeds its fixed scratch (nb * V <= 2097152)");
    const int S = pl->Nx + pl->Ny + pl->Nz;
    const size_t q_bytes = ((size_t)S * nb * sizeof(float) + 255) / 256 * 256;
    const size_t k_bytes = (size_t)3 * nb * sizeof(double);
    if (q_bytes + k_bytes > kNoAllocTableBytes)
        return set_error(BLOCH_EINVAL, "bloch_apply_K_noalloc: (Nx+Ny+Nz+6) * nb exceeds its 1 MiB table scratch");
    for (int i = 0; i < 3 * nb; ++i)
        if (!std::isfinite(k[i])) return set_error(BLOCH_ENONFINITE, "wave vector has a non-finite component");

    void* base = nullptr;
    bloch_status st = noalloc_scratch(&base);
    if (st != BLOCH_OK) return st;
    unsigned char* b = (unsigned char*)base;
    float2* E = (float2*)b;
    float* qtab = (float*)(b + kNoAllocPassBytes);
    double* kvec = (double*)(b + kNoAllocPassBytes + q_bytes);

    if ((st = launch_qtab<float>(pl, nb, k, kvec, qtab)) != BLOCH_OK) return st;
    launch_K_on(pl, nb, (const float2*)u, E, qtab, (float2*)Ku, (float)pl->Kscale);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(e, "bloch_apply_K_noalloc launch");
    return BLOCH_OK;
}
