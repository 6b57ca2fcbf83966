// FP64 tracking kernels of the linear map (the kernel template is in kernels_f64.cuh),
// their selection, occupancy and launch, and the sine diagnostics.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "internal.h"
#include "kernels_f64.cuh"
#include "ops_f32c.cuh"
#include "ops_f64.cuh"

namespace phtl {
namespace {

using namespace f64;

template <int S, bool T, bool M>
const void* kernel_ptr(int ppt, int mode)
{
    return ppt == 1 ? kf64::track_kernel<S, T, M, false, false, 1>(mode) : kf64::track_kernel<S, T, M, false>(mode);
}

const void* select_kernel(const MapConsts& c, int scheme, bool trans, bool mon, int ppt)
{
    if (c.general) return general_kernel_single(scheme, PHTL_F64, c.dual_rf != 0, c.rf_mode);
    const int mode = c.rf_mode;
#define PHTL_SEL(S)                                                                                     \
    if (scheme == S) {                                                                                  \
        if (trans) return mon ? kernel_ptr<S, true, true>(ppt, mode) : kernel_ptr<S, true, false>(ppt, mode); \
        return mon ? kernel_ptr<S, false, true>(ppt, mode) : kernel_ptr<S, false, false>(ppt, mode);    \
    }
    PHTL_SEL(PHTL_EULER_CROMER)
    PHTL_SEL(PHTL_LEAPFROG)
    PHTL_SEL(PHTL_RUTH4)
#undef PHTL_SEL
    return nullptr;
}

}  // namespace

// Two particles a thread share the turn's instructions beyond the particles' own and keep the pipes
// busy; one halves what a warp issues in a turn, which is what a bunch too small to fill the SMs
// waits for.  The limits are where the two cross (warps per SM at two particles a thread; us per
// turn, 1 against 2):
//   no planes, no moments   1e4 particles leap-frog 0.46 / 0.75, Ruth4 1.13 / 1.87, Euler-Cromer 0.74 /
//                           0.91; 2e5 1.31 / 1.46; 2.7e5 1.78 / 1.76
//   no planes, moments      1e4 0.84 / 1.19; 6e4 1.32 / 1.40; 8e4 1.59 / 1.56
//   planes                  1e4 0.95 / 1.20 (1.51 / 2.01 with moments); 3e4 1.24 / 1.25; 4.5e4 1.69 / 1.37
// The general map's kernels always take two.
int f64_particles_per_thread(bool trans, bool mon, int gen, int64_t n, int nsm)
{
    const double warps = static_cast<double>(n) / (32.0 * P * std::max(nsm, 1));
    const double limit = trans ? 3.0 : (mon ? 7.0 : 24.0);
    return gen == 0 && warps < limit ? 1 : P;
}

int occupancy_f64(const MapConsts& c, int scheme, bool trans, bool mon, int block, int ppt)
{
    const void* k = select_kernel(c, scheme, trans, mon, ppt);
    if (!k) return 0;
    int nb = 0;
    const size_t smem = mon ? 2u * (block / 32) * 16 * sizeof(double) : 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, block, smem) != cudaSuccess) return 0;
    return nb;
}

cudaError_t launch_track_f64(const LaunchDesc& L, const MapConsts& c, const MonitorArgs& m,
                             cudaStream_t s)
{
    const bool trans = L.c[2] != nullptr || L.c[4] != nullptr;
    const bool mon = m.rows != nullptr;
    const void* k = select_kernel(c, L.scheme, trans, mon, L.ppt);
    if (!k) return cudaErrorInvalidValue;
    const size_t smem = mon ? 2u * (L.block / 32) * 16 * sizeof(double) : 0;
    LaunchDesc Lc = L;
    MapConsts cc = c;
    MonitorArgs mm = m;
    void* args[] = {&Lc, &cc, &mm};
    return cudaLaunchKernel(k, dim3(L.grid), dim3(L.block), args, smem, s);
}

namespace {

__global__ void k_eval_sin(const double* __restrict__ x, double* __restrict__ y, int64_t n,
                           int which)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    {
        if (which == 2) {
            const DF2 r = f32c::sin_df(split_bits(x[i]));
            y[i] = static_cast<double>(r.h) + static_cast<double>(r.l);
        } else {
            y[i] = which == 0 ? sin_f64(x[i]) : sin(x[i]);
        }
    }
}

__global__ void k_eval_sin_kz(double k, PhaseScale kap, const double* __restrict__ z,
                              double* __restrict__ y, int64_t n)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    {
        // kap is |k|'s: sin(k z) = sin(|k| (-z)) for a negative k
        const double u = k < 0.0 ? -z[i] : z[i];
        bool ok;
        const double s = sin_kz_fixed<false>(kap, u, ok);
        y[i] = ok ? s : sin_kz_rest(fabs(k), kap, u);
    }
}

int eval_grid(int64_t n, int block)
{
    const int64_t want = (n + block - 1) / block;
    return static_cast<int>(want < 152 * 16 ? want : 152 * 16);
}

}  // namespace

}  // namespace phtl

extern "C" int phtl_eval_sin(const double* x, double* y, int64_t n, int which, void* stream)
{
    if (n < 0 || which < 0 || which > 2) return PHTL_E_INVALID;
    if (n > 0 && (!x || !y)) return PHTL_E_INVALID;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return PHTL_E_NODEVICE;
    }
    if (n == 0) return PHTL_OK;
    const int block = 256;
    phtl::k_eval_sin<<<phtl::eval_grid(n, block), block, 0, static_cast<cudaStream_t>(stream)>>>(
        x, y, n, which);
    if (cudaGetLastError() != cudaSuccess) return PHTL_E_CUDA;
    return PHTL_OK;
}

extern "C" int phtl_eval_sin_kz(double k, const double* z, double* y, int64_t n, void* stream)
{
    if (n < 0 || !std::isfinite(k)) return PHTL_E_INVALID;
    if (n > 0 && (!z || !y)) return PHTL_E_INVALID;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return PHTL_E_NODEVICE;
    }
    if (n == 0) return PHTL_OK;
    const int block = 256;
    phtl::k_eval_sin_kz<<<phtl::eval_grid(n, block), block, 0, static_cast<cudaStream_t>(stream)>>>(
        k, phtl::phase_scale(std::fabs(k)), z, y, n);
    if (cudaGetLastError() != cudaSuccess) return PHTL_E_CUDA;
    return PHTL_OK;
}
