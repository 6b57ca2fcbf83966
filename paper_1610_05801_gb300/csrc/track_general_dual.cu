// Single-bunch kernels of the widened map with the second RF system (double RF): the
// widened map's kernel templates with DUAL = true, kept apart so that rings without a
// second system run kernels without its code (fewer registers).  FP64 and PHTL_F32C here,
// PHTL_F32CD and PHTL_F32CS in track_general_dual_f32.cu (they build in parallel).
#include <cuda_runtime.h>

#include "internal.h"
#include "kernels_f64.cuh"

namespace phtl {
const void* general_kernel_single_dual(int scheme, int dtype, int mode)
{
    if (dtype != PHTL_F64) return general_kernel_single_dual_f32(scheme, dtype);
    if (scheme == PHTL_EULER_CROMER) return kf64::track_kernel<PHTL_EULER_CROMER, true, true, true, true>(mode);
    if (scheme == PHTL_LEAPFROG) return kf64::track_kernel<PHTL_LEAPFROG, true, true, true, true>(mode);
    if (scheme == PHTL_RUTH4) return kf64::track_kernel<PHTL_RUTH4, true, true, true, true>(mode);
    if (scheme == PHTL_RK4) return kf64::track_kernel<PHTL_RK4, true, true, true, true>(mode);
    return nullptr;
}

}  // namespace phtl
