// Per-turn bunch-moment reduction shared by the tracking kernels.
//
// Each thread holds NF partial sums (field j of a monitor row, see phtl.h): 64-bit integers
// in the FP64 kernels (ops_f64.cuh), floats in the FP32 ones (ops_f32c.cuh).  A warp
// reduce-scatter halves the number of fields per lane at every butterfly step, so a
// lane performs NF adds in total instead of 5*NF for NF independent butterflies.  After the
// scatter, lane L holds the warp total of field L / (32 / NF).  The warps' totals meet in
// shared memory (double-buffered by record parity, so one __syncthreads per record
// suffices) and warp 0 adds them up and issues one FP64 atomicAdd per field.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "phtl.h"

namespace phtl {

constexpr unsigned kFullMask = 0xffffffffu;

// Reduce-scatter NF fields (NF in {8, 16}) of 64-bit integer partial sums (exact, so the order of
// the additions is free) across the warp; returns this lane's field total.  Which field:
// NF == 16 -> lane >> 1, NF == 8 -> lane >> 2.
template <int NF>
__device__ __forceinline__ int64_t warp_reduce_scatter_int(int64_t (&f)[NF], int lane)
{
    static_assert(NF == 8 || NF == 16, "NF must be 8 or 16");
#pragma unroll
    for (int o = 16; o >= (NF == 16 ? 2 : 4); o >>= 1) {
        const int h = (NF == 16) ? (o >> 1) : (o >> 2);
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < NF / 2; ++i) {
            if (i < h) {
                const int64_t send = upper ? f[i] : f[i + h];
                const int64_t keep = upper ? f[i + h] : f[i];
                f[i] = keep + __shfl_xor_sync(kFullMask, static_cast<long long>(send), o);
            }
        }
    }
    int64_t v = f[0];
    if (NF == 8) v += __shfl_xor_sync(kFullMask, static_cast<long long>(v), 2);
    v += __shfl_xor_sync(kFullMask, static_cast<long long>(v), 1);
    return v;
}

}  // namespace phtl
