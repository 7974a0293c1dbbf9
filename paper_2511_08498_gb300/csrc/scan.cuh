// Bounds for the exact early termination (ray_done), found by scanning the records
// before a solve.  They travel in the solve's own output: J of a batch's first
// wavelength, at cells that the solve overwrites, so that no workspace is needed
// and concurrent solves stay independent.
#pragma once

#include "dex_internal.h"

namespace dex {

// The CTA's joined bound, for every thread.
__device__ __forceinline__ float join_cta(float m)
{
    __shared__ float s_m[32];
    for (int o = 16; o > 0; o >>= 1) m = join_bounds(m, __shfl_xor_sync(0xffffffffu, m, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) m = join_bounds(m, s_m[q]);
    return m;
}

}  // namespace dex
