// Bounds for the exact early termination (ray_done), found by scanning the records
// before a solve.  They travel in the solve's own output: J of a batch's first
// wavelength, at cells that the solve overwrites, so that no workspace is needed
// and concurrent solves stay independent.
#pragma once

#include "hdda.cuh"

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

namespace {

// Bound over the W wavelengths of float32, bfloat16 or float16 bricks: every
// record of a block's chain, all levels.
template <int W, int ST>
__device__ __forceinline__ float chain_bound(const float* __restrict__ brick, int chain)
{
    using BF = BrickFmt<W, ST>;
    float m = 0.0f;
    for (int v = threadIdx.x; v < chain; v += blockDim.x) {
        int level = 0;
        while (level < 4 && v >= level_offset(level + 1)) ++level;
        const int side = DEX_BLOCK >> level, q = v - level_offset(level);
        const Record<W> r =
            BF::load(brick + BF::offset(level_offset(level), q / side, q % side, side), BF::chi_off(side));
#pragma unroll
        for (int w = 0; w < W; ++w) m = join_bounds(m, bound_of(r.S[w], r.chi[w]));
    }
    return m;
}

// CTA (a, b): the bound of active block a and batch b, to the block's first cell.
template <int W, int ST>
__global__ void __launch_bounds__(128) k_scan_bricks(const HddaParams P)
{
    const int a = blockIdx.x, b = blockIdx.y;
    if (a >= *P.n_active) return;
    const float* brick = P.bricks + ((size_t)b * P.cap_active + a) * P.chain * RecFmt<W, ST>::kStride;
    const float m = join_cta(chain_bound<W, ST>(brick, P.chain));
    const int blk = P.active[a];
    if (threadIdx.x == 0)
        P.J[(size_t)(b * W) * P.n_cells + (size_t)(blk / P.nbx * DEX_BLOCK) * P.nx + blk % P.nbx * DEX_BLOCK] = m;
}

// Every cell of every active block gets the batch's bound.  First cells that
// another CTA has filled already hold the maximum itself, so reading them in
// place of their block's bound changes nothing.
__global__ void __launch_bounds__(256) k_spread_bounds(const HddaParams P)
{
    float* J = P.J + (size_t)(blockIdx.y * P.W) * P.n_cells;
    const int na = *P.n_active;
    float m = 0.0f;
    for (int a = threadIdx.x; a < na; a += blockDim.x) {
        const int blk = P.active[a];
        m = join_bounds(m, __ldcg(J + (size_t)(blk / P.nbx * DEX_BLOCK) * P.nx + blk % P.nbx * DEX_BLOCK));
    }
    m = join_cta(m);
    for (int a = blockIdx.x; a < na; a += gridDim.x) {
        const int blk = P.active[a];
        J[(size_t)(blk / P.nbx * DEX_BLOCK + (threadIdx.x >> 4)) * P.nx + blk % P.nbx * DEX_BLOCK + (threadIdx.x & 15)] = m;
    }
}

inline void launch_spread(cudaStream_t s, const HddaParams& P)
{
    const int ctas = P.cap_active < 152 ? P.cap_active : 152;
    k_spread_bounds<<<dim3((unsigned)ctas, (unsigned)P.n_batch), 256, 0, s>>>(P);
}

}  // namespace
}  // namespace dex
