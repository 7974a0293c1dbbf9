// Hierarchical DDA formal solver with one walk per ray for a pair of
// wavelength batches (Section 2.3, Algorithm 1 with Section 2.3.1; Section
// 4.1's wavelength batches and distance limits; Eq. RteIntegral per segment).
//
// The per-batch solver (k_hdda.cu) traces every ray once per batch of 8
// wavelengths, and about two thirds of its instructions are the walk: plane
// arithmetic, block crossings and level look-ups.  Here one thread carries the
// 16 wavelengths of two batches along one walk and integrates both batches'
// records of every voxel it leaves.  The batches pair mirror-wise within
// consecutive groups (pair_batches: b with n_batch - 1 - b for one group of all
// batches; a line's own batches when each group is one line's samples).  A
// line's batches lie symmetrically about its centre, so the two batches of a
// pair see the same part of the profile and tend to take the same levels (on
// the benchmark's static-line atmosphere every block's levels agree); the walk
// uses, in every block, the smaller of the two levels (Section 2.2), capped by
// the distance limits as usual.  No batch is integrated more coarsely than at
// its own levels.
//
// The walk and the update are those of k_solve_hdda_t (trace_ray) with a
// two-record voxel model; J and I equal, bit for bit, those of the per-batch
// walk given state words that hold the pair's minimum for both batches.  The
// middle batch of a group of odd size is solved by the per-batch walk.
#include "hdda.cuh"

namespace dex {

namespace {

// Launch shape per brick format.  The pair's state (16 intensities and
// transmissions, two records loaded at the top of each step) takes about 125
// registers with float32 records: 2 CTAs of 256 threads per SM.  Bfloat16
// records hold half the registers and run at 5 CTAs of 128 threads (at most 102
// registers).  Measured on the 1024^2 static-line solve at IoD 1e-2, float32 on
// brick rows (the whole step, of which the solve is about 94%):
//   256 threads, 2 CTAs (this)  94.9 ms     128 threads, 5 CTAs (96 registers)  98.2 ms
//   128 threads, 4 CTAs         93.9        64 threads, 8 CTAs                  93.6
// (every CTA stages the block table, 64 KB on the largest grids, of which two fit).
// The bound: issue slots 63% and the FP32 pipe 58% busy at 16 warps, with 25 of 32
// lanes active.  Before rays ended early on the bound of what is left the order was the
// same, 158.8 ms for this shape and 294 ms at 3 CTAs (80 registers, spills); bfloat16
// 165.0 (this), 171.5 at 256 threads and 2 CTAs, 174.3 at 128 and 6.
template <int ST>
constexpr int pair_threads() { return ST == kStoreBF16 ? 128 : 256; }
template <int ST>
constexpr int pair_min_blocks() { return ST == kStoreBF16 ? 5 : 2; }
// probes per CTA: 16 x (threads / 16) rows of a block; CTAs per active block and pair
template <int ST>
constexpr int pair_parts() { return DEX_BLOCK * DEX_BLOCK / pair_threads<ST>(); }

template <int ST>
using PairModel = PairRecModel<ST, pair_min_blocks<ST>()>;

// EXT: each probe's own-voxel emission is left out (the first segment of every
// ray, as k_solve_hdda_t with EXT).
// SPLIT: a CTA's warps share the directions of one 8 x 4 tile (split_solve).
// TWIN: for the solve that walks once per batch: only pairs whose blocks all have
// the same levels (states_agree), for which the shared walk is each batch's own.
// Where a batch's records have no bound (a source function that overflowed, say) each
// batch is walked by itself, as a pair with itself: there a ray must end where its
// own batch's transmissions do.
template <int ST, bool COUNT, bool EXT, bool SPLIT, bool TWIN = false>
__global__ void __launch_bounds__(pair_threads<ST>(), pair_min_blocks<ST>()) k_solve_hdda_pair(const HddaParams P)
{
    using Model = PairModel<ST>;
    constexpr int kParts = SPLIT ? 8 : pair_parts<ST>(), NW = pair_threads<ST>() / 32;
    extern __shared__ int s_info[];
    __shared__ float s_J[SPLIT ? 1 : 16][pair_threads<ST>()];
    __shared__ int s_box[4];
    const int a0 = blockIdx.x / kParts, part = blockIdx.x - a0 * kParts;
    if (a0 >= *P.n_active) return;
    int b1, b2;
    pair_batches(blockIdx.y, P.n_batch, P.pair_group, b1, b2);
    const int tid = threadIdx.x;
    const unsigned long long* w1 = P.words + (size_t)b1 * P.n_words;
    const unsigned long long* w2 = P.words + (size_t)b2 * P.n_words;
    if constexpr (TWIN) {
        if (*P.n_active < P.twins || (P.active_to && *P.n_active >= P.active_to)) return;
        if (!states_agree(w1, w2, P.n_words)) return;
    }
    const int n_blocks = P.nbx * P.nbz;
    for (int q = tid; q < n_blocks; q += blockDim.x)
        s_info[q] = pack_block_info(P.block_offset[q], min(block_state(w1, q), block_state(w2, q)));
    if constexpr (!SPLIT) {
#pragma unroll
        for (int w = 0; w < 16; ++w) s_J[w][tid] = 0.0f;
    }
    if (tid < 4) s_box[tid] = (tid & 1) ? -1 : 0x7fffffff;
    __syncthreads();
    {
        // box around the non-empty blocks, in block units
        int xlo = 0x7fffffff, xhi = -1, zlo = 0x7fffffff, zhi = -1;
        const int na = *P.n_active;
        for (int q = tid; q < na; q += blockDim.x) {
            const int blk = P.active[q];
            const int bz = blk / P.nbx, bx = blk - bz * P.nbx;
            xlo = min(xlo, bx);
            xhi = max(xhi, bx);
            zlo = min(zlo, bz);
            zhi = max(zhi, bz);
        }
        xlo = __reduce_min_sync(0xffffffffu, xlo);
        xhi = __reduce_max_sync(0xffffffffu, xhi);
        zlo = __reduce_min_sync(0xffffffffu, zlo);
        zhi = __reduce_max_sync(0xffffffffu, zhi);
        if ((tid & 31) == 0) {
            atomicMin(&s_box[0], xlo);
            atomicMax(&s_box[1], xhi);
            atomicMin(&s_box[2], zlo);
            atomicMax(&s_box[3], zhi);
        }
    }
    __syncthreads();

    const int blk0 = P.active[a0];
    const int bx0 = blk0 % P.nbx, bz0 = blk0 / P.nbx;
    // the CTA's probes: rows part * (16 / kParts) .. of the block; warp w covers an
    // 8 x 4 tile of them (as in k_solve_hdda_t)
    const int wrp = tid >> 5, lane = tid & 31, tile = SPLIT ? part : part * NW + wrp;
    const int i = bx0 * DEX_BLOCK + (tile & 1) * 8 + (lane & 7);
    const int j = bz0 * DEX_BLOCK + (tile >> 1) * 4 + (lane >> 3);
    const size_t cell = (size_t)j * P.nx + i;
    const int state0 = (s_info[blk0] & 7) - 1;
    if (state0 < 0) {  // state words do not describe this active block
        raise_status(P.status, DEX_ERR_TRAVERSAL_CAP);
        if (P.scanned) P.J[(size_t)(b1 * 8) * P.n_cells + cell] = P.J[(size_t)(b2 * 8) * P.n_cells + cell] = 0.0f;  // the bounds
        return;
    }
    const size_t batch_floats = (size_t)P.cap_active * P.chain * Model::kStride;
    Geo G;
    G.nx = P.nx;
    G.nz = P.nz;
    G.nbx = P.nbx;
    G.nbz = P.nbz;
    G.chain = P.chain;
    G.cap_active = P.cap_active;
    G.batch_base = P.bricks + (size_t)b1 * batch_floats;
    G.x_lo = s_box[0] * DEX_BLOCK;
    G.x_hi = (s_box[1] + 1) * DEX_BLOCK;
    G.z_lo = s_box[2] * DEX_BLOCK;
    G.z_hi = (s_box[3] + 1) * DEX_BLOCK;
#pragma unroll
    for (int q = 0; q < 4; ++q) G.band[q] = P.band[q];
    G.stop = -1.0f;
    [[maybe_unused]] float bound1 = 0.0f, bound2 = 0.0f;
    if (!COUNT && P.scanned) {
        bound1 = P.J[(size_t)(b1 * 8) * P.n_cells + cell];
        bound2 = P.J[(size_t)(b2 * 8) * P.n_cells + cell];
        G.stop = stop_factor(join_bounds(bound1, bound2), P.i_bc);
    }
    typename Model::Params M{(long long)(b2 - b1) * (long long)batch_floats};
    const int mip0 = min(state0, distance_cap(G, 0.0f));
    unsigned int nseg = 0;
    bool capped = false;

    auto ray = [&](int k, float* I, float* T) {
#pragma unroll
        for (int w = 0; w < 16; ++w) {
            I[w] = 0.0f;
            T[w] = 1.0f;
        }
        trace_ray<16, COUNT, Model, InfoLookup, EXT>(G, M, b1, i, j, bx0, bz0, a0, mip0, P.quad.dx[k], P.quad.dz[k],
                                                     InfoLookup{s_info}, I, T, nseg, capped);
    };
    auto lambda = [&](int w) { return w < 8 ? b1 * 8 + w : b2 * 8 + (w - 8); };
    auto store_I = [&](int w, int k, float Iw) {
        if (P.I != nullptr && lambda(w) < P.n_lambda)
            P.I[((size_t)lambda(w) * P.quad.n_dir + k) * P.n_cells + cell] = Iw;
    };
    [[maybe_unused]] __shared__ int s_next;
    auto solve = [&]() {
        if constexpr (SPLIT) {
            split_solve<16, NW>(
                P.quad, reinterpret_cast<float*>(s_info) + P.split_at, &s_next, wrp, lane,
                [&](int k, float* out) {
                    float I[16], T[16];
                    ray(k, I, T);
#pragma unroll
                    for (int w = 0; w < 16; ++w) {
                        const float Iw = fmaf(T[w], P.i_bc, I[w]);
                        out[w * 32] = Iw;
                        store_I(w, k, Iw);
                    }
                },
                [&](int w, float J) {
                    if (lambda(w) < P.n_lambda) P.J[(size_t)lambda(w) * P.n_cells + cell] = J;
                });
        } else {
            for (int k = 0; k < P.quad.n_dir; ++k) {
                float I[16], T[16];
                ray(k, I, T);
                const float wk = P.quad.w[k];
#pragma unroll
                for (int w = 0; w < 16; ++w) {
                    const float Iw = fmaf(T[w], P.i_bc, I[w]);
                    s_J[w][tid] = fmaf(wk, Iw, s_J[w][tid]);
                    store_I(w, k, Iw);
                }
            }
#pragma unroll
            for (int w = 0; w < 16; ++w)
                if (lambda(w) < P.n_lambda) P.J[(size_t)lambda(w) * P.n_cells + cell] = s_J[w][tid];
        }
    };
    if constexpr (TWIN) {
        const int second = b2;
        const long long off = M.off;
        bool apart = join_bounds(bound1, bound2) < 0.0f;
        if (apart) {
            b2 = b1;
            M.off = 0;
            G.stop = stop_factor(bound1, P.i_bc);
        }
        for (;;) {
            solve();
            if (!apart) break;
            apart = false;
            b1 = b2 = second;
            G.batch_base += off;
            G.stop = stop_factor(bound2, P.i_bc);
            if constexpr (!SPLIT) {
#pragma unroll
                for (int w = 0; w < 16; ++w) s_J[w][tid] = 0.0f;
            }
        }
    } else {
        solve();
    }
    if (capped) raise_status(P.status, DEX_ERR_TRAVERSAL_CAP);
    // segments of the two batches
    if (COUNT && P.seg_count != nullptr) atomicAdd(P.seg_count, 2ull * nseg);
}

template <int ST>
cudaError_t launch_pair(cudaStream_t s, const HddaParams& P0, bool twin = false, bool twin_split = false)
{
    HddaParams P = P0;
    const unsigned pairs = (unsigned)pair_count(P.n_batch, P.pair_group);
    P.split_at = (P.nbx * P.nbz + 3) & ~3;
    const bool split = twin ? twin_split : split_directions(P);
    const int blocks = P.active_to ? min(P.active_to, P.cap_active) : P.cap_active;
    const size_t smem = sizeof(int) * (size_t)P.split_at + (split ? split_bytes<16>() : 0);
    const dim3 grid((unsigned)blocks * (split ? 8u : (unsigned)pair_parts<ST>()), pairs);
    auto kernel = P.seg_count ? (P.exclude_own ? k_solve_hdda_pair<ST, true, true, false>
                                               : k_solve_hdda_pair<ST, true, false, false>)
                  : twin      ? (split ? k_solve_hdda_pair<ST, false, false, true, true>
                                       : k_solve_hdda_pair<ST, false, false, false, true>)
                  : split     ? (P.exclude_own ? k_solve_hdda_pair<ST, false, true, true>
                                               : k_solve_hdda_pair<ST, false, false, true>)
                              : (P.exclude_own ? k_solve_hdda_pair<ST, false, true, false>
                                               : k_solve_hdda_pair<ST, false, false, false>);
    if (smem > 24 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kernel<<<grid, pair_threads<ST>(), smem, s>>>(P);
    return cudaGetLastError();
}

}  // namespace

bool solve_hdda_paired_applies(const HddaParams& P)
{
    const long long n_blocks = (long long)P.nbx * P.nbz;
    return P.traversal == DEX_TRAVERSAL_PAIRED && P.W == 8 && n_blocks <= kPairInfoMaxBlocks &&
           (!P.exclude_own || P.storage == kStoreF32);
}

cudaError_t launch_solve_hdda_twins(cudaStream_t s, const HddaParams& P, bool split)
{
    switch (P.storage) {
        case kStoreF32: return launch_pair<kStoreF32>(s, P, true, split);
        case kStoreBF16: return launch_pair<kStoreBF16>(s, P, true, split);
        case kStoreF16: return launch_pair<kStoreF16>(s, P, true, split);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_solve_hdda_paired(cudaStream_t s, const HddaParams& P)
{
    if (P.cap_active == 0 || P.n_batch == 0) return cudaSuccess;
    if (pair_count(P.n_batch, P.pair_group) > 0) {
        cudaError_t e;
        switch (P.storage) {
            case kStoreF32: e = launch_pair<kStoreF32>(s, P); break;
            case kStoreBF16: e = launch_pair<kStoreBF16>(s, P); break;
            case kStoreF16: e = launch_pair<kStoreF16>(s, P); break;
            default: return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
    }
    // the middle batch of every group of odd size alone, by the per-batch walk on
    // a view of that batch
    for (int q = 0; q < pair_lone_count(P.n_batch, P.pair_group); ++q) {
        const int m = pair_lone_batch(q, P.n_batch, P.pair_group);
        HddaParams Q = P;
        Q.traversal = DEX_TRAVERSAL_PER_BATCH;
        Q.n_batch = 1;
        Q.n_lambda = min(8, P.n_lambda - m * 8);
        Q.bricks = P.bricks + (size_t)m * P.cap_active * P.chain * record_floats(8, P.storage);
        Q.words = P.words + (size_t)m * P.n_words;
        Q.J = P.J + (size_t)m * 8 * P.n_cells;
        Q.I = P.I ? P.I + (size_t)m * 8 * P.quad.n_dir * P.n_cells : nullptr;
        if (cudaError_t e = launch_solve_hdda(s, Q)) return e;
    }
    return cudaSuccess;
}

}  // namespace dex
