// Many independent atmospheres in one persistent launch.
//
// Work items are (atmosphere, wavelength batch, active block, part of the
// block), numbered atmosphere by atmosphere (item_base[a] + (batch * capacity_a
// + rank) * parts + part).  A fixed grid of CTAs pulls `chunk` items at a time
// from a device counter (the queue) until it runs dry; each item is the block
// solve of k_solve_hdda_t (shared trace_ray) over 256 / parts of its probes.  Where
// pairs of batches may share a walk there are two such launches, the pairs' and the
// other batches' (twins_apply).  Consecutive items mostly share an atmosphere and
// batch, so the staged block states and quadrature are reused, and the L2 working set stays
// one atmosphere batch wide.  Per-atmosphere completion times (globaltimer, ns)
// are recorded when requested.

#include "scan.cuh"

namespace dex {

namespace {

// Scratch of the allocation-free entry point (dex_batch_solve_noalloc): a
// statically sized device array, present on every GPU that loads the library
// until the process exits.  Word 0 is the work counter.  Calls that overlap on
// the GPU share it and race.
static __device__ __align__(256) unsigned int g_noalloc_scratch[DEX_NOALLOC_SCRATCH_WORDS];

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

template <int W>
struct StaticRec {
    static constexpr int kStride = 2 * W;
    static constexpr bool kSplit = true;  // float32 brick rows: S of the row, then chi
    static constexpr int kSplitStride = W;
    static constexpr bool kEarlyLoad = true;  // as the float32 static model of the single-grid solve
    static constexpr bool kZeroNoop = true;
    struct Params {
        int unused;
    };
    using Voxel = Record<W>;
    __device__ __forceinline__ static Voxel load_split(const Params&, const float* p, int coff)
    {
        return BrickFmt<W, kStoreF32>::load(p, coff);
    }
    __device__ __forceinline__ static void integrate(const Params&, const Voxel& v, int, float, float, float nl2,
                                                     float* I, float* T, float)
    {
        segments<W>(v.S, v.chi, nl2, I, T);
    }
};

// kMinCtas: CTAs per SM the register budget is sized for (768 / NT: 80 registers, three
// 256-thread CTAs of residency, at W = 8 with up to 48 bytes spilled, 150 where shared
// walks are looked for; 1024 / NT: 64 registers, four, 120 and 230 bytes; pairs 512 / NT:
// 128 registers, two).
// NT threads per CTA = probes per work item (a 16 x (NT / 16) part of a block,
// warps on 8 x 4 tiles as in k_solve_hdda_t); a CTA claims `chunk` consecutive
// items per queue increment.  kInfo: the block table is staged as one word per
// block (offset * 8 + state); otherwise the packed 3-bit state words.  Every
// probe accumulates J over all directions in its thread, in the order of the
// single-grid solve, so results do not depend on these choices.
// kPair (W = 8): a work unit is a pair of batches (pair_batches) walked once on
// the smaller of their two levels, 16 wavelengths per thread, or a lone batch
// (pair_lone_batch) walked alone, as dex_formal_solve_hdda's paired walk.
// kTwin (W = 8): with kPair the pairs whose blocks all have the same levels, as the TWIN
// walk of k_solve_hdda_pair, without it the batches of no such pair (kernels of their
// own: the check in the others' loop cost the small launches 2 to 3%).
template <int W, int NT, bool kInfo, int kMinCtas, bool kPair = false, bool kTwin = false>
__global__ void __launch_bounds__(NT, kMinCtas) k_batch_solve(const BatchParams P)
{
    extern __shared__ unsigned long long s_dyn[];
    __shared__ float s_J[kPair ? 2 * W : W][NT];
    __shared__ float s_dx[DEX_MAX_DIRS], s_dz[DEX_MAX_DIRS], s_w[DEX_MAX_DIRS];
    __shared__ unsigned int s_item;
    constexpr int kParts = 256 / NT;
    int* s_info = reinterpret_cast<int*>(s_dyn);
    const int tid = threadIdx.x;
    int cur_atm = -1, cur_batch = -1;
    [[maybe_unused]] int skip_atm = -1, skip_batch = -1;
    unsigned int nseg_unused = 0;
    bool capped = false;
    if (P.start_ns != nullptr && tid == 0) atomicMin(P.start_ns, global_ns());

    for (;;) {
        __syncthreads();  // every thread is done with the previous claim
        if (tid == 0) s_item = atomicAdd(P.queue, (unsigned int)P.chunk);
        __syncthreads();
        const unsigned int first = s_item;
        if ((long long)first >= P.n_items) break;
        for (int c = 0; c < P.chunk; ++c) {
            const long long item = (long long)first + c;
            if (item >= P.n_items) break;
            int a = 0;
            while (a + 1 < P.n_atm && item >= P.atm[a + 1].item_base) ++a;
            const AtmDesc& A = P.atm[a];
            const long long local = item - A.item_base;
            const long long unit = local / kParts;
            const int part = (int)(local % kParts);
            const int b = (int)(unit / A.cap_active), r = (int)(unit % A.cap_active);
            if (r >= *A.n_active || (kTwin && a == skip_atm && b == skip_batch)) continue;
            // kPair: b numbers the atmosphere's pairs, then its lone batches
            int b1 = b, b2 = -1;
            if constexpr (kPair) {
                const int n_batch = (A.n_lambda + W - 1) / W, np = pair_count(n_batch, P.pair_group);
                if (b < np) pair_batches(b, n_batch, P.pair_group, b1, b2);
                else b1 = pair_lone_batch(b - np, n_batch, P.pair_group);
            }
            __syncthreads();  // every thread is done with the previous item's shared data
            if (a != cur_atm || b != cur_batch) {
                if constexpr (kTwin) {
                    const int other = kPair ? (b2 >= 0 ? b2 : b1) : pair_partner(b, (A.n_lambda + W - 1) / W, P.pair_group);
                    const bool twins = other != b1 && states_agree(A.words + (size_t)b1 * A.n_words,
                                                                   A.words + (size_t)other * A.n_words, A.n_words);
                    if (twins != kPair) {
                        skip_atm = a;
                        skip_batch = b;
                        continue;
                    }
                }
                if constexpr (kPair) {
                    // one word per block, offset * 8 + the smaller of the pair's states
                    const int nb = A.nbx * A.nbz;
                    const unsigned long long* w1 = A.words + (size_t)b1 * A.n_words;
                    const unsigned long long* w2 = A.words + (size_t)(b2 >= 0 ? b2 : b1) * A.n_words;
                    for (int q = tid; q < nb; q += NT)
                        s_info[q] = pack_block_info(A.block_offset[q], min(block_state(w1, q), block_state(w2, q)));
                } else if constexpr (kInfo) {
                    const int nb = A.nbx * A.nbz;
                    const unsigned long long* wb = A.words + (size_t)b * A.n_words;
                    for (int q = tid; q < nb; q += NT) s_info[q] = pack_block_info(A.block_offset[q], block_state(wb, q));
                } else {
                    for (int q = tid; q < A.n_words; q += NT) s_dyn[q] = A.words[(size_t)b * A.n_words + q];
                }
                if (a != cur_atm)
                    for (int q = tid; q < A.n_dir; q += NT) {
                        s_dx[q] = A.dirs[2 * q];
                        s_dz[q] = A.dirs[2 * q + 1];
                        s_w[q] = A.weights[q];
                    }
                cur_atm = a;
                cur_batch = b;
            }
#pragma unroll
            for (int w = 0; w < (kPair ? 2 * W : W); ++w) s_J[w][tid] = 0.0f;
            __syncthreads();

            const int blk0 = A.active[r];
            const int bx0 = blk0 % A.nbx, bz0 = blk0 / A.nbx;
            const int wrp = tid >> 5;
            const int i = bx0 * DEX_BLOCK + (wrp & 1) * 8 + (tid & 7);
            const int j = bz0 * DEX_BLOCK + part * (DEX_BLOCK / kParts) + (wrp >> 1) * 4 + ((tid & 31) >> 3);
            const int state0 = (kInfo || kPair ? (s_info[blk0] & 7) : block_state(s_dyn, blk0)) - 1;
            const size_t cell = (size_t)j * A.nx + i;
            const size_t plane = (size_t)W * A.nx * A.nz;
            if (state0 < 0) {
                capped = true;
                A.J[b1 * plane + cell] = 0.0f;  // it held the bound
                if (kPair && b2 >= 0) A.J[b2 * plane + cell] = 0.0f;
                continue;
            }
            Geo G;
            G.nx = A.nx;
            G.nz = A.nz;
            G.nbx = A.nbx;
            G.nbz = A.nbz;
            G.chain = A.chain;
            G.cap_active = A.cap_active;
            const size_t batch_floats = (size_t)A.cap_active * A.chain * (2 * W);
            G.batch_base = A.bricks + (size_t)b1 * batch_floats;
            set_box_full(G);
#pragma unroll
            for (int q = 0; q < 4; ++q) G.band[q] = A.band[q];
            // the batch's bound (k_scan_batch) waits where this thread's first J will go
            float bound = A.J[b1 * plane + cell];
            [[maybe_unused]] float bound2 = 0.0f;
            [[maybe_unused]] int second = -1;  // kTwin: a batch to be walked by itself after b1
            if (kPair && b2 >= 0) {
                bound2 = A.J[b2 * plane + cell];
                if (kTwin && join_bounds(bound, bound2) < 0.0f) {
                    second = b2;
                    b2 = b1;
                } else {
                    bound = join_bounds(bound, bound2);
                }
            }
            G.stop = stop_factor(bound, A.i_bc);
            const int mip0 = min(state0, distance_cap(G, 0.0f));
            typename StaticRec<W>::Params M{};
            const long long n_cells = (long long)A.nx * A.nz;
            auto solve = [&]() {
                for (int k = 0; k < A.n_dir; ++k) {
                    const float wk = s_w[k];
                    if ((kPair && kTwin) || (kPair && b2 >= 0)) {
                        // the pair: 16 wavelengths along one walk
                        using PM = PairRecModel<kStoreF32, kMinCtas>;
                        const typename PM::Params M2{(long long)(b2 - b1) * (long long)batch_floats};
                        float I[2 * W], T[2 * W];
#pragma unroll
                        for (int w = 0; w < 2 * W; ++w) { I[w] = 0.0f; T[w] = 1.0f; }
                        trace_ray<2 * W, false, PM>(G, M2, b1, i, j, bx0, bz0, r, mip0, s_dx[k], s_dz[k],
                                                    InfoLookup{s_info}, I, T, nseg_unused, capped);
#pragma unroll
                        for (int w = 0; w < 2 * W; ++w) s_J[w][tid] = fmaf(wk, fmaf(T[w], A.i_bc, I[w]), s_J[w][tid]);
                    } else {
                        float I[W], T[W];
#pragma unroll
                        for (int w = 0; w < W; ++w) { I[w] = 0.0f; T[w] = 1.0f; }
                        if constexpr (kInfo || kPair)
                            trace_ray<W, false, StaticRec<W>>(G, M, b1, i, j, bx0, bz0, r, mip0, s_dx[k], s_dz[k],
                                                               InfoLookup{s_info}, I, T, nseg_unused, capped);
                        else
                            trace_ray<W, false, StaticRec<W>>(G, M, b1, i, j, bx0, bz0, r, mip0, s_dx[k], s_dz[k],
                                                               WordLookup{s_dyn, A.block_offset}, I, T, nseg_unused,
                                                               capped);
#pragma unroll
                        for (int w = 0; w < W; ++w) s_J[w][tid] = fmaf(wk, fmaf(T[w], A.i_bc, I[w]), s_J[w][tid]);
                    }
                }
#pragma unroll
                for (int w = 0; w < (kPair ? 2 * W : W); ++w) {
                    const int l = w < W ? b1 * W + w : b2 * W + (w - W);
                    if ((w < W || b2 >= 0) && l < A.n_lambda) A.J[(size_t)l * n_cells + (size_t)j * A.nx + i] = s_J[w][tid];
                }
            };
            if constexpr (kPair && kTwin) {
                for (;;) {
                    solve();
                    if (second < 0) break;
                    G.batch_base += (size_t)(second - b1) * batch_floats;
                    b1 = b2 = second;
                    second = -1;
                    G.stop = stop_factor(bound2, A.i_bc);
#pragma unroll
                    for (int w = 0; w < 2 * W; ++w) s_J[w][tid] = 0.0f;
                }
            } else {
                solve();
            }
            if (P.done_ns != nullptr) {
                __syncthreads();
                if (tid == 0) atomicMax(P.done_ns + a, global_ns());
            }
        }
    }
    if (capped) raise_status(P.status, DEX_ERR_TRAVERSAL_CAP);
}

// Bounds of the early termination, as k_scan_bricks and k_spread_bounds for every
// atmosphere (blockIdx.z) and wavelength batch (blockIdx.y).
template <int W>
__global__ void __launch_bounds__(128) k_scan_batch(const BatchParams P)
{
    const AtmDesc& A = P.atm[blockIdx.z];
    const int b = blockIdx.y;
    if (b * W >= A.n_lambda || blockIdx.x >= A.cap_active) return;
    const int na = *A.n_active;
    float* J = A.J + (size_t)(b * W) * A.nx * A.nz;
    for (int a = blockIdx.x; a < na; a += gridDim.x) {
        const float m = join_cta(chain_bound<W, kStoreF32>(A.bricks + ((size_t)b * A.cap_active + a) * A.chain * (2 * W), A.chain));
        const int blk = A.active[a];
        if (threadIdx.x == 0) J[(size_t)(blk / A.nbx * DEX_BLOCK) * A.nx + blk % A.nbx * DEX_BLOCK] = m;
    }
}

template <int W>
__global__ void __launch_bounds__(256) k_spread_batch(const BatchParams P)
{
    const AtmDesc& A = P.atm[blockIdx.z];
    const int b = blockIdx.y;
    if (b * W >= A.n_lambda || blockIdx.x >= A.cap_active) return;
    const int na = *A.n_active;
    float* J = A.J + (size_t)(b * W) * A.nx * A.nz;
    float m = 0.0f;
    for (int a = threadIdx.x; a < na; a += blockDim.x) {
        const int blk = A.active[a];
        m = join_bounds(m, __ldcg(J + (size_t)(blk / A.nbx * DEX_BLOCK) * A.nx + blk % A.nbx * DEX_BLOCK));
    }
    m = join_cta(m);
    for (int a = blockIdx.x; a < na; a += gridDim.x) {
        const int blk = A.active[a];
        J[(size_t)(blk / A.nbx * DEX_BLOCK + (threadIdx.x >> 4)) * A.nx + blk % A.nbx * DEX_BLOCK + (threadIdx.x & 15)] = m;
    }
}

template <int W>
void scan_batch(cudaStream_t s, const BatchParams& P)
{
    int cap = 1, n_batch = 1;
    for (int a = 0; a < P.n_atm; ++a) {
        cap = max(cap, P.atm[a].cap_active);
        n_batch = max(n_batch, (P.atm[a].n_lambda + W - 1) / W);
    }
    const dim3 scan((unsigned)min(cap, 608), (unsigned)n_batch, (unsigned)P.n_atm);
    const dim3 spread((unsigned)min(cap, 76), (unsigned)n_batch, (unsigned)P.n_atm);
    k_scan_batch<W><<<scan, 128, 0, s>>>(P);
    k_spread_batch<W><<<spread, 256, 0, s>>>(P);
}

template <int W, int NT, bool kInfo, int kMinCtas, bool kPair = false, bool kTwin = false>
cudaError_t launch_batch_t(cudaStream_t s, const BatchParams& P, int ctas, size_t smem)
{
    auto kernel = k_batch_solve<W, NT, kInfo, kMinCtas, kPair, kTwin>;
    if (smem > 16 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kernel<<<(unsigned)ctas, NT, smem, s>>>(P);
    return cudaSuccess;
}

template <int W, bool kOcc, bool kTwin = false>
cudaError_t launch_batch_w(cudaStream_t s, const BatchParams& P, int ctas, int packet, bool info, size_t smem)
{
    switch (packet * 2 + (info ? 1 : 0)) {
        case 256 * 2: return launch_batch_t<W, 256, false, kOcc ? 4 : 3, false, kTwin>(s, P, ctas, smem);
        case 256 * 2 + 1: return launch_batch_t<W, 256, true, kOcc ? 4 : 3, false, kTwin>(s, P, ctas, smem);
        case 128 * 2: return launch_batch_t<W, 128, false, kOcc ? 8 : 6, false, kTwin>(s, P, ctas, smem);
        case 128 * 2 + 1: return launch_batch_t<W, 128, true, kOcc ? 8 : 6, false, kTwin>(s, P, ctas, smem);
        case 64 * 2: return launch_batch_t<W, 64, false, kOcc ? 16 : 12, false, kTwin>(s, P, ctas, smem);
        case 64 * 2 + 1: return launch_batch_t<W, 64, true, kOcc ? 16 : 12, false, kTwin>(s, P, ctas, smem);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Device address of the static scratch array on the current device.  The array's
// host-side name is not a device address, so kernels must be given this pointer.
// It is looked up on every call (a runtime table look-up, no allocation) rather
// than cached: after a cudaDeviceReset the device's context, and with it the
// array, is a new one, and a cached address would point into the old context.
cudaError_t noalloc_scratch(unsigned int** out)
{
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    *out = static_cast<unsigned int*>(p);
    return cudaSuccess;
}

// Where pairs are looked for: W = 8, grids that the pair kernel's table covers, and
// enough blocks of pairs that the second launch's start, after the last item of the
// first, costs less than the shared walks give.  Eight to twelve atmospheres of static
// lines (about half of the pairs agree), one walk per batch -> with pairs: 3168 blocks of
// pairs 23.4 -> 22.1 ms, 3904 39.4 -> 36.5, 6784 72.6 -> 64.9; but 2816 13.6 -> 14.2,
// 1968 13.5 -> 15.4, 352 3.5 -> 5.1.
constexpr long long kTwinItems = 3040;  // ten rounds of the pair kernel's 304 resident CTAs

static bool twins_apply(const BatchParams& P, int W, size_t max_blocks)
{
    if (W != 8 || max_blocks > (size_t)kInfoMaxBlocks) return false;
    long long pairs = 0;
    for (int a = 0; a < P.n_atm; ++a)
        pairs += (long long)pair_count((P.atm[a].n_lambda + 7) / 8, P.pair_group) * P.atm[a].cap_active;
    return pairs >= kTwinItems;
}

cudaError_t launch_batch_solve(cudaStream_t s, const BatchParams& P, int ctas, int W, int packet, bool info,
                               bool occupancy, size_t max_words, size_t max_blocks)
{
    const size_t smem_bytes = info ? sizeof(int) * max_blocks : sizeof(unsigned long long) * max_words;
    cudaError_t e = cudaMemsetAsync(P.queue, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess || P.n_items == 0) return e;
    if (occupancy && W != 8) return cudaErrorInvalidValue;
    switch (W) {
        case 1: scan_batch<1>(s, P); break;
        case 2: scan_batch<2>(s, P); break;
        case 4: scan_batch<4>(s, P); break;
        case 8: scan_batch<8>(s, P); break;
        default: return cudaErrorInvalidValue;
    }
    // pairs of batches (W = 8): one word per block staged, the compiler's budget
    // bounded at 128 registers (two 256-thread CTAs per SM)
    auto launch_pairs = [&](const BatchParams& Q, auto twin) {
        constexpr bool kTwin = decltype(twin)::value;
        const size_t smem = sizeof(int) * max_blocks;
        switch (packet) {
            case 256: return launch_batch_t<8, 256, true, 2, true, kTwin>(s, Q, ctas, smem);
            case 128: return launch_batch_t<8, 128, true, 4, true, kTwin>(s, Q, ctas, smem);
            case 64: return launch_batch_t<8, 64, true, 8, true, kTwin>(s, Q, ctas, smem);
            default: return cudaErrorInvalidValue;
        }
    };
    if (P.paired) {
        if (W != 8) return cudaErrorInvalidValue;
        if ((e = launch_pairs(P, std::false_type{})) != cudaSuccess) return e;
        return cudaGetLastError();
    }
    const bool twins = twins_apply(P, W, max_blocks);
    if (twins) {
        BatchParams Q = P;
        Q.n_items = 0;
        for (int a = 0; a < P.n_atm; ++a) {
            Q.atm[a].item_base = Q.n_items;
            Q.n_items += (long long)pair_count((P.atm[a].n_lambda + 7) / 8, P.pair_group) * P.atm[a].cap_active * P.parts;
        }
        if ((e = launch_pairs(Q, std::true_type{})) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(P.queue, 0, sizeof(unsigned int), s)) != cudaSuccess) return e;
    }
    switch (W) {
        case 1: e = launch_batch_w<1, false>(s, P, ctas, packet, info, smem_bytes); break;
        case 2: e = launch_batch_w<2, false>(s, P, ctas, packet, info, smem_bytes); break;
        case 4: e = launch_batch_w<4, false>(s, P, ctas, packet, info, smem_bytes); break;
        case 8:
            if (twins)
                e = occupancy ? launch_batch_w<8, true, true>(s, P, ctas, packet, info, smem_bytes)
                              : launch_batch_w<8, false, true>(s, P, ctas, packet, info, smem_bytes);
            else
                e = occupancy ? launch_batch_w<8, true>(s, P, ctas, packet, info, smem_bytes)
                              : launch_batch_w<8, false>(s, P, ctas, packet, info, smem_bytes);
            break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace dex
