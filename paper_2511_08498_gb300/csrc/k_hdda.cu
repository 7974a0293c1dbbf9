// Hierarchical DDA formal solver over the sparse, mipmapped block grid
// (Section 2.3, Algorithm 1, with the robustness requirements of Section 2.3.1).
//
// One CTA per (active block, wavelength batch); one thread per probe cell of
// the block, walking every quadrature direction (J accumulates in registers).
// The packed 3-bit block states of the batch are staged in shared memory: they
// are the structure the traversal consults at every block crossing.
//
// Traversal of one ray p(t) = p_c + t d:
//  * inside a region of constant voxel size vox = 2^mip (16 for an empty block,
//    mip = -1) it is the DDA of Amanatides & Woo: the next plane on each axis is
//    at the voxel's far face, the nearer one ends the segment;
//  * segments in non-empty blocks are integrated with the voxel's (S, chi) record
//    at level mip; empty blocks are crossed in one step and add nothing;
//  * on entering a block with another level the tracer is re-initialised: the
//    MIP-0 cell entered is known exactly on the stepped axis (the plane just
//    crossed) and taken from p(t) on the other axis, clamped to the voxel the ray
//    was in; both are floored to the new voxel size.
// Plane parameters are two-float sums (see AxisParam) and t never decreases: a
// plane found behind the ray (rounding after a re-initialisation) yields a
// zero-length step.  These replace the paper's two nudges (advancing t by 1e-2
// voxel on entering empty space, forcing t_h > t) with exact bookkeeping.  A ray
// ends where it leaves the box around the non-empty blocks (nothing beyond it
// adds to I or T); a ray that would step out of the grid before that sets
// DEX_ERR_TRAVERSAL_CAP.
#include "scan.cuh"

namespace dex {

namespace {

// Static voxel model: a record holds (S, chi) for the W wavelengths of a batch,
// stored in format ST (float32, bfloat16 or scaled float16; see RecFmt).
template <int W, int ST = kStoreF32>
struct StaticModel {
    static constexpr int kStride = RecFmt<W, ST>::kStride;
    static constexpr bool kSplit = BrickFmt<W, ST>::kSplit;  // float32: brick rows of S, then chi
    static constexpr int kSplitStride = BrickFmt<W, ST>::kX;
    static constexpr bool kPerBatch = true;
    static constexpr int kMinBlocks = 4;  // CTAs per SM the register budget targets
    static constexpr bool kTwins = true;
    // record loaded at the top of each step: -3.3% (float32) on the 1024^2 benchmark
    // solve; +5% with the bfloat16 / float16 unpacking (register pressure)
    static constexpr bool kEarlyLoad = ST == kStoreF32;
    static constexpr bool kZeroNoop = true;  // zero records integrate to no change
    struct Params {
        int unused;
    };
    using Voxel = Record<W>;
    __device__ __forceinline__ static Voxel load(const float* p) { return RecFmt<W, ST>::load(p); }
    __device__ __forceinline__ static Voxel load_split(const Params&, const float* p, int coff)
    {
        return BrickFmt<W, ST>::load(p, coff);
    }
    __device__ __forceinline__ static void integrate(const Params&, const Voxel& v, int, float, float, float nl2,
                                                     float* I, float* T, float)
    {
        segments<W>(v.S, v.chi, nl2, I, T);
    }
};

template <typename K, typename MP>
cudaError_t launch_hdda_kernel(K kernel, dim3 grid, size_t smem, cudaStream_t s, const HddaParams& P, const MP& M)
{
    if (smem > 24 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kernel<<<grid, 256, smem, s>>>(P, M);
    return cudaSuccess;
}

}  // namespace

// Bounds of the exact early termination for the static solves (not for counting
// ones, whose segment counts run to exactly zero transmission).
static void scan_bricks(cudaStream_t s, HddaParams& P)
{
    const dim3 grid((unsigned)P.cap_active, (unsigned)P.n_batch);
    switch (P.W * 4 + P.storage) {
#define DEX_SCAN(WW, ST) \
    case WW * 4 + ST: k_scan_bricks<WW, ST><<<grid, 128, 0, s>>>(P); break;
        DEX_SCAN(1, kStoreF32)
        DEX_SCAN(2, kStoreF32)
        DEX_SCAN(4, kStoreF32)
        DEX_SCAN(8, kStoreF32)
        DEX_SCAN(4, kStoreBF16)
        DEX_SCAN(8, kStoreBF16)
        DEX_SCAN(4, kStoreF16)
        DEX_SCAN(8, kStoreF16)
#undef DEX_SCAN
        default: return;
    }
    launch_spread(s, P);
    P.scanned = 1;
}

// Where the per-batch solve looks for pairs of batches that it may walk once (twins):
// W = 8 and a grid that the pair kernel's table covers.  The pairs and the other batches
// are two launches, so where some batch is certain to be left for the second (the middle
// one of an odd number) the first must fill the chip: two rounds of the pair kernel's 304
// resident CTAs, five where directions are split; with an even number, of which some pairs
// may differ, one and a half (256 x 320, 31 wavelengths, 60% empty, 256 blocks of pairs:
// 2.90 ms instead of 2.24), and always where split.  That is counted in active blocks, which
// the device knows (HddaParams::twins: from how many on; 0 never): by the grid's blocks,
// 384 x 400 cells, 40 wavelengths, 60% of them empty, took 4.73 ms instead of 3.76.
// Static lines, 32 directions, 40% empty, one walk per batch -> with pairs:
//   768^2, 32 wavelengths  35.2 -> 28.7 ms    256^2, 32 (split)  3.38 -> 2.98 ms
//   512^2, 16              14.5 -> 11.8       96^2, 16 (split)   0.284 -> 0.250
//   512^2, 24              15.4 -> 14.2       384^2, 24          7.80 -> 9.00 (not taken)
//   320^2, 24 (split)      4.12 -> 3.79       160^2, 24 (split)  0.741 -> 0.782 (not taken)
// bfloat16 pairs run 128-thread CTAs, 760 resident, and gain nothing when split (160^2,
// 32: 1.04 -> 1.15) or below two rounds (400 x 336, 32, 578 blocks of pairs: 4.76 -> 5.14).
// Where the levels differ the check costs 0.3% (768^2, 20: 36.6 both ways).
static int twins_from(const HddaParams& P, bool split)
{
    if (P.W != 8 || P.seg_count || !P.scanned || (long long)P.nbx * P.nbz > kPairInfoMaxBlocks) return 0;
    if (split && P.storage == kStoreBF16) return 0;
    const int pairs = pair_count(P.n_batch, P.pair_group);
    if (pairs == 0) return 0;
    const bool even = pair_lone_count(P.n_batch, P.pair_group) == 0;
    const int unsplit = P.storage == kStoreBF16 ? 760 : even ? 456 : 608;
    const int ctas = split ? (even ? 1 : 190) : unsplit;
    const int from = max((ctas + pairs - 1) / pairs, P.active_from);
    return (P.active_to ? min(P.active_to - 1, P.cap_active) : P.cap_active) >= from ? from : 0;
}

// One walk per batch, directions split or not.
static cudaError_t launch_per_batch(cudaStream_t s, HddaParams P, bool info, bool split)
{
    const size_t smem = sizeof(float) * ((size_t)P.split_at + (split ? (size_t)split_chunk<8>() * P.W * 32 : 0));
    const int blocks = P.active_to ? min(P.active_to, P.cap_active) : P.cap_active;
    const dim3 grid((unsigned)blocks * (split ? 8u : 1u), (unsigned)P.n_batch);
    cudaError_t e = cudaSuccess;
    P.twins = twins_from(P, split);
    if (P.twins && (e = launch_solve_hdda_twins(s, P, split)) != cudaSuccess) return e;
    switch (P.W * 4 + P.storage) {
#define DEX_LAUNCH_(WW, ST, INFO)                                                                                     \
    {                                                                                                                 \
        using M_ = StaticModel<WW, ST>;                                                                               \
        if (P.seg_count) e = launch_hdda_kernel(k_solve_hdda_t<WW, true, M_, INFO>, grid, smem, s, P, M_::Params{});  \
        else if (split)                                                                                               \
            e = launch_hdda_kernel(k_solve_hdda_t<WW, false, M_, INFO, false, true>, grid, smem, s, P, M_::Params{}); \
        else e = launch_hdda_kernel(k_solve_hdda_t<WW, false, M_, INFO>, grid, smem, s, P, M_::Params{});             \
    }
#define DEX_LAUNCH(WW, ST) \
    case WW * 4 + ST: DEX_LAUNCH_(WW, ST, false) break;
#define DEX_LAUNCH_INFO(ST)                  \
    case 8 * 4 + ST:                         \
        if (info) DEX_LAUNCH_(8, ST, true)   \
        else DEX_LAUNCH_(8, ST, false)       \
        break;
        DEX_LAUNCH(1, kStoreF32)
        DEX_LAUNCH(2, kStoreF32)
        DEX_LAUNCH(4, kStoreF32)
        DEX_LAUNCH_INFO(kStoreF32)
        DEX_LAUNCH(4, kStoreBF16)
        DEX_LAUNCH_INFO(kStoreBF16)
        DEX_LAUNCH(4, kStoreF16)
        DEX_LAUNCH_INFO(kStoreF16)
#undef DEX_LAUNCH_INFO
#undef DEX_LAUNCH
#undef DEX_LAUNCH_
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_solve_hdda(cudaStream_t s, const HddaParams& P0)
{
    if (P0.cap_active == 0 || P0.n_batch == 0) return cudaSuccess;
    HddaParams P = P0;
    if (!P.scanned && !P.seg_count && !solve_hdda_shared_applies(P)) scan_bricks(s, P);
    if (P.traversal == DEX_TRAVERSAL_PAIRED) {
        if (!solve_hdda_paired_applies(P)) return cudaErrorNotSupported;
        return launch_solve_hdda_paired(s, P);
    }
    if (solve_hdda_shared_applies(P)) return launch_solve_hdda_shared(s, P);
    if (P.exclude_own) {
        // own-voxel emission left out: W = 8, float32 records (the MALI path)
        if (P.W != 8 || P.storage != kStoreF32) return cudaErrorNotSupported;
        const long long nb = (long long)P.nbx * P.nbz;
        const bool inf = nb <= kInfoMaxBlocks;
        const size_t sm = inf ? sizeof(int) * (size_t)nb : sizeof(unsigned long long) * (size_t)P.n_words;
        dim3 g((unsigned)P.cap_active, (unsigned)P.n_batch);
        using SM8 = StaticModel<8, kStoreF32>;
        cudaError_t e;
        if (inf && P.seg_count) e = launch_hdda_kernel(k_solve_hdda_t<8, true, SM8, true, true>, g, sm, s, P, SM8::Params{});
        else if (inf) e = launch_hdda_kernel(k_solve_hdda_t<8, false, SM8, true, true>, g, sm, s, P, SM8::Params{});
        else if (P.seg_count) e = launch_hdda_kernel(k_solve_hdda_t<8, true, SM8, false, true>, g, sm, s, P, SM8::Params{});
        else e = launch_hdda_kernel(k_solve_hdda_t<8, false, SM8, false, true>, g, sm, s, P, SM8::Params{});
        if (e != cudaSuccess) return e;
        return cudaGetLastError();
    }
    // W = 8 on grids of at most kInfoMaxBlocks blocks: one shared-memory word per
    // block (InfoLookup); otherwise the packed state words (WordLookup)
    const long long n_blocks = (long long)P.nbx * P.nbz;
    const bool info = P.W == 8 && n_blocks <= kInfoMaxBlocks;
    P.split_at = (int)(((info ? n_blocks : 2LL * P.n_words) + 3) & ~3LL);
    const bool split = split_directions(P);
    const long long ctas = (long long)P.cap_active * P.n_batch;
    if (!split && !P.seg_count && ctas < kSplitSparseCtas && P.split_at <= 24576) {
        HddaParams Q = P;
        P.active_from = Q.active_to = (int)((kSplitActiveCtas + P.n_batch - 1) / P.n_batch);
        const cudaError_t e = launch_per_batch(s, Q, info, true);
        if (e != cudaSuccess) return e;
    }
    return launch_per_batch(s, P, info, split);
}

}  // namespace dex

namespace dex {

int record_floats(int W, int storage)
{
    if (storage == kStoreF32) return 2 * W;
    if (storage == kStoreBF16) return W;
    if (storage == kStoreF16) return 4 + W;
    return 0;
}

}  // namespace dex
