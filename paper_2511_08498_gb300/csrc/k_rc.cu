// Radiance cascades around the hierarchical DDA (the formal solution of the
// paper's code, Section 4.1 "Model Configuration"): cascade i has probes on a
// lattice of spacing 2^i, n0 4^i directions and the radiance interval
// [t0 4^(i-1), t0 4^i] (cascade 0: [0, t0]); its intervals are traced through the
// sparse mipmapped grid at min(block level, the cascade's level cap).
//
// One launch per cascade, from the top down, fuses the trace with the merge:
//   L = I + T R,  R = i_bc where the ray left the grid inside its interval (and
//   on the top cascade), else the bilinear interpolation at this probe of the
//   mean over the 4 child directions (4k .. 4k+3) of the cascade above (its 4
//   nearest probes, indices clamped at the lattice edge).
// Thread = (direction, probe) of one wavelength batch, the four siblings 4k .. 4k+3
// of a direction in neighbouring lanes.  A cascade hands down the sum over the
// siblings, added in their order by shuffles, so the cascade below reads 4 values
// per ray and wavelength instead of 16 and a quarter of the radiance is stored (the
// 16 scalar reads kept the lower cascades at 85% of the L1 data pipe).  Cascade 0
// likewise adds its directions into J where there are four; otherwise it stores
// them and a final kernel averages.  On the lower cascades a warp holds eight
// neighbouring probes; on the upper ones (long intervals from probes 16 or more
// cells apart) 32 neighbouring directions of one probe, whose rays fan out and read
// neighbouring bricks.  CTAs of 64 threads: a warp's rays end together, those of a
// 256-thread CTA did not, and its finished warps held their registers (10 of 16
// resident warps active on the long cascades).  Cascade 0 skips probes in empty
// blocks (J is not defined there).
//
// The tracer starts at t_s: the entry cell is floor(p(t_s)) (a rounding that
// lands in the next cell back only yields a zero-length first step), plane
// offsets from the probe are exact (probes sit at multiples of 1/2), and the
// last segment is clipped at min(t_e, grid exit).
#include "scan.cuh"

namespace dex {

namespace {

__host__ __device__ constexpr int rc_level_offset(int m) { return 341 - (341 >> (2 * m)); }

__device__ __forceinline__ int rc_block_state(const unsigned long long* words, int blk)
{
    const int wi = blk / DEX_STATES_PER_WORD, sh = DEX_STATE_BITS * (blk - wi * DEX_STATES_PER_WORD);
    return (int)((words[wi] >> sh) & 7ull);
}

// Emission I and transmission T of the interval [t_s, t_e] of the ray o + t d
// through the sparse mipmapped grid; returns true when the ray leaves the grid
// before t_e.  NB = 2: two wavelength batches (bricks `off` floats apart) along one
// walk on the smaller of their levels; I and T hold 2 W values, the second batch's
// from index W.  info: the walk's word per block, offset * 8 + state
// (k_rc_info): one load per block entered, where the packed states of one or two
// batches and the offset table took three in a row and two divisions by 21.
template <int W, bool COUNT, int ST, int NB = 1>
__device__ __forceinline__ bool rc_interval(const RcParams& P, const float* __restrict__ base, long long off,
                                            const int* __restrict__ info, float ox, float oz,
                                            float dx, float dz, float stop, float* I, float* T,
                                            unsigned int& nseg, bool& capped)
{
    using BF = BrickFmt<W, ST>;
    constexpr int REC = BF::kRec;
    const bool negx = dx < 0.0f, negz = dz < 0.0f;
    const int sx = negx ? -1 : 1, sz = negz ? -1 : 1;
    const AxisParam ax = axis_param(dx), az = axis_param(dz);
    const float t_exit = fminf((negx ? -ox : (float)P.nx - ox) * ax.ih, (negz ? -oz : (float)P.nz - oz) * az.ih);
    const bool left = t_exit <= P.t_e;
    const float t_end = fminf(t_exit, P.t_e);
    if (!(t_end > P.t_s)) return true;
    const int cap = 2 * (P.nx + P.nz) + 64;

    // entry cell, block, level and voxel at t_s
    const int cx = min(max(__float2int_rd(fmaf(P.t_s, dx, ox)), 0), P.nx - 1);
    const int cz = min(max(__float2int_rd(fmaf(P.t_s, dz, oz)), 0), P.nz - 1);
    int bxc = cx >> 4, bzc = cz >> 4;
    int blk = bzc * P.nbx + bxc;
    int key = __ldg(info + blk), st = (key & 7) - 1;
    int mip = st < 0 ? -1 : min(st, P.level_cap);
    int shift = mip >= 0 ? mip : 4;
    int vox = 1 << shift, side = DEX_BLOCK >> shift;
    int lx = (cx - bxc * DEX_BLOCK) >> shift, lz = (cz - bzc * DEX_BLOCK) >> shift;
    float Px = (float)(bxc * DEX_BLOCK + (lx + (negx ? 0 : 1)) * vox) - ox;
    float Pz = (float)(bzc * DEX_BLOCK + (lz + (negz ? 0 : 1)) * vox) - oz;
    const float* rp = base;
    if (mip >= 0)
        rp = base + BF::offset((long long)(key >> 3) * P.chain + rc_level_offset(mip), lz, lx, side);
    float th_prev = P.t_s, tl_prev = 0.0f;

    Record<W> r, r2;
    for (int it = 0;; ++it) {
        // the current voxel's record is issued first: the stepping and crossing
        // bookkeeping below hides its latency
        if (mip >= 0) {
            r = BF::load(rp, BF::chi_off(side));
            if constexpr (NB == 2) r2 = BF::load(rp + off, BF::chi_off(side));
        }
        const float tnx = Px * ax.ih, tnz = Pz * az.ih;
        const bool on_x = tnx <= tnz;
        float th = on_x ? tnx : tnz;
        float tl = plane_lo(on_x ? Px : Pz, on_x ? ax : az, th);
        const bool last = th >= t_end;
        if (last) {  // clipped at the interval end (or the grid exit)
            th = t_end;
            tl = 0.0f;
        }
        const float len = fmaxf((th - th_prev) + (tl - tl_prev), 0.0f);
        const int cur_mip = mip;
        if (!last) {
            if (it >= cap) { capped = true; break; }
            const float fv = (float)vox;
            bool cross;
            if (on_x) {
                lx += sx;
                Px += negx ? -fv : fv;
                rp += negx ? -BF::kX : BF::kX;
                cross = (unsigned)lx >= (unsigned)side;
            } else {
                lz += sz;
                Pz += negz ? -fv : fv;
                rp += negz ? -side * REC : side * REC;
                cross = (unsigned)lz >= (unsigned)side;
            }
            // counted segments run to the block in which every transmission has become zero
            if (COUNT && cross && all_opaque<NB * W>(T)) break;
            if (cross) {
                const int bxn = bxc + (on_x ? sx : 0), bzn = bzc + (on_x ? 0 : sz);
                if ((unsigned)bxn >= (unsigned)P.nbx || (unsigned)bzn >= (unsigned)P.nbz) {
                    capped = true;
                    break;
                }
                blk = bzn * P.nbx + bxn;
                key = __ldg(info + blk);
                st = (key & 7) - 1;
                const int mip_new = st < 0 ? -1 : min(st, P.level_cap);
                if (mip_new == mip) {
                    if (on_x) lx = negx ? side - 1 : 0;
                    else lz = negz ? side - 1 : 0;
                } else {
                    // MIP-0 cell entered: exact on the stepped axis, from p(t) on the
                    // other one, clamped to the voxel just left
                    const int vo = vox;
                    int m0x, m0z;
                    if (on_x) {
                        m0x = bxn * DEX_BLOCK + (negx ? DEX_BLOCK - 1 : 0);
                        const int lo = bzc * DEX_BLOCK + lz * vo;
                        m0z = min(max(__float2int_rd(fmaf(th, dz, oz)), lo), lo + vo - 1);
                    } else {
                        m0z = bzn * DEX_BLOCK + (negz ? DEX_BLOCK - 1 : 0);
                        const int lo = bxc * DEX_BLOCK + lx * vo;
                        m0x = min(max(__float2int_rd(fmaf(th, dx, ox)), lo), lo + vo - 1);
                    }
                    mip = mip_new;
                    shift = mip >= 0 ? mip : 4;
                    vox = 1 << shift;
                    side = DEX_BLOCK >> shift;
                    lx = (m0x - bxn * DEX_BLOCK) >> shift;
                    lz = (m0z - bzn * DEX_BLOCK) >> shift;
                    Px = (float)(bxn * DEX_BLOCK + (lx + (negx ? 0 : 1)) * vox) - ox;
                    Pz = (float)(bzn * DEX_BLOCK + (lz + (negz ? 0 : 1)) * vox) - oz;
                }
                bxc = bxn;
                bzc = bzn;
                if (mip >= 0)
                    rp = base + BF::offset((long long)(key >> 3) * P.chain + rc_level_offset(mip), lz, lx, side);
            }
        }
        if (cur_mip >= 0) {
            segments<W>(r.S, r.chi, len * kNegLog2e, I, T);
            if constexpr (NB == 2) segments<W>(r2.S, r2.chi, len * kNegLog2e, I + W, T + W);
            if (COUNT) nseg += NB * (th > th_prev);
        }
        // the rest changes no bit of the radiance
        if (last || (!COUNT && (it & 3) == 3 && ray_done<NB * W>(I, T, stop))) break;
        th_prev = th;
        tl_prev = tl;
    }
    return left;
}

constexpr int kRcThreads = 64;

// W consecutive floats, 16-byte aligned for W >= 4
template <int W>
__device__ __forceinline__ void load_w(const float* __restrict__ p, float* v)
{
    if constexpr (W >= 4) {
#pragma unroll
        for (int w = 0; w < W; w += 4) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(p + w));
            v[w] = a.x; v[w + 1] = a.y; v[w + 2] = a.z; v[w + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int w = 0; w < W; ++w) v[w] = __ldg(p + w);
    }
}

template <int W>
__device__ __forceinline__ void store_w(float* __restrict__ p, const float* v)
{
    if constexpr (W >= 4) {
#pragma unroll
        for (int w = 0; w < W; w += 4)
            *reinterpret_cast<float4*>(p + w) = make_float4(v[w], v[w + 1], v[w + 2], v[w + 3]);
    } else {
#pragma unroll
        for (int w = 0; w < W; ++w) p[w] = v[w];
    }
}

// ((s0 + s1) + s2) + s3 over four neighbouring lanes, in the first of them
__device__ __forceinline__ float sibling_sum(float v)
{
    const float s1 = __shfl_down_sync(0xffffffffu, v, 1), s2 = __shfl_down_sync(0xffffffffu, v, 2),
                s3 = __shfl_down_sync(0xffffffffu, v, 3);
    return ((v + s1) + s2) + s3;
}

// Walks (units) of a solve: the batches, or with P.paired the pairs, then the lone
// batches.
template <int NB>
__device__ __forceinline__ int rc_first_unit(const RcParams& P)
{
    return NB == 1 && P.paired ? pair_count(P.n_batch, P.pair_group) : 0;
}

// The word per block of every walk.
__global__ void __launch_bounds__(256) k_rc_info(const RcParams P, int n_pairs, int* __restrict__ info)
{
    const int nb = P.nbx * P.nbz, u = blockIdx.y;
    int b = u, b2;
    if (P.paired) {
        if (u < n_pairs) pair_batches(u, P.n_batch, P.pair_group, b, b2);
        else b = b2 = pair_lone_batch(u - n_pairs, P.n_batch, P.pair_group);
    } else {
        b2 = b;
    }
    const unsigned long long *w1 = P.words + (size_t)b * P.n_words, *w2 = P.words + (size_t)b2 * P.n_words;
    const int blk = blockIdx.x * blockDim.x + threadIdx.x;
    if (blk < nb)
        info[(size_t)u * nb + blk] =
            pack_block_info(P.block_offset[blk], min(rc_block_state(w1, blk), rc_block_state(w2, blk)));
}

// NB = 1: blockIdx.y is the batch (with P.paired: the lone batch
// pair_lone_batch(blockIdx.y)); NB = 2: the pair pair_batches(blockIdx.y), one
// walk for both batches on the smaller of their levels.
template <int W, bool COUNT, int ST, int NB>
__global__ void __launch_bounds__(kRcThreads, (NB == 1 ? 1024 : 512) / kRcThreads) k_rc_cascade(const RcParams P)
{
    int b = blockIdx.y, b2 = blockIdx.y;
    if constexpr (NB == 2) pair_batches(blockIdx.y, P.n_batch, P.pair_group, b, b2);
    else if (P.paired) b = b2 = pair_lone_batch(blockIdx.y, P.n_batch, P.pair_group);
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n_probe = (long long)P.pnx * P.pnz;
    // rays come in groups of `sib` sibling lanes (4, or 1 on a cascade 0 of other than
    // four directions per group of lanes): group q, ray s of it
    const int sib = P.siblings, s = sib == 4 ? (int)(g & 3) : 0;
    const long long q = sib == 4 ? g >> 2 : g;
    const int n_group = P.n_dir / sib;
    bool live = g < n_probe * P.n_dir;
    int j, p;
    if (P.dir_fastest) {  // lanes: neighbouring directions of one probe
        p = (int)(q / n_group);
        j = (int)(q - (long long)p * n_group);
    } else {              // lanes: neighbouring probes
        j = (int)(q / n_probe);
        p = (int)(q - (long long)j * n_probe);
    }
    const int k = j * sib + s;
    const int px = p % P.pnx, pz = p / P.pnx;
    const int* info = P.info + (size_t)(rc_first_unit<NB>(P) + blockIdx.y) * (P.nbx * P.nbz);
    if (live && P.spacing == 1)  // cascade 0: probes only in non-empty blocks
        live = (__ldg(info + (pz >> 4) * P.nbx + (px >> 4)) & 7) != 0;
    constexpr int REC = RecFmt<W, ST>::kStride;
    const size_t batch_floats = (size_t)P.cap_active * P.chain * REC;
    const float* base = P.bricks + (size_t)b * batch_floats;
    const long long off = (long long)(b2 - b) * (long long)batch_floats;
    const float ox = (float)P.spacing * ((float)px + 0.5f), oz = (float)P.spacing * ((float)pz + 0.5f);
    float I[NB * W], T[NB * W];
#pragma unroll
    for (int w = 0; w < NB * W; ++w) { I[w] = 0.0f; T[w] = 1.0f; }
    unsigned int nseg = 0;
    bool capped = false, left = true;
    if (live) {
        // the merged radiance above is bounded as the emission and the boundary are
        float stop = -1.0f;
        if (!COUNT && P.bounds != nullptr) {
            float m = __ldg(P.bounds + b);
            if (NB == 2) m = join_bounds(m, __ldg(P.bounds + b2));
            stop = stop_factor(m, P.i_bc);
        }
        left = rc_interval<W, COUNT, ST, NB>(P, base, off, info, ox, oz, P.dirs[2 * k], P.dirs[2 * k + 1], stop,
                                             I, T, nseg, capped);
    }

#pragma unroll
    for (int h = 0; h < NB; ++h) {
        const int bq = h == 0 ? b : b2;
        float R[W];
#pragma unroll
        for (int w = 0; w < W; ++w) R[w] = P.i_bc;
        if (!left && P.upper != nullptr) {
            // bilinear stencil on the coarser lattice: this probe sits at (p + 1/2)/2 - 1/2
            const int qnx = P.pnx >> 1, qnz = P.pnz >> 1;
            const float ux = 0.5f * ((float)px + 0.5f) - 0.5f, uz = 0.5f * ((float)pz + 0.5f) - 0.5f;
            const int x0 = (int)floorf(ux), z0 = (int)floorf(uz);
            const float fx = ux - (float)x0, fz = uz - (float)z0;
            const int xa = min(max(x0, 0), qnx - 1), xb = min(max(x0 + 1, 0), qnx - 1);
            const int za = min(max(z0, 0), qnz - 1), zb = min(max(z0 + 1, 0), qnz - 1);
            const long long q_probe = (long long)qnx * qnz;
            // sums over the four child directions 4k .. 4k + 3
            const float* up = P.upper + ((size_t)bq * P.n_dir + k) * q_probe * W;
            const int qs[4] = {za * qnx + xa, za * qnx + xb, zb * qnx + xa, zb * qnx + xb};
            const float ws[4] = {(1.0f - fz) * (1.0f - fx), (1.0f - fz) * fx, fz * (1.0f - fx), fz * fx};
#pragma unroll
            for (int w = 0; w < W; ++w) R[w] = 0.0f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float m[W];
                load_w<W>(up + (size_t)qs[c] * W, m);
#pragma unroll
                for (int w = 0; w < W; ++w) R[w] = fmaf(ws[c] * 0.25f, m[w], R[w]);
            }
        }
        float L[W];
#pragma unroll
        for (int w = 0; w < W; ++w) L[w] = fmaf(T[h * W + w], R[w], I[h * W + w]);
        if (sib == 4) {
#pragma unroll
            for (int w = 0; w < W; ++w) L[w] = sibling_sum(L[w]);
        }
        if (!live || s != 0) continue;
        if (P.J != nullptr) {  // cascade 0 of four directions: J is their mean
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const int l = bq * W + w;
                if (l < P.n_lambda) P.J[(size_t)l * n_probe + p] = L[w] * 0.25f;
            }
        } else {
            store_w<W>(P.out + (((size_t)bq * n_group + j) * n_probe + p) * W, L);
        }
    }
    if (capped) raise_status(P.status, DEX_ERR_TRAVERSAL_CAP);
    if (COUNT && nseg && P.seg_count != nullptr) atomicAdd(P.seg_count, (unsigned long long)nseg);
}

// J at every cell of every non-empty block: the mean of the cascade-0 radiance
// over its n0 directions (n0 other than four)
template <int W>
__global__ void __launch_bounds__(256) k_rc_mean(const RcParams P, const float* __restrict__ L0, float* __restrict__ J)
{
    const int b = blockIdx.y;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n_cells = (long long)P.nx * P.nz;
    if (c >= n_cells) return;
    const int x = (int)(c % P.nx), z = (int)(c / P.nx);
    if (rc_block_state(P.words + (size_t)b * P.n_words, (z >> 4) * P.nbx + (x >> 4)) == 0) return;
    float acc[W];
#pragma unroll
    for (int w = 0; w < W; ++w) acc[w] = 0.0f;
    const float* src = L0 + (size_t)b * (size_t)P.n_dir * n_cells * W;
    for (int k = 0; k < P.n_dir; ++k)
#pragma unroll
        for (int w = 0; w < W; ++w) acc[w] += src[((size_t)k * n_cells + c) * W + w];
    const float inv = 1.0f / (float)P.n_dir;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const int l = b * W + w;
        if (l < P.n_lambda) J[(size_t)l * n_cells + c] = acc[w] * inv;
    }
}

// Bounds of the exact early termination, in the workspace beside the walks' words:
// every block's of every batch, then the batches'.
template <int W, int ST>
__global__ void __launch_bounds__(128) k_rc_scan(const RcParams P, float* __restrict__ parts)
{
    const int blk = blockIdx.x, b = blockIdx.y, a = P.block_offset[blk];
    float m = 0.0f;
    if (a >= 0 && a < P.cap_active)
        m = join_cta(chain_bound<W, ST>(P.bricks + ((size_t)b * P.cap_active + a) * P.chain * RecFmt<W, ST>::kStride, P.chain));
    if (threadIdx.x == 0) parts[(size_t)b * P.nbx * P.nbz + blk] = m;
}

__global__ void __launch_bounds__(1024) k_rc_bound(int n_blocks, const float* __restrict__ parts,
                                                   float* __restrict__ bounds)
{
    float m = 0.0f;
    for (int q = threadIdx.x; q < n_blocks; q += blockDim.x) m = join_bounds(m, parts[(size_t)blockIdx.x * n_blocks + q]);
    m = join_cta(m);
    if (threadIdx.x == 0) bounds[blockIdx.x] = m;
}

template <int W, int ST, int NB>
void launch_rc_nb(cudaStream_t s, const RcParams& P, int n_units)
{
    if (n_units == 0) return;
    const long long n = (long long)P.pnx * P.pnz * P.n_dir;
    const dim3 grid((unsigned)((n + kRcThreads - 1) / kRcThreads), (unsigned)n_units);
    if (P.seg_count) k_rc_cascade<W, true, ST, NB><<<grid, kRcThreads, 0, s>>>(P);
    else k_rc_cascade<W, false, ST, NB><<<grid, kRcThreads, 0, s>>>(P);
}

template <int W, int ST>
void launch_rc_w(cudaStream_t s, const RcParams& P)
{
    if constexpr (W == 8) {
        if (P.paired) {
            // pairs of batches on one walk each, then the lone batches
            launch_rc_nb<8, ST, 2>(s, P, pair_count(P.n_batch, P.pair_group));
            launch_rc_nb<8, ST, 1>(s, P, pair_lone_count(P.n_batch, P.pair_group));
            return;
        }
    }
    launch_rc_nb<W, ST, 1>(s, P, P.n_batch);
}

}  // namespace

cudaError_t launch_rc_cascade(cudaStream_t s, const RcParams& P)
{
    if (P.n_batch == 0 || P.n_dir == 0) return cudaSuccess;
    switch (P.W * 4 + P.storage) {
        case 1 * 4 + kStoreF32: launch_rc_w<1, kStoreF32>(s, P); break;
        case 2 * 4 + kStoreF32: launch_rc_w<2, kStoreF32>(s, P); break;
        case 4 * 4 + kStoreF32: launch_rc_w<4, kStoreF32>(s, P); break;
        case 8 * 4 + kStoreF32: launch_rc_w<8, kStoreF32>(s, P); break;
        case 8 * 4 + kStoreBF16: launch_rc_w<8, kStoreBF16>(s, P); break;
        case 8 * 4 + kStoreF16: launch_rc_w<8, kStoreF16>(s, P); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_rc_tables(cudaStream_t s, RcParams& P, float* scratch, bool bounds)
{
    if (P.n_batch == 0) return cudaSuccess;
    const int nb = P.nbx * P.nbz;
    int* info = reinterpret_cast<int*>(scratch);
    const int n_pairs = P.paired ? pair_count(P.n_batch, P.pair_group) : 0;
    const int units = P.paired ? n_pairs + pair_lone_count(P.n_batch, P.pair_group) : P.n_batch;
    k_rc_info<<<dim3((unsigned)((nb + 255) / 256), (unsigned)units), 256, 0, s>>>(P, n_pairs, info);
    P.info = info;
    if (!bounds) return cudaGetLastError();
    float* parts = scratch + (size_t)nb * units;
    float* out = parts + (size_t)nb * P.n_batch;
    const dim3 grid((unsigned)nb, (unsigned)P.n_batch);
    switch (P.W * 4 + P.storage) {
        case 1 * 4 + kStoreF32: k_rc_scan<1, kStoreF32><<<grid, 128, 0, s>>>(P, parts); break;
        case 2 * 4 + kStoreF32: k_rc_scan<2, kStoreF32><<<grid, 128, 0, s>>>(P, parts); break;
        case 4 * 4 + kStoreF32: k_rc_scan<4, kStoreF32><<<grid, 128, 0, s>>>(P, parts); break;
        case 8 * 4 + kStoreF32: k_rc_scan<8, kStoreF32><<<grid, 128, 0, s>>>(P, parts); break;
        case 8 * 4 + kStoreBF16: k_rc_scan<8, kStoreBF16><<<grid, 128, 0, s>>>(P, parts); break;
        case 8 * 4 + kStoreF16: k_rc_scan<8, kStoreF16><<<grid, 128, 0, s>>>(P, parts); break;
        default: return cudaErrorInvalidValue;
    }
    k_rc_bound<<<(unsigned)P.n_batch, 1024, 0, s>>>(nb, parts, out);
    P.bounds = out;
    return cudaGetLastError();
}

cudaError_t launch_rc_mean(cudaStream_t s, const RcParams& P, const float* L0, float* J)
{
    if (P.n_batch == 0) return cudaSuccess;
    const long long n_cells = (long long)P.nx * P.nz;
    const dim3 grid((unsigned)((n_cells + 255) / 256), (unsigned)P.n_batch);
    switch (P.W) {
        case 1: k_rc_mean<1><<<grid, 256, 0, s>>>(P, L0, J); break;
        case 2: k_rc_mean<2><<<grid, 256, 0, s>>>(P, L0, J); break;
        case 4: k_rc_mean<4><<<grid, 256, 0, s>>>(P, L0, J); break;
        case 8: k_rc_mean<8><<<grid, 256, 0, s>>>(P, L0, J); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dex
