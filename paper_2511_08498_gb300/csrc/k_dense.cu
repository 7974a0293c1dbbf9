// Plain full-resolution formal solver (long characteristics + Amanatides & Woo DDA)
// and the packing of eta/chi into interleaved wavelength-batch records.
//
// Rays start at cell centres, so all rays of one direction cross the grid planes
// around their own cell at the same ray parameters: the sequence of crossed
// planes, segment lengths and cell offsets is one list per direction, and a ray
// is a prefix of it that ends on the ray's own exit plane.  A warp (32 probes,
// one wavelength batch, one direction at a time) builds that list 32 crossings
// at a time, one per lane, in shared memory; its lanes then only load a record
// at a common offset from their own cell and integrate it.
//
// Plane crossings are evaluated from exact half-integer plane offsets,
//   t = offset * fl(1/d)  (+ a low-order part, see AxisParam),
// instead of being accumulated (t += 1/d): every t is within one rounding of
// exact, and the boundary plane's t is bit-identical to the exit parameter, so
// a ray never steps outside the grid.
//
// The angular sum J = sum_k w_k I_k is taken in the order of the directions, in
// registers when a warp walks all of them (k_solve_dense), and through shared
// memory when the eight warps of a CTA walk eight directions of the same probes
// (k_solve_dense_split: grids too small to fill the chip with one warp per 32
// probes); both give the same bits.  Wavelength batch is the slowest grid
// dimension so that one batch (nx * nz * 8W bytes) is the L2-resident working
// set at a time.
#include "scan.cuh"

namespace dex {

namespace {

__global__ void k_pack_planes(long long n_cells, int n_lambda, int W, int n_batch,
                              const float* __restrict__ eta, const float* __restrict__ chi,
                              float* __restrict__ planes, unsigned int* status)
{
    const long long total = n_cells * n_batch;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const long long c = q % n_cells;
        const int b = (int)(q / n_cells);
        float* rec = planes + q * (2 * W);
        bool bad = false;
        for (int w = 0; w < W; ++w) {
            const int l = b * W + w;
            float S = 0.0f, x = 0.0f;
            if (l < n_lambda) {
                const float e = eta[(long long)l * n_cells + c];
                const float k = chi[(long long)l * n_cells + c];
                if (!(k >= 0.0f) || !(e >= 0.0f) || !isfinite(k) || !isfinite(e) ||
                    (k == 0.0f && e > kEmitterMaxEta)) {
                    bad = true;
                } else {
                    encode_voxel(e, k, S, x);
                }
            }
            rec[w] = S;
            rec[W + w] = x;
        }
        if (bad) raise_status(status, DEX_ERR_NUMERIC);
    }
}

// One crossing of the list: the segment that ends there.
struct __align__(16) PathStep {
    float nl2;   // -length log2(e)
    float th;    // ray parameter of the crossed plane (rounded)
    int off;     // cells from the probe's cell to the segment's
    int moved;   // 1 where the segment's end is beyond its start (counted segments)
};

// The crossings [c0, c0 + 32) of a direction, one per lane.
struct PathBuilder {
    AxisParam ax, az;
    float sx, sz, fx;     // signs of the direction, |dx| / (|dx| + |dz|)
    int stepx, stepz;     // cells per step
    float th_last, tl_last;

    __device__ __forceinline__ PathBuilder(float dx, float dz, int nx)
    {
        // a zero component counts as positive, so its plane offsets are positive
        // and their parameters (offset * inf) are +inf: that axis never steps
        const bool negx = dx < 0.0f, negz = dz < 0.0f;
        ax = axis_param(dx);
        az = axis_param(dz);
        sx = negx ? -1.0f : 1.0f;
        sz = negz ? -1.0f : 1.0f;
        stepx = negx ? -1 : 1;
        stepz = negz ? -nx : nx;
        fx = fabsf(dx) / (fabsf(dx) + fabsf(dz));
        th_last = tl_last = 0.0f;
    }
    __device__ __forceinline__ float px(int m) const { return sx * ((float)m + 0.5f); }
    __device__ __forceinline__ float pz(int n) const { return sz * ((float)n + 0.5f); }
    __device__ __forceinline__ float tx(int m) const { return px(m) * ax.ih; }
    __device__ __forceinline__ float tz(int n) const { return pz(n) * az.ih; }

    // Crossing r: m x planes and r - m z planes precede it in the merged order (x
    // first on ties).  Within rounding m is r |dx| / (|dx| + |dz|); the two loops
    // correct it to the order of the rounded parameters (0 to 2 steps).
    __device__ __forceinline__ PathStep next(int c0, int lane)
    {
        const int r = c0 + lane;
        int m = min(max(__float2int_rn((float)r * fx), 0), r);
        while (m > 0 && !(tx(m - 1) <= tz(r - m))) --m;
        while (m < r && tx(m) <= tz(r - m - 1)) ++m;
        const int n = r - m;
        const float tnx = tx(m), tnz = tz(n);
        const bool on_x = tnx <= tnz;
        const float th = on_x ? tnx : tnz;
        const float tl = plane_lo(on_x ? px(m) : pz(n), on_x ? ax : az, th);
        float th_prev = __shfl_up_sync(0xffffffffu, th, 1), tl_prev = __shfl_up_sync(0xffffffffu, tl, 1);
        if (lane == 0) {
            th_prev = th_last;
            tl_prev = tl_last;
        }
        th_last = __shfl_sync(0xffffffffu, th, 31);
        tl_last = __shfl_sync(0xffffffffu, tl, 31);
        // where an x and a z plane share the rounded parameter (a corner), the lo
        // parts order them and the zero-length step between them can come out a
        // few ulps negative: clamped, or e^{-chi len} overflows in thick cells
        const float len = fmaxf((th - th_prev) + (tl - tl_prev), 0.0f);
        PathStep s;
        s.nl2 = len * kNegLog2e;
        s.th = th;
        s.off = m * stepx + n * stepz;
        s.moved = th > th_prev;
        return s;
    }
};

// One direction's ray of every lane of a warp (cell (i, j), record rec0): I and T
// over the list's prefix up to the lane's exit plane.  Every lane of the warp
// calls it; `live` is false for lanes without a probe.
// EXT: the probe's own-cell emission (the first segment of every ray) is left
// out, so I and J hold the radiation arriving from beyond the cell, attenuated
// by it -- the part of J that MALI's effective mean intensity needs without
// subtracting the own-cell term from J (Section 4.1's preconditioning)
template <int W, bool COUNT, bool EXT>
__device__ __forceinline__ void dense_ray(const DenseParams& P, PathStep* path, int lane, int i, int j,
                                          const float* __restrict__ rec0, float dx, float dz, float stop, bool live,
                                          float* I, float* T, unsigned int& nseg)
{
    constexpr int REC = 2 * W;
    PathBuilder B(dx, dz, P.nx);
    const float Ex = dx < 0.0f ? (float)(-i) - 0.5f : (float)(P.nx - i) - 0.5f;
    const float Ez = dz < 0.0f ? (float)(-j) - 0.5f : (float)(P.nz - j) - 0.5f;
    const float t2 = fminf(Ex * B.ax.ih, Ez * B.az.ih);
#pragma unroll
    for (int w = 0; w < W; ++w) { I[w] = 0.0f; T[w] = 1.0f; }
    // a ray crosses at most nx + nz planes
    for (int c0 = 0; c0 < P.nx + P.nz; c0 += 32) {
        const PathStep mine = B.next(c0, lane);
        __syncwarp();  // every lane is done with the previous crossings
        path[lane] = mine;
        __syncwarp();
        if (live) {
#pragma unroll 4
            for (int q = 0; q < 32; ++q) {
                const PathStep s = path[q];
                const Record<W> r = RecFmt<W, kStoreF32>::load(rec0 + (long long)s.off * REC);
                segments<W>(r.S, r.chi, s.nl2, I, T);
                if constexpr (EXT) {
                    if (c0 + q == 0) {
#pragma unroll
                        for (int w = 0; w < W; ++w) I[w] = 0.0f;
                    }
                }
                if (COUNT) nseg += s.moved;
                if (s.th >= t2) {
                    live = false;
                    break;
                }
                // the counting variant walks every cell: its count is the full-resolution
                // segment count that throughput figures are normalised by
                if (!COUNT && (q & 7) == 7 && ray_done<W>(I, T, stop)) {
                    live = false;
                    break;
                }
            }
        }
        if (!__any_sync(0xffffffffu, live)) break;
    }
}

// The probe of a thread: every cell (32 x rows tile of the grid: lanes along x) or
// the probe list; false without one.
__device__ __forceinline__ bool dense_probe(const DenseParams& P, int tile_rows, int row, int lane, int& i, int& j,
                                            int& p)
{
    if (P.probes == nullptr) {
        const int tiles_x = (P.nx + 31) >> 5;
        const int tx = blockIdx.x % tiles_x, tz = blockIdx.x / tiles_x;
        i = tx * 32 + lane;
        j = tz * tile_rows + row;
        p = j * P.nx + i;
        return i < P.nx && j < P.nz;
    }
    i = j = 0;
    p = (blockIdx.x * tile_rows + row) * 32 + lane;
    if (p >= P.n_probe) return false;
    const int c = P.probes[p];
    if (c < 0 || (long long)c >= P.n_cells) {
        raise_status(P.status, DEX_ERR_TRAVERSAL_CAP);
        return false;
    }
    i = c % P.nx;
    j = c / P.nx;
    return true;
}

template <int W, bool COUNT, bool EXT = false>
__global__ void __launch_bounds__(256, 4) k_solve_dense(const DenseParams P)
{
    __shared__ PathStep s_path[8][32];
    const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int i, j, p;
    const bool live = dense_probe(P, 8, warp, lane, i, j, p);
    const float* rec0 = P.planes + ((size_t)b * P.n_cells + (size_t)j * P.nx + i) * (2 * W);
    const float stop = !COUNT && P.scanned && live ? stop_factor(P.J[(size_t)(b * W) * P.n_probe + p], P.i_bc) : -1.0f;
    float Jw[W];
#pragma unroll
    for (int w = 0; w < W; ++w) Jw[w] = 0.0f;
    unsigned int nseg = 0;
    for (int k = 0; k < P.quad.n_dir; ++k) {
        float I[W], T[W];
        dense_ray<W, COUNT, EXT>(P, s_path[warp], lane, i, j, rec0, P.quad.dx[k], P.quad.dz[k], stop, live, I, T, nseg);
        const float wk = P.quad.w[k];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const float Iw = fmaf(T[w], P.i_bc, I[w]);
            Jw[w] = fmaf(wk, Iw, Jw[w]);
            const int l = b * W + w;
            if (P.I != nullptr && live && l < P.n_lambda) P.I[((size_t)l * P.quad.n_dir + k) * P.n_probe + p] = Iw;
        }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const int l = b * W + w;
        if (live && l < P.n_lambda) P.J[(size_t)l * P.n_probe + p] = Jw[w];
    }
    if (COUNT && P.seg_count != nullptr) atomicAdd(P.seg_count, (unsigned long long)nseg);
}

// Eight directions at a time of 32 probes, one per warp; warp w then adds the
// eight intensities of wavelength w to J in the order of the directions.
template <int W, bool COUNT, bool EXT = false>
__global__ void __launch_bounds__(256, 4) k_solve_dense_split(const DenseParams P)
{
    __shared__ PathStep s_path[8][32];
    __shared__ float s_I[8][W][32];
    const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int i, j, p;
    const bool live = dense_probe(P, 1, 0, lane, i, j, p);
    const float* rec0 = P.planes + ((size_t)b * P.n_cells + (size_t)j * P.nx + i) * (2 * W);
    const float stop = !COUNT && P.scanned && live ? stop_factor(P.J[(size_t)(b * W) * P.n_probe + p], P.i_bc) : -1.0f;
    const int lw = b * W + warp;  // the wavelength whose J this warp sums
    float Jw = 0.0f;
    unsigned int nseg = 0;
    for (int k0 = 0; k0 < P.quad.n_dir; k0 += 8) {
        if (k0 + warp < P.quad.n_dir) {
            float I[W], T[W];
            dense_ray<W, COUNT, EXT>(P, s_path[warp], lane, i, j, rec0, P.quad.dx[k0 + warp], P.quad.dz[k0 + warp],
                                     stop, live, I, T, nseg);
#pragma unroll
            for (int w = 0; w < W; ++w) s_I[warp][w][lane] = fmaf(T[w], P.i_bc, I[w]);
        }
        __syncthreads();
        if (warp < W) {
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                if (k0 + g >= P.quad.n_dir) break;
                const float Iw = s_I[g][warp][lane];
                Jw = fmaf(P.quad.w[k0 + g], Iw, Jw);
                if (P.I != nullptr && live && lw < P.n_lambda)
                    P.I[((size_t)lw * P.quad.n_dir + k0 + g) * P.n_probe + p] = Iw;
            }
        }
        __syncthreads();
    }
    if (warp < W && live && lw < P.n_lambda) P.J[(size_t)lw * P.n_probe + p] = Jw;
    if (COUNT && P.seg_count != nullptr) atomicAdd(P.seg_count, (unsigned long long)nseg);
}

// Bounds for the exact early termination (ray_done): the largest |S| of a batch's
// planes, or -1 where a record is not (finite S, finite chi >= 0).  Two launches, with
// the results in J, which the solve overwrites: CTA q of a batch writes the part
// it has scanned to J[first wavelength][q]; then every probe's entry gets the
// maximum of the parts.
constexpr int kScanCtas = 304;

// Grids of fewer warps (32 probes x batch) than two full loads of the chip's 152 x
// 32 resident ones split the directions.  128 x 128, one wavelength, 16 directions:
// 512 warps took 231 us one after the other, split 61 us.
constexpr long long kSplitWarps = 2 * 152 * 32;


template <int W>
__global__ void __launch_bounds__(256) k_dense_scan(const DenseParams P)
{
    const int b = blockIdx.y;
    const float* base = P.planes + (size_t)b * P.n_cells * (2 * W);
    float m = 0.0f;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < P.n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        const Record<W> r = RecFmt<W, kStoreF32>::load(base + c * (2 * W));
#pragma unroll
        for (int w = 0; w < W; ++w) m = join_bounds(m, bound_of(r.S[w], r.chi[w]));
    }
    m = join_cta(m);
    if (threadIdx.x == 0) P.J[(size_t)(b * W) * P.n_probe + blockIdx.x] = m;
}

// Entries already replaced by another CTA hold the maximum itself, so reading
// them in place of their parts changes nothing.
__global__ void __launch_bounds__(256) k_dense_spread(const DenseParams P, int n_parts)
{
    float* J = P.J + (size_t)(blockIdx.y * P.W) * P.n_probe;
    float m = 0.0f;
    for (int q = threadIdx.x; q < n_parts; q += blockDim.x) m = join_bounds(m, __ldcg(J + q));
    m = join_cta(m);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.n_probe; p += gridDim.x * blockDim.x) J[p] = m;
}

template <int W>
void launch_dense_w(bool split, dim3 grid, cudaStream_t s, const DenseParams& P)
{
    if (P.scanned) {
        const int parts = P.n_probe < kScanCtas ? P.n_probe : kScanCtas;
        k_dense_scan<W><<<dim3((unsigned)parts, (unsigned)P.n_batch), 256, 0, s>>>(P);
        const int ctas = (P.n_probe + 1023) / 1024;
        k_dense_spread<<<dim3((unsigned)(ctas < 304 ? ctas : 304), (unsigned)P.n_batch), 256, 0, s>>>(P, parts);
    }
#define DEX_LAUNCH_DENSE(K)                                               \
    if (P.exclude_own) {                                                  \
        if (P.seg_count) K<W, true, true><<<grid, 256, 0, s>>>(P);        \
        else K<W, false, true><<<grid, 256, 0, s>>>(P);                   \
    } else if (P.seg_count) {                                             \
        K<W, true><<<grid, 256, 0, s>>>(P);                               \
    } else {                                                              \
        K<W, false><<<grid, 256, 0, s>>>(P);                              \
    }
    if (split) {
        DEX_LAUNCH_DENSE(k_solve_dense_split)
    } else {
        DEX_LAUNCH_DENSE(k_solve_dense)
    }
#undef DEX_LAUNCH_DENSE
}

}  // namespace

cudaError_t launch_pack_planes(cudaStream_t s, long long n_cells, int n_lambda, int W,
                               const float* eta, const float* chi, float* planes, unsigned int* status)
{
    const int n_batch = (n_lambda + W - 1) / W;
    const long long total = n_cells * n_batch;
    if (total == 0) return cudaSuccess;
    long long blocks = (total + 255) / 256;
    if (blocks > 152LL * 64) blocks = 152LL * 64;
    k_pack_planes<<<(unsigned)blocks, 256, 0, s>>>(n_cells, n_lambda, W, n_batch, eta, chi, planes, status);
    return cudaGetLastError();
}

cudaError_t launch_solve_dense(cudaStream_t s, const DenseParams& P0)
{
    if (P0.n_probe == 0 || P0.n_batch == 0) return cudaSuccess;
    DenseParams P = P0;
    // scan the planes for the early termination's bound where the solve reads at
    // least sixteen times as many records
    P.scanned = !P.seg_count && (double)P.n_probe * P.quad.n_dir * 0.5 * ((double)P.nx + P.nz) >= 16.0 * (double)P.n_cells;
    // one warp per 32 probes, or eight (one per direction) where those would not
    // fill the chip
    const long long warps = (P.n_probe + 31LL) / 32 * P.n_batch;
    const bool split = warps < kSplitWarps;
    const int rows = split ? 1 : 8;
    const unsigned tiles = P.probes == nullptr ? (unsigned)(((P.nx + 31) / 32) * ((P.nz + rows - 1) / rows))
                                               : (unsigned)((P.n_probe + 32 * rows - 1) / (32 * rows));
    const dim3 grid(tiles, (unsigned)P.n_batch);
    switch (P.W) {
        case 1: launch_dense_w<1>(split, grid, s, P); break;
        case 2: launch_dense_w<2>(split, grid, s, P); break;
        case 4: launch_dense_w<4>(split, grid, s, P); break;
        case 8: launch_dense_w<8>(split, grid, s, P); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dex
