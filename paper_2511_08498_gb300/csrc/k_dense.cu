// Plain full-resolution formal solver (long characteristics + Amanatides & Woo DDA)
// and the packing of eta/chi into interleaved wavelength-batch records.
//
// Rays start at cell centres, so all rays of one direction cross the grid planes
// around their own cell at the same ray parameters: the sequence of crossed
// planes, segment lengths and cell offsets is one list per direction, and a ray
// is a prefix of it that ends on the ray's own exit plane.  A warp (32 probes,
// one wavelength batch, one direction at a time) builds that list 32 crossings
// at a time, one per lane, in shared memory; its lanes then only load a record
// at a common offset from their own cell and integrate it (with eight wavelengths per
// batch only in k_solve_dense_tile: dense_ray).
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
    long long off;  // bytes from the probe's record to the segment's (grids of up to 2^32 cells)
};

// The crossings [c0, c0 + 32) of a direction, one per lane.
struct PathBuilder {
    AxisParam ax, az;
    float sx, sz, fx;     // signs of the direction, |dx| / (|dx| + |dz|)
    int stepx, stepz;     // bytes per step
    float th_last, tl_last;

    __device__ __forceinline__ PathBuilder(float dx, float dz, int nx, int rec_bytes)
    {
        // a zero component counts as positive, so its plane offsets are positive
        // and their parameters (offset * inf) are +inf: that axis never steps
        const bool negx = dx < 0.0f, negz = dz < 0.0f;
        ax = axis_param(dx);
        az = axis_param(dz);
        sx = negx ? -1.0f : 1.0f;
        sz = negz ? -1.0f : 1.0f;
        stepx = negx ? -rec_bytes : rec_bytes;
        stepz = stepx * (negx == negz ? nx : -nx);  // at most 64 x 65536 bytes
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
    __device__ __forceinline__ int x_planes(int r) const
    {
        int m = min(max(__float2int_rn((float)r * fx), 0), r);
        while (m > 0 && !(tx(m - 1) <= tz(r - m))) --m;
        while (m < r && tx(m) <= tz(r - m - 1)) ++m;
        return m;
    }
    __device__ __forceinline__ PathStep next(int c0, int lane, int& m)
    {
        const int r = c0 + lane;
        m = x_planes(r);
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
        s.off = (long long)m * stepx + (long long)n * stepz;
        return s;
    }
};

// One direction's ray of every lane of a warp (cell (i, j), record rec0): I and T up to
// the lane's exit plane.  Every lane of the warp calls it; `live` is false for lanes
// without a probe.
// W = 8: every lane walks its own ray, the record requested before the plane arithmetic
// that hides its latency.  Other W: over a prefix of the warp's list of crossings, where
// the plane arithmetic, several times the update of one or two wavelengths, is shared.
// With eight the list only adds its read to every step's chain; 256 x 264, 6 directions,
// split: 417 us on the list, 309 walking; 200 x 208, 96 wavelengths, 24 directions, a
// probe list: 6.26 and 5.65 ms.
// EXT: the probe's own-cell emission (the first segment of every ray) is left
// out, so I and J hold the radiation arriving from beyond the cell, attenuated
// by it -- the part of J that MALI's effective mean intensity needs without
// subtracting the own-cell term from J (Section 4.1's preconditioning)
// The counting variant walks every cell: its count is the full-resolution segment
// count that throughput figures are normalised by.
template <int W, bool COUNT, bool EXT>
__device__ __forceinline__ void dense_ray(const DenseParams& P, PathStep* path, int lane, int i, int j,
                                          const float* __restrict__ rec0, float dx, float dz, float stop, bool live,
                                          float* I, float* T, unsigned int& nseg)
{
    constexpr int REC = 2 * W;
    PathBuilder B(dx, dz, P.nx, REC * (int)sizeof(float));
    const float Ex = dx < 0.0f ? (float)(-i) - 0.5f : (float)(P.nx - i) - 0.5f;
    const float Ez = dz < 0.0f ? (float)(-j) - 0.5f : (float)(P.nz - j) - 0.5f;
    const float t2 = fminf(Ex * B.ax.ih, Ez * B.az.ih);
#pragma unroll
    for (int w = 0; w < W; ++w) { I[w] = 0.0f; T[w] = 1.0f; }
    if constexpr (W == 8) {
        if (!live) return;
        const char* rp = reinterpret_cast<const char*>(rec0);
        float Px = B.px(0), Pz = B.pz(0), th_prev = 0.0f, tl_prev = 0.0f;
        // a ray crosses at most nx + nz planes
        for (int it = 0; it < P.nx + P.nz; ++it) {
            const Record<W> r = RecFmt<W, kStoreF32>::load(reinterpret_cast<const float*>(rp));
            const float tnx = Px * B.ax.ih, tnz = Pz * B.az.ih;
            const bool on_x = tnx <= tnz;
            const float th = on_x ? tnx : tnz;
            const float tl = plane_lo(on_x ? Px : Pz, on_x ? B.ax : B.az, th);
            const float len = fmaxf((th - th_prev) + (tl - tl_prev), 0.0f);  // as PathBuilder::next
            segments<W>(r.S, r.chi, len * kNegLog2e, I, T);
            if constexpr (EXT) {
                if (it == 0) {
#pragma unroll
                    for (int w = 0; w < W; ++w) I[w] = 0.0f;
                }
            }
            if (COUNT) nseg += th > th_prev;
            if (th >= t2 || (!COUNT && (it & 7) == 7 && ray_done<W>(I, T, stop))) break;
            th_prev = th;
            tl_prev = tl;
            if (on_x) {
                Px += B.sx;
                rp += B.stepx;
            } else {
                Pz += B.sz;
                rp += B.stepz;
            }
        }
    } else {
        constexpr int GROUP = W == 1 ? 8 : (W == 2 ? 4 : 2);
        float th_end = 0.0f;  // the last crossing of the chunk before
        [[maybe_unused]] float th_count = 0.0f;
        // a ray crosses at most nx + nz planes
        for (int c0 = 0; c0 < P.nx + P.nz; c0 += 32) {
            int m;
            const PathStep mine = B.next(c0, lane, m);
            __syncwarp();  // every lane is done with the previous crossings
            path[lane] = mine;
            __syncwarp();
            if (live) {
                // a few records at a time, loaded before the first of them is used: a step's
                // latency, not its arithmetic, sets the time of small grids.  A segment beyond
                // the ray's exit (the crossing before it is at or past t2) reads nothing.
                float th_before = c0 == 0 ? 0.0f : th_end;
                for (int q0 = 0; q0 < 32 && live; q0 += GROUP) {
                    PathStep s[GROUP];
                    Record<W> r[GROUP];
#pragma unroll
                    for (int g = 0; g < GROUP; ++g) {
                        s[g] = path[q0 + g];
                        if (g == 0 || th_before < t2)
                            r[g] = RecFmt<W, kStoreF32>::load(
                                reinterpret_cast<const float*>(reinterpret_cast<const char*>(rec0) + s[g].off));
                        th_before = s[g].th;
                    }
#pragma unroll
                    for (int g = 0; g < GROUP; ++g) {
                        segments<W>(r[g].S, r[g].chi, s[g].nl2, I, T);
                        if constexpr (EXT) {
                            if (c0 + q0 + g == 0) {
#pragma unroll
                                for (int w = 0; w < W; ++w) I[w] = 0.0f;
                            }
                        }
                        if (COUNT) {
                            nseg += s[g].th > th_count;  // segments whose end is beyond their start
                            th_count = s[g].th;
                        }
                        if (s[g].th >= t2) {
                            live = false;
                            break;
                        }
                    }
                    if (!COUNT && live && ((q0 + GROUP) & 7) == 0 && ray_done<W>(I, T, stop)) live = false;
                }
                th_end = th_before;
            }
            if (!__any_sync(0xffffffffu, live)) break;
        }
    }
}

// Every cell a probe, W = 8, grids that fill the chip: CTAs of 32 x 12 probes stage
// the records that their rays cross in the next 32 crossings -- the tile, widened by
// the crossings' x and z steps -- in shared memory (cp.async, at most 38 x 38 cells),
// and read them there.  In planes, S and chi lie side by side per cell, so the two
// 256-bit loads of a warp each touch every line of its 2 KB and take 16 passes of the
// L1 data pipe each where 8 would do: that pipe was 82% busy and bound k_solve_dense.
// Here the four 16-byte pieces of a record lie in four planes, so that lanes at
// neighbouring cells read neighbouring pieces: 16 passes per warp and step, plus a
// tenth for the staging (43% busy).  Two CTAs per SM: one stages while the other
// integrates.  601 x 437, 20 wavelengths, 24 directions: 24.3 -> 22.9 ms; what is left
// is the update itself (the FP32 pipe, 14 ms) and the shared loads' latency, which
// 80 registers (12 rows, the next record read a step ahead) hide better than 64 (16
// rows, 23.1 ms) and than two probes per thread at 123 (26.1 ms).
constexpr int kTileRows = 12, kTileThreads = 32 * kTileRows;
// the most of (32 + a) (kTileRows + b) over a + b = 32
constexpr int tile_cells()
{
    int most = 0;
    for (int a = 0; a <= 32; ++a)
        most = (32 + a) * (kTileRows + 32 - a) > most ? (32 + a) * (kTileRows + 32 - a) : most;
    return most;
}
constexpr int kTilePlane = ((tile_cells() * 16 + 127) / 128) * 128 + 32;  // bytes of one piece of every cell

template <bool EXT>
__global__ void __launch_bounds__(kTileThreads, 2) k_solve_dense_tile(const DenseParams P)
{
    extern __shared__ __align__(128) unsigned char s_rec[];  // four planes of pieces, then 32 crossings
    PathStep* s_path = reinterpret_cast<PathStep*>(s_rec + 4 * kTilePlane);
    const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles_x = (P.nx + 31) >> 5;
    const int i0 = blockIdx.x % tiles_x * 32, j0 = blockIdx.x / tiles_x * kTileRows;
    const int i = i0 + lane, j = j0 + warp;
    const bool probe = i < P.nx && j < P.nz;
    const int p = (int)((unsigned)j * P.nx + i);
    const unsigned char* base = reinterpret_cast<const unsigned char*>(P.planes + (size_t)b * P.n_cells * 16);
    const float stop = P.scanned && probe ? stop_factor(P.J[(size_t)(b * 8) * P.n_probe + p], P.i_bc) : -1.0f;
    const uint32_t rec = (uint32_t)__cvta_generic_to_shared(s_rec) + (lane & 3) * kTilePlane + (lane >> 2) * 16;
    float Jw[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) Jw[w] = 0.0f;
    for (int k = 0; k < P.quad.n_dir; ++k) {
        const float dx = P.quad.dx[k], dz = P.quad.dz[k];
        PathBuilder B(dx, dz, P.nx, 64);
        const float Ex = dx < 0.0f ? (float)(-i) - 0.5f : (float)(P.nx - i) - 0.5f;
        const float Ez = dz < 0.0f ? (float)(-j) - 0.5f : (float)(P.nz - j) - 0.5f;
        const float t2 = fminf(Ex * B.ax.ih, Ez * B.az.ih);
        bool live = probe;
        float I[8], T[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) { I[w] = 0.0f; T[w] = 1.0f; }
        int m0 = 0;
        for (int c0 = 0; c0 < P.nx + P.nz; c0 += 32) {
            // x and z planes crossed before this chunk and before the next: the records of
            // the chunk's segments lie within these steps of the tile
            const int n0 = c0 - m0, m1 = B.x_planes(c0 + 32), n1 = c0 + 32 - m1;
            const int rw = 32 + m1 - m0, rh = kTileRows + n1 - n0;
            const int x0 = dx < 0.0f ? i0 - m1 : i0 + m0, z0 = dz < 0.0f ? j0 - n1 : j0 + n0;
            if (!__syncthreads_or(live)) break;  // and every warp is done with the previous records
            for (int r = warp; r < rh; r += kTileRows) {
                const int z = z0 + r;
                if ((unsigned)z >= (unsigned)P.nz) continue;
                const unsigned char* src = base + ((long long)z * P.nx + x0) * 64 + lane * 16;
                const uint32_t dst = rec + r * rw * 16;
                // eight cells (lanes: four pieces of each) at a time
                for (int x = 0; x < rw; x += 8)
                    if (x + (lane >> 2) < rw && (unsigned)(x0 + x + (lane >> 2)) < (unsigned)P.nx)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + x * 16), "l"(src + x * 64)
                                     : "memory");
            }
            if (warp == 0) {
                int m;
                PathStep mine = B.next(c0, lane, m);
                const int n = c0 + lane - m;
                mine.off = ((dz < 0.0f ? n1 - n : n - n0) * rw + (dx < 0.0f ? m1 - m : m - m0)) * 16;
                s_path[lane] = mine;
                if (lane == 0) s_path[32] = mine;  // read ahead, never used
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            m0 = m1;
            if (live) {
                const unsigned char* q0 = s_rec + (warp * rw + lane) * 16;
                // the next step's record is read before this one is integrated
                auto piece = [&](int off, int c) { return *reinterpret_cast<const float4*>(q0 + off + c * kTilePlane); };
                PathStep ns = s_path[0];  // offsets within the staged planes
                float4 n0_ = piece((int)ns.off, 0), n1_ = piece((int)ns.off, 1), n2_ = piece((int)ns.off, 2), n3_ = piece((int)ns.off, 3);
#pragma unroll 4
                for (int q = 0; q < 32; ++q) {
                    const PathStep s = ns;
                    const float S[8] = {n0_.x, n0_.y, n0_.z, n0_.w, n1_.x, n1_.y, n1_.z, n1_.w};
                    const float chi[8] = {n2_.x, n2_.y, n2_.z, n2_.w, n3_.x, n3_.y, n3_.z, n3_.w};
                    ns = s_path[q + 1];
                    n0_ = piece((int)ns.off, 0);
                    n1_ = piece((int)ns.off, 1);
                    n2_ = piece((int)ns.off, 2);
                    n3_ = piece((int)ns.off, 3);
                    segments<8>(S, chi, s.nl2, I, T);
                    if constexpr (EXT) {
                        if (c0 + q == 0) {
#pragma unroll
                            for (int w = 0; w < 8; ++w) I[w] = 0.0f;
                        }
                    }
                    if (s.th >= t2 || ((q & 7) == 7 && ray_done<8>(I, T, stop))) {
                        live = false;
                        break;
                    }
                }
            }
        }
        const float wk = P.quad.w[k];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const float Iw = fmaf(T[w], P.i_bc, I[w]);
            Jw[w] = fmaf(wk, Iw, Jw[w]);
            const int l = b * 8 + w;
            if (P.I != nullptr && probe && l < P.n_lambda) P.I[((size_t)l * P.quad.n_dir + k) * P.n_probe + p] = Iw;
        }
    }
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const int l = b * 8 + w;
        if (probe && l < P.n_lambda) P.J[(size_t)l * P.n_probe + p] = Jw[w];
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
        p = (int)((unsigned)j * P.nx + i);  // may wrap beyond the last row, where it is not used
        return i < P.nx && j < P.nz;
    }
    i = j = 0;
    p = (blockIdx.x * tile_rows + row) * 32 + lane;
    if (p >= P.n_probe) return false;
    const int c = P.probes[p];
    if (c < 0 || (long long)c >= P.n_cells) {
        raise_status(P.status, DEX_ERR_TRAVERSAL_CAP);
        if (P.scanned) P.J[(size_t)(blockIdx.y * P.W) * P.n_probe + p] = 0.0f;  // it held the bound
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

// Several directions at a time of 32 probes, one per warp; the CTA then adds their
// intensities to J in the order of the directions, thread (warp, lane) the wavelengths
// warp, warp + warps, ... of its probe.
template <int W, bool COUNT, bool EXT = false>
__global__ void __launch_bounds__(256, 4) k_solve_dense_split(const DenseParams P)
{
    __shared__ PathStep s_path[8][32];
    __shared__ float s_I[8][W][32];
    __shared__ float s_J[W][32];
    const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warp = blockDim.x >> 5;
    int i, j, p;
    const bool live = dense_probe(P, 1, 0, lane, i, j, p);
    const float* rec0 = P.planes + ((size_t)b * P.n_cells + (size_t)j * P.nx + i) * (2 * W);
    const float stop = !COUNT && P.scanned && live ? stop_factor(P.J[(size_t)(b * W) * P.n_probe + p], P.i_bc) : -1.0f;
    for (int w = warp; w < W; w += n_warp) s_J[w][lane] = 0.0f;
    unsigned int nseg = 0;
    for (int k0 = 0; k0 < P.quad.n_dir; k0 += n_warp) {
        if (k0 + warp < P.quad.n_dir) {
            float I[W], T[W];
            dense_ray<W, COUNT, EXT>(P, s_path[warp], lane, i, j, rec0, P.quad.dx[k0 + warp], P.quad.dz[k0 + warp],
                                     stop, live, I, T, nseg);
#pragma unroll
            for (int w = 0; w < W; ++w) s_I[warp][w][lane] = fmaf(T[w], P.i_bc, I[w]);
        }
        __syncthreads();
        for (int w = warp; w < W; w += n_warp) {
            const int l = b * W + w;
            float Jw = s_J[w][lane];
            for (int g = 0; g < n_warp && k0 + g < P.quad.n_dir; ++g) {
                const float Iw = s_I[g][w][lane];
                Jw = fmaf(P.quad.w[k0 + g], Iw, Jw);
                if (P.I != nullptr && live && l < P.n_lambda) P.I[((size_t)l * P.quad.n_dir + k0 + g) * P.n_probe + p] = Iw;
            }
            s_J[w][lane] = Jw;
        }
        __syncthreads();
    }
    for (int w = warp; w < W; w += n_warp)
        if (live && b * W + w < P.n_lambda) P.J[(size_t)(b * W + w) * P.n_probe + p] = s_J[w][lane];
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
// 512 warps took 231 us one after the other, split 61 us (39 with a few records in
// flight per ray).
constexpr long long kSplitWarps = 2 * 152 * 32;

// Fewer than eight directions of a whole grid, W = 8: a split CTA is small and its rays
// part at once, so k_solve_dense_tile takes over as soon as its CTAs fill the chip (two
// per SM).  4 directions, split -> tile: 350 x 358, 16 wavelengths (360 CTAs) 1.36 ->
// 1.19 ms; 200 x 208, 24 (378) 472 -> 468 us; 8 (126) 184, tile 218; 6 directions,
// 256 x 264, 8 (176) 309, tile 421.  With more directions splitting stays ahead: 300 x
// 308, 9, 24 directions 3.41, tile 3.85 ms; 250 x 258, 24, 10 directions 1.37, 1.50.
constexpr long long kTileCtas = 2 * 152;

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
    // 64 bits: up to 2^31 - 1 probes, and the last step goes beyond them
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P.n_probe; p += gridDim.x * blockDim.x)
        J[p] = m;
}

// CTAs of k_solve_dense_tile
long long tile_grid(const DenseParams& P)
{
    return (P.nx + 31LL) / 32 * ((P.nz + kTileRows - 1) / kTileRows) * P.n_batch;
}

cudaError_t launch_dense_tile(cudaStream_t s, const DenseParams& P)
{
    const dim3 grid((unsigned)(tile_grid(P) / P.n_batch), (unsigned)P.n_batch);
    auto kernel = P.exclude_own ? k_solve_dense_tile<true> : k_solve_dense_tile<false>;
    const size_t smem = 4 * kTilePlane + 33 * sizeof(PathStep);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, kTileThreads, smem, s>>>(P);
    return cudaGetLastError();
}

template <int W>
void launch_dense_scan(cudaStream_t s, const DenseParams& P)
{
    const int parts = P.n_probe < kScanCtas ? P.n_probe : kScanCtas;
    k_dense_scan<W><<<dim3((unsigned)parts, (unsigned)P.n_batch), 256, 0, s>>>(P);
    const long long ctas = (P.n_probe + 1023LL) / 1024;
    k_dense_spread<<<dim3((unsigned)(ctas < 304 ? ctas : 304), (unsigned)P.n_batch), 256, 0, s>>>(P, parts);
}

template <int W>
void launch_dense_w(bool split, dim3 grid, cudaStream_t s, const DenseParams& P)
{
    if (P.scanned) launch_dense_scan<W>(s, P);
#define DEX_LAUNCH_DENSE(K)                                               \
    if (P.exclude_own) {                                                  \
        if (P.seg_count) K<W, true, true><<<grid, threads, 0, s>>>(P);    \
        else K<W, false, true><<<grid, threads, 0, s>>>(P);               \
    } else if (P.seg_count) {                                             \
        K<W, true><<<grid, threads, 0, s>>>(P);                           \
    } else {                                                              \
        K<W, false><<<grid, threads, 0, s>>>(P);                          \
    }
    // split: as many warps as share the directions evenly over rounds of at most eight
    // (idle ones would hold their registers: 350 x 358, 16 wavelengths, 4 directions on
    // eight warps 3.10 ms, on four 1.77)
    const int rounds = (P.quad.n_dir + 7) / 8;
    const int threads = split ? 32 * ((P.quad.n_dir + rounds - 1) / rounds) : 256;
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
    // scan the planes for the early termination's bound where the rays cross at least
    // sixteen times as many records, and 2^27 of them (two launches cost 5 us, a tenth
    // of the 128 x 128 solve with 16 directions, whose rays cross 2^25)
    const double crossed = (double)P.n_probe * P.quad.n_dir * 0.5 * ((double)P.nx + P.nz);
    P.scanned = !P.seg_count && crossed * P.n_batch >= 134217728.0 && crossed >= 16.0 * (double)P.n_cells;
    // one warp per 32 probes, or eight (one per direction) where those would not
    // fill the chip
    const long long warps = (P.n_probe + 31LL) / 32 * P.n_batch;
    const bool tile = P.W == 8 && P.probes == nullptr && !P.seg_count;
    const bool split = warps < kSplitWarps && !(tile && P.quad.n_dir < 8 && tile_grid(P) >= kTileCtas);
    if (!split && tile) {
        if (P.scanned) launch_dense_scan<8>(s, P);
        return launch_dense_tile(s, P);
    }
    const int rows = split ? 1 : 8;
    const unsigned tiles = P.probes == nullptr ? (unsigned)(((P.nx + 31) / 32) * ((P.nz + rows - 1) / rows))
                                               : (unsigned)((P.n_probe + 32LL * rows - 1) / (32 * rows));
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
