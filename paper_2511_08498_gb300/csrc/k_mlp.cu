// Learned Voigt-profile surrogate: a 3 -> 64 -> 64 -> 1 multilayer perceptron
// with tanh-form GELU activations that predicts ln H(a, x - u) from the
// wavelength offset x (Doppler widths, rest frame), the damping a and the
// projected velocity u (Doppler widths).  It stands in for the on-the-fly
// profile evaluation of the Core-and-Voigt treatment (Section 3.2); the exact
// HUM1WEI24 evaluation remains the fallback and the accuracy reference.
//
// Precision: weights are used as BF16 (rounded from an FP32 master copy), the
// hidden activations that feed the tensor cores are BF16, every sum is FP32.
//
// Tensor cores (tcgen05, kind::f16, accumulators in tensor memory) do every
// contraction over the hidden width or over the samples of a tile; CUDA cores
// do the 3-input first layer, the activations and the output dot product.
// Tiles hold 128 samples, sample = TMEM lane: inference one thread per sample (128
// threads), training two (256; each has half of the hidden units).  Per tile:
//   forward   D2 = H1 W2^T                      (M 128, N 64, K 64)
//   backward  D3 = Delta2 W2                    (M 128, N 64, K 64)   -> dL/dh1
//             D4 += [Delta2, dy h2]^T [H1, 1]   (M 128, N 80, K 128)  -> dW2, db2, dw3
//             D5 += [Delta1, .]^T [F, 1]        (M 128, N 16, K 128)  -> dW1, db1
// (tensor-memory columns: D2 0-63, D3 64-127, D4 128-207, D5 224-239 of 256).  The
// sums over samples read the row-per-sample tiles as MN-major operands, so nothing
// is stored twice; W2 likewise serves D2 and D3.
// D4 and D5 accumulate over all tiles of the CTA and are added to the global
// gradient once at the end.  Every mbarrier wait is bounded; on expiry the CTA
// records DEX_ERR_TIMEOUT, waits (bounded) once more, frees its tensor memory
// and returns.
#include <cmath>

#include "dex_internal.h"
#include "mlp.cuh"
#include "umma.cuh"
#include "voigt.cuh"

namespace dex {

namespace {

using namespace umma;
using mlp::kB1;
using mlp::kB2;
using mlp::kB3;
using mlp::kH;
using mlp::kW1;
using mlp::kW2;
using mlp::kW3;

constexpr int kTile = 128;  // samples per tile (MMA M)
constexpr int kWaitPolls = 1 << 20;

constexpr int kColsH1 = 80;  // 64 hidden units, the ones column 64, zero columns 65..79
constexpr int kColsF = 16;   // 3 features, the ones column 3, zero columns 4..15

// TMEM columns
constexpr uint32_t kColD2 = 0, kColD3 = 64, kColD4 = 128, kColD5 = 224;
constexpr uint32_t kColsTrain = 256, kColsInfer = 64;

// layer-1 weights by input feature: neighbouring units side by side
struct SmemNet {
    alignas(16) float w1t[3][kH];
    alignas(16) float b1[kH];
    float b2[kH], w3[kH], b3;
};

struct SmemInfer {
    alignas(16) unsigned char W2[kH * kH * 2];     // B of D2: rows out j, K in i
    alignas(16) unsigned char H1[kTile * kH * 2];  // A of D2: rows sample, K in i
    SmemNet net;
    unsigned long long mbar;
    unsigned int tmem;
};

struct SmemTrain {
    alignas(16) unsigned char W2[kH * kH * 2];          // [out j][in i]: B of D2, transposed B of D3
    alignas(16) unsigned char H1[kTile * kColsH1 * 2];  // [sample][in i, 1]: A of D2, transposed B of D4
    alignas(16) unsigned char D[kTile * 2 * kH * 2];    // [sample][delta2 | dy h2]: A of D3, transposed A of D4;
                                                        // then delta1 in its first half: transposed A of D5
    alignas(16) unsigned char F[kTile * kColsF * 2];    // [sample][feature, 1]: transposed B of D5
    SmemNet net;
    float y[2][kTile];
    float red_loss[4], red_gb3[4];
    unsigned long long mbar;
    unsigned int tmem;
};

// Dynamic shared memory requested per CTA bounds the CTAs per SM so that their
// tensor-memory allocations always fit its 512 columns: 8 x 64 inference, 2 x 256
// training.
constexpr size_t kSmemInfer = 27 * 1024;
constexpr size_t kSmemTrain = 80 * 1024;
static_assert(sizeof(SmemInfer) <= kSmemInfer && 9 * (kSmemInfer + 1024) > 228 * 1024, "inference shared memory");
static_assert(sizeof(SmemTrain) <= kSmemTrain && 3 * kSmemTrain > 228 * 1024, "training shared memory");

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// A sample's inputs as stored.
struct Sample {
    float x, a, u;
};

__device__ __forceinline__ Sample load_sample(const float* xau, long long s)
{
    return {xau[3 * s], xau[3 * s + 1], xau[3 * s + 2]};
}

// input features: x / 16, log10(a) + 2, u / 16; false (and zeros) for a
// non-finite input or a <= 0
__device__ __forceinline__ bool features(Sample v, float* f)
{
    const float x = v.x, a = v.a, u = v.u;
    if (!(a > 0.0f) || !isfinite(a) || !isfinite(x) || !isfinite(u)) {
        f[0] = f[1] = f[2] = 0.0f;
        return false;
    }
    mlp::features(x, a, u, f);
    return true;
}

__device__ __forceinline__ unsigned int pack_bf16(float2 v)
{
    const __nv_bfloat162 b = __float22bfloat162_rn(v);
    return *reinterpret_cast<const unsigned int*>(&b);
}

__device__ void stage_weights(SmemNet& net, unsigned char* W2, const float* __restrict__ p)
{
    const int t = threadIdx.x;
    for (int q = 2 * t; q < kH * kH; q += 2 * blockDim.x)
        *reinterpret_cast<unsigned int*>(W2 + tile_offset(q / kH, q % kH, kH)) =
            pack_bf16(make_float2(p[kW2 + q], p[kW2 + q + 1]));
    for (int q = t; q < kH * 3; q += blockDim.x) net.w1t[q % 3][q / 3] = bf16_round(p[kW1 + q]);
    if (t < kH) {
        net.b1[t] = p[kB1 + t];
        net.b2[t] = p[kB2 + t];
        net.w3[t] = bf16_round(p[kW3 + t]);
    }
    if (t == 0) net.b3 = p[kB3];
}

// The larger of a and b, NaN if either is.
__device__ __forceinline__ float max_nan(float a, float b)
{
    float m;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
    return m;
}

// GELU of two hidden units on the packed FP32 pipe.  The two logistic functions share
// one reciprocal, 1/a = b / (a b): three special-function operations for two
// activations instead of four, in kernels whose issue slots and FP32 pipe they share.
// Pre-activations count as at least -7.6, where 2^x is 2^62.7, so that the product of
// two stays below 2^126 and its reciprocal is normal; there and below the activation
// comes out as -1e-18 (its value is between that and 0).
struct Gelu2 {
    float2 z, z2, s;
    __device__ __forceinline__ explicit Gelu2(float2 zz) : z(make_float2(max_nan(zz.x, -7.6f), max_nan(zz.y, -7.6f)))
    {
        // -2 log2(e) c (z + k z^3), c = sqrt(2 / pi), k = 0.044715
        constexpr float c1 = -2.3022081986f, c2 = -0.1029432397f;
        z2 = __fmul2_rn(z, z);
        const float2 a = __fmul2_rn(z, __ffma2_rn(make_float2(c2, c2), z2, make_float2(c1, c1)));
        const float2 d = __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(mlp::mlp_ex2(a.x), mlp::mlp_ex2(a.y)));
        const float r = mlp::mlp_rcp(d.x * d.y);
        s = __fmul2_rn(make_float2(r, r), make_float2(d.y, d.x));
    }
    __device__ __forceinline__ float2 g() const { return __fmul2_rn(z, s); }
    // s + z s (1 - s) 2 c (1 + 3 k z^2), from g = z s
    __device__ __forceinline__ float2 dg(float2 g) const
    {
        constexpr float k0 = 1.5957691216f, k1 = 0.2140644488f;  // 2 c, 6 c k
        const float2 q = __ffma2_rn(make_float2(-g.x, -g.y), s, g);
        return __ffma2_rn(q, __ffma2_rn(make_float2(k1, k1), z2, make_float2(k0, k0)), s);
    }
};

// GELU of two hidden units, every lane rounded as mlp::gelu(z).g: for activations
// that are rounded to bfloat16 next, where another float32 rounding now and then
// lands on the other side of a bfloat16 boundary.
__device__ __forceinline__ float2 gelu2(float2 z)
{
    const float c = 0.79788456080286536f, k = 0.044715f;
    const float m2log2e = -2.8853900817779268f;
    const float2 z2 = __fmul2_rn(z, z);
    const float2 u = __fmul2_rn(__fmul2_rn(make_float2(c, c), z), __ffma2_rn(make_float2(k, k), z2, make_float2(1.0f, 1.0f)));
    const float2 a = __fmul2_rn(u, make_float2(m2log2e, m2log2e));
    const float2 d = __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(mlp::mlp_ex2(a.x), mlp::mlp_ex2(a.y)));
    return __fmul2_rn(z, make_float2(mlp::mlp_rcp(d.x), mlp::mlp_rcp(d.y)));
}

// z1 of units i .. i + 3
__device__ __forceinline__ void layer1_z4(const SmemNet& net, const float* f, int i, float2& za, float2& zb)
{
    const float4 b = *reinterpret_cast<const float4*>(&net.b1[i]);
    const float4 w0 = *reinterpret_cast<const float4*>(&net.w1t[0][i]);
    const float4 w1 = *reinterpret_cast<const float4*>(&net.w1t[1][i]);
    const float4 w2 = *reinterpret_cast<const float4*>(&net.w1t[2][i]);
    const float2 f0 = make_float2(f[0], f[0]), f1 = make_float2(f[1], f[1]), f2 = make_float2(f[2], f[2]);
    za = __ffma2_rn(make_float2(w2.x, w2.y), f2,
                    __ffma2_rn(make_float2(w1.x, w1.y), f1, __ffma2_rn(make_float2(w0.x, w0.y), f0, make_float2(b.x, b.y))));
    zb = __ffma2_rn(make_float2(w2.z, w2.w), f2,
                    __ffma2_rn(make_float2(w1.z, w1.w), f1, __ffma2_rn(make_float2(w0.z, w0.w), f0, make_float2(b.z, b.w))));
}

// one MMA chain: D (+)= A B^T over K/16 K-steps, issued by the calling thread
__device__ __forceinline__ void mma_chain(uint32_t d, Operand A, Operand B, int K, uint32_t idesc, bool accumulate)
{
    for (int k = 0; k < K / 16; ++k) mma_bf16(d, A.step(k), B.step(k), idesc, accumulate || k > 0);
}

// make every thread's shared-memory writes and TMEM reads ordered before the
// MMAs thread 0 issues next
__device__ __forceinline__ void sync_for_mma()
{
    fence_async_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
}

// bounded wait by every thread; returns true on success for the whole CTA
__device__ __forceinline__ bool wait_all(unsigned long long* mbar, uint32_t& phase)
{
    const bool ok = mbar_wait(mbar, phase, kWaitPolls);
    phase ^= 1u;
    const bool all = !__syncthreads_or(ok ? 0 : 1);
    fence_after_sync();
    return all;
}

// ------------------------------------------------------------ inference --
// Bound by instruction issue (about 10 per activation) with the FP32 pipe and the
// special-function units at 60% and 40%; eight CTAs per
// SM, whose phases interleave, hide the barriers and the MMA's latency.
__global__ void __launch_bounds__(128, 8) k_mlp_forward(const MlpParams P)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SmemInfer& sm = *reinterpret_cast<SmemInfer*>(smem_raw);
    const int t = threadIdx.x, warp = t >> 5;
    stage_weights(sm.net, sm.W2, P.params);
    if (t == 0) mbar_init(&sm.mbar, 1);
    if (warp == 0) tmem_alloc(&sm.tmem, kColsInfer);
    sync_for_mma();
    const uint32_t tm = sm.tmem;
    uint32_t phase = 0;
    const long long n_tiles = (P.n + kTile - 1) / kTile;
    bool ok = true;
    // the next tile's inputs are on their way while this one is evaluated
    const long long stride = (long long)gridDim.x * kTile;
    long long s = blockIdx.x * (long long)kTile + t;
    Sample next = s < P.n ? load_sample(P.xau, s) : Sample{0.0f, 1.0f, 0.0f};
    for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, s += stride) {
        bool valid = s < P.n;
        float f[3] = {0.0f, 0.0f, 0.0f};
        const Sample now = next;
        if (s + stride < P.n) next = load_sample(P.xau, s + stride);
        if (valid && !features(now, f)) {
            raise_status(P.status, DEX_ERR_NUMERIC);
            valid = false;
        }
#pragma unroll 2
        for (int i0 = 0; i0 < kH; i0 += 8) {
            uint4 h;
            unsigned int* hw = reinterpret_cast<unsigned int*>(&h);
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                float2 za, zb;
                layer1_z4(sm.net, f, i0 + 2 * q, za, zb);
                hw[q] = pack_bf16(gelu2(za));
                hw[q + 1] = pack_bf16(gelu2(zb));
            }
            *reinterpret_cast<uint4*>(sm.H1 + tile_offset(t, i0, kTile)) = h;
        }
        sync_for_mma();
        if (t == 0) {
            mma_chain(tm + kColD2, {smem_u32(sm.H1), kTile, false}, {smem_u32(sm.W2), kH, false}, kH,
                      idesc_bf16_f32(kTile, kH), false);
            mma_commit(&sm.mbar);
        }
        if (!(ok = wait_all(&sm.mbar, phase))) break;
        // output unit: two partial sums (even and odd hidden units) on the packed pipe
        float2 y2 = make_float2(sm.net.b3, 0.0f);
#pragma unroll 1
        for (int j = 0; j < kH; j += 16) {
            float z[16];
            tmem_ld16(tmem_at(tm, warp * 32, kColD2 + j), z);
#pragma unroll
            for (int q = 0; q < 16; q += 4) {
                const float4 b = *reinterpret_cast<const float4*>(&sm.net.b2[j + q]);
                const float4 w = *reinterpret_cast<const float4*>(&sm.net.w3[j + q]);
                const Gelu2 a(__fadd2_rn(make_float2(z[q], z[q + 1]), make_float2(b.x, b.y)));
                const Gelu2 c(__fadd2_rn(make_float2(z[q + 2], z[q + 3]), make_float2(b.z, b.w)));
                y2 = __ffma2_rn(make_float2(w.z, w.w), c.g(), __ffma2_rn(make_float2(w.x, w.y), a.g(), y2));
            }
        }
        const float y = y2.x + y2.y;
        if (valid) P.out[s] = y;
    }
    if (!ok) {
        raise_status(P.status, DEX_ERR_TIMEOUT);
        mbar_wait(&sm.mbar, phase ^ 1u, kWaitPolls);  // the MMA still in flight, if any
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tm, kColsInfer);
}

// ------------------------------------------------------------- training --
// Four consecutive gradient entries; one 16-byte reduction where aligned.
__device__ __forceinline__ void add4(float* p, float4 v, bool wide)
{
    if (wide) {
        atomicAdd(reinterpret_cast<float4*>(p), v);
    } else {
        atomicAdd(p, v.x);
        atomicAdd(p + 1, v.y);
        atomicAdd(p + 2, v.z);
        atomicAdd(p + 3, v.w);
    }
}

// A minibatch is about one tile per CTA, so a step's time is one tile's chain of
// phases: two threads per sample halve it, each keeping its 32 units' activations
// and derivatives in registers from the pass that first needs them.
__global__ void __launch_bounds__(256, 2) k_mlp_grad(const MlpParams P)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SmemTrain& sm = *reinterpret_cast<SmemTrain*>(smem_raw);
    constexpr int kHalf = kH / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quarter = warp & 3, t = quarter * 32 + lane;  // sample of the tile, TMEM lane
    const int h0 = (warp >> 2) * kHalf;                     // first hidden unit of this thread
    const bool first = h0 == 0;
    stage_weights(sm.net, sm.W2, P.params);
    // constant columns: H1 column 64 = 1, 65..79 = 0; F column 3 = 1, 4..15 = 0
    if (first) {
        const uint4 one = make_uint4(0x3f80u, 0u, 0u, 0u), zero = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(sm.H1 + tile_offset(t, kH, kTile)) = one;
        *reinterpret_cast<uint4*>(sm.H1 + tile_offset(t, kH + 8, kTile)) = zero;
        *reinterpret_cast<uint4*>(sm.F + tile_offset(t, 8, kTile)) = zero;
    }
    if (threadIdx.x == 0) mbar_init(&sm.mbar, 1);
    if (warp == 0) tmem_alloc(&sm.tmem, kColsTrain);
    sync_for_mma();
    const uint32_t tm = sm.tmem;
    const Operand W2{smem_u32(sm.W2), kH, false}, W2t{smem_u32(sm.W2), kH, true};
    const Operand H1{smem_u32(sm.H1), kTile, false}, H1t{smem_u32(sm.H1), kTile, true};
    const Operand D{smem_u32(sm.D), kTile, false}, Dt{smem_u32(sm.D), kTile, true}, Ft{smem_u32(sm.F), kTile, true};
    uint32_t phase = 0;
    const long long n_tiles = (P.n + kTile - 1) / kTile;
    bool ok = true, any = false;
    float loss = 0.0f, gb3 = 0.0f;
    for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const long long s = tile * kTile + t;
        bool valid = s < P.n;
        float f[3] = {0.0f, 0.0f, 0.0f}, target = 0.0f;
        if (valid) {
            target = P.target[s];
            if (!features(load_sample(P.xau, s), f) || !isfinite(target)) {
                raise_status(P.status, DEX_ERR_NUMERIC);
                valid = false;
                f[0] = f[1] = f[2] = 0.0f;
            }
        }
        // layer 1
        float2 dg1[kHalf / 2];
#pragma unroll
        for (int i0 = 0; i0 < kHalf; i0 += 8) {
            uint4 h;
            unsigned int* hw = reinterpret_cast<unsigned int*>(&h);
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                float2 za, zb;
                layer1_z4(sm.net, f, h0 + i0 + 2 * q, za, zb);
                const Gelu2 a(za), b(zb);
                const float2 ga = a.g(), gb = b.g();
                hw[q] = pack_bf16(ga);
                hw[q + 1] = pack_bf16(gb);
                dg1[i0 / 2 + q] = a.dg(ga);
                dg1[i0 / 2 + q + 1] = b.dg(gb);
            }
            *reinterpret_cast<uint4*>(sm.H1 + tile_offset(t, h0 + i0, kTile)) = h;
        }
        if (first)
            *reinterpret_cast<uint4*>(sm.F + tile_offset(t, 0, kTile)) =
                make_uint4(pack_bf16(make_float2(f[0], f[1])), pack_bf16(make_float2(f[2], 1.0f)), 0u, 0u);
        sync_for_mma();
        if (threadIdx.x == 0) {
            mma_chain(tm + kColD2, H1, W2, kH, idesc_bf16_f32(kTile, kH), false);
            mma_commit(&sm.mbar);
        }
        if (!(ok = wait_all(&sm.mbar, phase))) break;

        // forward output, then dy
        float2 g2[kHalf / 2], dg2[kHalf / 2], y2 = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int c = 0; c < kHalf; c += 16) {
            float z[16];
            tmem_ld16(tmem_at(tm, quarter * 32, kColD2 + h0 + c), z);
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
                const float2 b = *reinterpret_cast<const float2*>(&sm.net.b2[h0 + c + q]);
                const float2 w = *reinterpret_cast<const float2*>(&sm.net.w3[h0 + c + q]);
                const Gelu2 a(__fadd2_rn(make_float2(z[q], z[q + 1]), b));
                const float2 g = a.g();
                y2 = __ffma2_rn(w, g, y2);
                g2[(c + q) / 2] = g;
                dg2[(c + q) / 2] = __fmul2_rn(w, a.dg(g));
            }
        }
        sm.y[warp >> 2][t] = y2.x + y2.y;
        __syncthreads();
        const float y = sm.net.b3 + (sm.y[0][t] + sm.y[1][t]);
        const float r = valid ? y - target : 0.0f;
        const float dy = 2.0f * r;
        if (first) {
            loss = fmaf(r, r, loss);
            gb3 += dy;
        }
        // delta2 = dy w3 g'(z2) and dy h2, row by sample
        const float2 dy2 = make_float2(dy, dy);
#pragma unroll
        for (int c = 0; c < kHalf; c += 8) {
            uint4 d, e;
            unsigned int *dw = reinterpret_cast<unsigned int*>(&d), *ew = reinterpret_cast<unsigned int*>(&e);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                dw[q] = pack_bf16(__fmul2_rn(dy2, dg2[c / 2 + q]));
                ew[q] = pack_bf16(__fmul2_rn(dy2, g2[c / 2 + q]));
            }
            *reinterpret_cast<uint4*>(sm.D + tile_offset(t, h0 + c, kTile)) = d;
            *reinterpret_cast<uint4*>(sm.D + tile_offset(t, kH + h0 + c, kTile)) = e;
        }
        sync_for_mma();
        if (threadIdx.x == 0) {
            mma_chain(tm + kColD3, D, W2t, kH, idesc_bf16_f32(kTile, kH, false, true), false);
            mma_chain(tm + kColD4, Dt, H1t, kTile, idesc_bf16_f32(kTile, kColsH1, true, true), any);
            mma_commit(&sm.mbar);
        }
        if (!(ok = wait_all(&sm.mbar, phase))) break;

        // delta1 = (dL/dh1) g'(z1) over delta2
#pragma unroll
        for (int c = 0; c < kHalf; c += 16) {
            float dh[16];
            tmem_ld16(tmem_at(tm, quarter * 32, kColD3 + h0 + c), dh);
#pragma unroll
            for (int q0 = 0; q0 < 16; q0 += 8) {
                uint4 d;
                unsigned int* dw = reinterpret_cast<unsigned int*>(&d);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    dw[q] = pack_bf16(__fmul2_rn(make_float2(dh[q0 + 2 * q], dh[q0 + 2 * q + 1]), dg1[(c + q0) / 2 + q]));
                *reinterpret_cast<uint4*>(sm.D + tile_offset(t, h0 + c + q0, kTile)) = d;
            }
        }
        sync_for_mma();
        if (threadIdx.x == 0) {
            mma_chain(tm + kColD5, Dt, Ft, kTile, idesc_bf16_f32(kTile, kColsF, true, true), any);
            mma_commit(&sm.mbar);
        }
        if (!(ok = wait_all(&sm.mbar, phase))) break;
        any = true;
    }
    if (!ok) {
        raise_status(P.status, DEX_ERR_TIMEOUT);
        mbar_wait(&sm.mbar, phase ^ 1u, kWaitPolls);
    } else {
        const float inv_n = 1.0f / (float)P.n;
        // loss and db3: warp sums, then one atomic per CTA
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            loss += __shfl_xor_sync(0xffffffffu, loss, o);
            gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        }
        if (first && lane == 0) {
            sm.red_loss[warp] = loss;
            sm.red_gb3[warp] = gb3;
        }
        __syncthreads();
        if (threadIdx.x == 0 && any) {
            atomicAdd(P.loss, (sm.red_loss[0] + sm.red_loss[1] + sm.red_loss[2] + sm.red_loss[3]) * inv_n);
            atomicAdd(P.grad + kB3, (sm.red_gb3[0] + sm.red_gb3[1] + sm.red_gb3[2] + sm.red_gb3[3]) * inv_n);
        }
        if (any) {
            // D4 row r < 64: dW2[r][0..63], db2[r] (column 64); row 64 + j: dw3[j] (column 64)
            const bool wide = (reinterpret_cast<uintptr_t>(P.grad) & 15) == 0;
            float v[16];
#pragma unroll 1
            for (int c = h0; c < h0 + kHalf; c += 16) {
                tmem_ld16(tmem_at(tm, quarter * 32, kColD4 + c), v);
                if (t < kH)
#pragma unroll
                    for (int q = 0; q < 16; q += 4)
                        add4(P.grad + kW2 + t * kH + c + q,
                             make_float4(v[q] * inv_n, v[q + 1] * inv_n, v[q + 2] * inv_n, v[q + 3] * inv_n), wide);
            }
            if (first) {
                tmem_ld16(tmem_at(tm, quarter * 32, kColD4 + kH), v);
                if (t < kH) atomicAdd(P.grad + kB2 + t, v[0] * inv_n);
                else atomicAdd(P.grad + kW3 + (t - kH), v[0] * inv_n);
            } else {
                // D5 row r < 64: dW1[r][0..2], db1[r] (column 3)
                tmem_ld16(tmem_at(tm, quarter * 32, kColD5), v);
                if (t < kH) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) atomicAdd(P.grad + kW1 + 3 * t + k, v[k] * inv_n);
                    atomicAdd(P.grad + kB1 + t, v[3] * inv_n);
                }
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tm, kColsTrain);
}

// the sums' start: one launch in place of two memsets
__global__ void k_mlp_zero(float* __restrict__ grad, int n, float* __restrict__ loss)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n) grad[q] = 0.0f;
    if (q == 0) *loss = 0.0f;
}

// ----------------------------------------------------------------- Adam --
__global__ void k_mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const float gq = g[q];
    const float mq = fmaf(b1, m[q], (1.0f - b1) * gq);
    const float vq = fmaf(b2, v[q], (1.0f - b2) * gq * gq);
    m[q] = mq;
    v[q] = vq;
    p[q] -= lr * (mq * c1) / (sqrtf(vq * c2) + eps);
}

// ------------------------------------------------------ training targets --
__global__ void k_mlp_targets(long long n, const float* __restrict__ xau, float* __restrict__ out, VoigtCoef C)
{
    stage_dawson(C);
    __syncthreads();
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x)
        out[s] = logf(voigt_h<false>(C, xau[3 * s + 1], xau[3 * s] - xau[3 * s + 2]));
}

}  // namespace

int mlp_param_count() { return mlp::kParams; }

static int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

cudaError_t launch_mlp_forward(cudaStream_t s, const MlpParams& P)
{
    if (P.n == 0) return cudaSuccess;
    const int sms = sm_count();
    if (sms == 0) return cudaErrorInvalidDevice;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemInfer);
    if (e == cudaSuccess)  // room for all eight CTAs
        e = cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    const long long tiles = (P.n + kTile - 1) / kTile;
    // Setting up a CTA (weights, tensor memory) costs about as much as two tiles, so small
    // numbers of tiles go to as few CTAs per SM as get 2.3 tiles each, from two to the
    // eight that fit: 311000 samples 38.6 us with one tile per CTA, 27.2 with six CTAs per
    // SM; 117000 19.1, 17.0 with three; 78000 15.9, 13.9 with two.  From sixteen tiles per
    // slot on CTAs of eight tiles each: one CTA per slot for all of them left the younger
    // CTAs of an SM behind (2^22 samples 225 us against 216), while 1.5 million samples
    // take 87.7 us with one per slot, 89.6 with CTAs of eight tiles.
    const long long slots = 8LL * sms;
    const long long k = llround((double)tiles / (2.3 * sms));
    const long long grid = tiles >= 16 * slots ? (tiles + 7) / 8 : min(tiles, max(2LL, min(8LL, k)) * sms);
    k_mlp_forward<<<(unsigned)grid, 128, kSmemInfer, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_mlp_grad(cudaStream_t s, const MlpParams& P)
{
    k_mlp_zero<<<(mlp_param_count() + 255) / 256, 256, 0, s>>>(P.grad, mlp_param_count(), P.loss);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || P.n == 0) return e;
    const int sms = sm_count();
    if (sms == 0) return cudaErrorInvalidDevice;
    e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemTrain);
    if (e != cudaSuccess) return e;
    const long long tiles = (P.n + kTile - 1) / kTile;
    const long long grid = tiles < 2LL * sms ? tiles : 2LL * sms;
    k_mlp_grad<<<(unsigned)grid, 256, kSmemTrain, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(cudaStream_t s, float* p, const float* g, float* m, float* v, int step, float lr,
                            float b1, float b2, float eps)
{
    const int n = mlp_param_count();
    const float c1 = (float)(1.0 / (1.0 - pow((double)b1, step)));
    const float c2 = (float)(1.0 / (1.0 - pow((double)b2, step)));
    k_mlp_adam<<<(n + 255) / 256, 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t launch_mlp_targets(cudaStream_t s, long long n, const float* xau, float* out)
{
    if (n == 0) return cudaSuccess;
    const long long ctas = (n + 255) / 256;
    k_mlp_targets<<<(unsigned)(ctas < 152 * 8 ? ctas : 152 * 8), 256, 0, s>>>(n, xau, out, voigt_coefficients());
    return cudaGetLastError();
}

}  // namespace dex
