// Voigt function H(a, x) = Re w(x + i a) on the GPU: the HUM1WEI24 form named in
// Section 3.2 (Schreier 2018), float32, with changes for float32 conditioning and
// for the number of instructions.  a < 0.25 (every damping of a resonance line):
//   |x| + a >= 15  : region I of Humlicek (1982), w = i z / (sqrt(pi) (z^2 - 1/2));
//   6 <= |x| + a < 15 : the asymptotic series w = (i / sqrt(pi)) sum_k m_k z^-(2k+1),
//                    m_k = (2k-1)!! / 2^k (Abramowitz & Stegun 7.1.23), whose real
//                    part is expanded in (a / x)^2: with y = 1 / x^2, e = a^2 y and
//                    Re[i (1 + i a/x)^-n] = n a/x - n(n+1)(n+2)/3! (a/x)^3 + ...,
//                    H = (a y / sqrt(pi)) (A(y) - e (B(y) - e C(y)));
//   |x| + a < 6    : w = e^{-z^2} + (2 i / sqrt(pi)) D(z), D Dawson's integral, so
//                    H = e^{a^2 - x^2} cos(2 a x) - (2 / sqrt(pi)) Im D(x + i a),
//                    with Im D from D's Taylor series about the nearest multiple of
//                    1/8 on the real axis: real coefficients, a complex argument
//                    delta + i a, so the two-term recurrence b_k = c_k + 2 delta
//                    b_{k+1} - (delta^2 + a^2) b_{k+2} gives Im D = a b_1.
// a >= 0.25 (voigt_thick):
//   |x| + a >= 15  : region I;
//   5 <= |x| + a < 15 : 8-term Laplace continued fraction (Gautschi 1970),
//                    w = (i/sqrt(pi)) / (z - (1/2)/(z - 1/(z - (3/2)/...)));
//   |x| + a < 5    : Weideman (1994), N = 24,
//                    w = 2 p(Z) / (L - i z)^2 + 1 / (sqrt(pi) (L - i z)),
//                    Z = (L + i z) / (L - i z), p(Z) = sum_{n=1..24} a_n Z^(n-1).
// Why: at small damping the line wing H ~ a / (sqrt(pi) x^2) is a small difference
// of O(0.05) real parts in Weideman's form, and in float32 the complex sum loses
// up to ~1e-3 of it.  In the three forms above nothing cancels: a float32 model of
// them stays within 6e-7 relative of the Faddeeva function for a from 1e-4 to 0.25
// and |x| + a < 15, the kernel within 6.4e-7 (8.2e-7 down to a = 1e-6; the Taylor
// series about the real axis built on Weideman's sum that they replaced: 9e-6 and, at
// a = 1e-6, 6e-4).  Cost: about 36 instructions in the core and 25 in the wing against
// 165 and 60; the Core-and-Voigt solve, whose warps meet both, ran at the rate it
// fetched them.
// The coefficients (a_n: Fourier coefficients of exp(-t^2)(L^2 + t^2), t = L
// tan(theta/2); D's Taylor coefficients) are computed on the host and passed as a
// kernel parameter; D's are read at a node per lane, so kernels copy them to
// shared memory (stage_dawson).
#pragma once

#include <cuda_runtime.h>

namespace dex {

constexpr int kWeidemanN = 24;
constexpr float kWeidemanL = 4.1195342878f;         // sqrt(24 / sqrt 2)
constexpr float kInvSqrtPi = 0.56418958354775628f;
constexpr int kDawsonNodes = 49;                    // x = 0, 1/8, ..., 6
constexpr int kDawsonTerms = 8;                     // c_1 .. c_8 of each node

struct VoigtCoef {
    float a[kWeidemanN];  // a_1 .. a_24
    alignas(16) float dawson[kDawsonNodes * kDawsonTerms];
};

// Host: the coefficients, computed once in double from the definitions
// (trapezoid rule on 4N points; D from its power series times e^{-x^2}, its
// derivatives from D' = 1 - 2 x D, D^(n+1) = -2 x D^(n) - 2 n D^(n-1)) and rounded
// to float.
const VoigtCoef& voigt_coefficients();

// The shared-memory copy of D's coefficients of the kernel that calls it.
__device__ __forceinline__ float* dawson_table()
{
    __shared__ __align__(16) float s_dawson[kDawsonNodes * kDawsonTerms];
    return s_dawson;
}

// Fill it; the caller synchronises the CTA before voigt_h.
__device__ __forceinline__ void stage_dawson(const VoigtCoef& C)
{
    float* t = dawson_table();
    for (int q = threadIdx.x; q < kDawsonNodes * kDawsonTerms; q += blockDim.x) t[q] = C.dawson[q];
}

// region I: Re[i z / (sqrt(pi) (z^2 - 1/2))], z = x + i a
__device__ __forceinline__ float voigt_far(float a, float x)
{
    const float zr = x, zi = a;
    const float dr = zr * zr - zi * zi - 0.5f, di = 2.0f * zr * zi;   // z^2 - 1/2
    const float nr = -zi, ni = zr;                                     // i z
    const float inv = __fdividef(1.0f, dr * dr + di * di);
    return kInvSqrtPi * (nr * dr + ni * di) * inv;                     // Re(n / d)
}

__device__ __forceinline__ float voigt_thick_inline(const VoigtCoef& C, float a, float x)
{
    const float s = fabsf(x) + a;
    if (s >= 15.0f) return voigt_far(a, x);
    if (s >= 5.0f) {
        // f = z - (k/2) / f, innermost k = 8; w = (i / sqrt(pi)) / f -> Re w = Im f / (sqrt(pi) |f|^2)
        float fr = x, fi = a;
#pragma unroll
        for (int k = 8; k >= 1; --k) {
            const float c = 0.5f * (float)k;
            const float q = __fdividef(c, fmaf(fr, fr, fi * fi));
            fr = fmaf(-q, fr, x);
            fi = fmaf(q, fi, a);
        }
        return kInvSqrtPi * __fdividef(fi, fmaf(fr, fr, fi * fi));
    }
    // den = L - i z = (L + a) - i x ; num = L + i z = (L - a) + i x
    const float denr = kWeidemanL + a, deni = -x;
    const float numr = kWeidemanL - a, numi = x;
    // correctly rounded: a 2-ulp reciprocal would be amplified by the cancelling sum
    const float dd = __frcp_rn(fmaf(denr, denr, deni * deni));
    // Z = num / den
    const float Zr = (numr * denr + numi * deni) * dd;
    const float Zi = (numi * denr - numr * deni) * dd;
    float pr = C.a[kWeidemanN - 1], pi = 0.0f;
#pragma unroll
    for (int n = kWeidemanN - 2; n >= 0; --n) {  // Horner
        const float tr = fmaf(pr, Zr, fmaf(-pi, Zi, C.a[n]));
        pi = fmaf(pr, Zi, pi * Zr);
        pr = tr;
    }
    // 1 / den and 1 / den^2
    const float ir = denr * dd, ii = -deni * dd;
    const float i2r = ir * ir - ii * ii, i2i = 2.0f * ir * ii;
    return 2.0f * (pr * i2r - pi * i2i) + kInvSqrtPi * ir;
}

static __device__ __noinline__ float voigt_thick(const VoigtCoef& C, float a, float x)
{
    return voigt_thick_inline(C, a, x);
}

// m_k (2k+1) ... (2k+2t+1) / (2t+1)! of the asymptotic series
__host__ __device__ constexpr float wing_coef(int k, int t)
{
    double v = 1.0;
    for (int j = 1; j <= k; ++j) v *= (2.0 * j - 1.0) / 2.0;
    for (int q = 1; q <= 2 * t + 1; ++q) v *= (2.0 * k + q) / q;
    return (float)v;
}

template <int N, int T>
__device__ __forceinline__ float wing_poly(float y)
{
    float p = wing_coef(N - 1, T);
#pragma unroll
    for (int k = N - 2; k >= 0; --k) p = fmaf(p, y, wing_coef(k, T));
    return p;
}

// CALL: a >= 0.25 in a called function, for kernels that meet it rarely among much other
// code; elementwise ones inline it (2^22 values: 53 -> 41 us).
template <bool CALL = true>
__device__ __forceinline__ float voigt_h(const VoigtCoef& C, float a, float x)
{
    if (!(a < 0.25f)) return CALL ? voigt_thick(C, a, x) : voigt_thick_inline(C, a, x);
    const float ax = fabsf(x), s = ax + a;
    if (s >= 15.0f) return voigt_far(a, x);
    if (s >= 6.0f) {
        const float y = __fdividef(1.0f, ax * ax), e = a * a * y;
        const float q = fmaf(-e, wing_poly<2, 2>(y), wing_poly<5, 1>(y));
        return kInvSqrtPi * a * y * fmaf(-e, q, wing_poly<8, 0>(y));
    }
    const int node = min((int)(ax * 8.0f + 0.5f), kDawsonNodes - 1);
    const float d = fmaf((float)node, -0.125f, ax), d2 = d + d, nr2 = -fmaf(a, a, d * d);
    const float4* t = reinterpret_cast<const float4*>(dawson_table() + node * kDawsonTerms);
    const float4 lo = t[0], hi = t[1];  // c_1 .. c_4, c_5 .. c_8
    float b2 = hi.w, b1 = fmaf(d2, hi.w, hi.z), b0;
#define DEX_DAWSON_STEP(c)                \
    b0 = fmaf(d2, b1, fmaf(nr2, b2, c));  \
    b2 = b1;                              \
    b1 = b0;
    DEX_DAWSON_STEP(hi.y)
    DEX_DAWSON_STEP(hi.x)
    DEX_DAWSON_STEP(lo.w)
    DEX_DAWSON_STEP(lo.z)
    DEX_DAWSON_STEP(lo.y)
    DEX_DAWSON_STEP(lo.x)
#undef DEX_DAWSON_STEP
    // e^{a^2 - x^2} with the exponent's rounding error carried to first order
    const float l2e = 1.4426950408889634f, ln2 = 0.69314718f;
    const float r = (a - ax) * (a + ax), p = r * l2e;
    float ex;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(p));
    ex = fmaf(ex * ln2, fmaf(r, l2e, -p), ex);
    return fmaf(-2.0f * kInvSqrtPi * a, b1, ex * __cosf(2.0f * a * ax));
}

}  // namespace dex
