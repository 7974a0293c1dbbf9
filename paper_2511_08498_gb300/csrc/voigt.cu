// Voigt function: host-side coefficients (Weideman's sum, Dawson's integral) and
// an elementwise kernel behind dex_voigt.
#include <cmath>
#include <mutex>

#include "dex_internal.h"
#include "voigt.cuh"

namespace dex {

namespace {

void weideman_coefficients(double* a, int n)
{
    const int M = 2 * n;
    const double L = std::sqrt(n / std::sqrt(2.0));
    for (int m = 1; m <= n; ++m) {
        double s = 0.0;
        for (int k = -M + 1; k <= M - 1; ++k) {  // theta = -pi contributes f = 0
            const double theta = k * M_PI / M;
            const double t = L * std::tan(theta / 2.0);
            s += std::exp(-t * t) * (L * L + t * t) * std::cos(m * theta);
        }
        a[m - 1] = s / (2.0 * M);
    }
}

// D^(n)(x) / n!, n = 1 .. kDawsonTerms
void dawson_coefficients(double x, float* c)
{
    // D(x) = e^{-x^2} sum_k x^(2k+1) / (k! (2k+1))
    double term = x, sum = x;
    for (int k = 1; k < 200; ++k) {
        term *= x * x / k;
        sum += term / (2 * k + 1);
    }
    double prev = std::exp(-x * x) * sum, cur = 1.0 - 2.0 * x * prev, fact = 1.0;
    for (int n = 1; n <= kDawsonTerms; ++n) {
        fact *= n;
        c[n - 1] = (float)(cur / fact);
        const double next = -2.0 * x * cur - 2.0 * n * prev;
        prev = cur;
        cur = next;
    }
}

__global__ void k_voigt(const VoigtCoef C, long long n, const float* __restrict__ a, const float* __restrict__ x,
                        float* __restrict__ h)
{
    stage_dawson(C);
    __syncthreads();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        h[i] = voigt_h<false>(C, a[i], x[i]);
}

}  // namespace

const VoigtCoef& voigt_coefficients()
{
    static VoigtCoef coef;
    static std::once_flag once;
    std::call_once(once, [] {
        double a[kWeidemanN];
        weideman_coefficients(a, kWeidemanN);
        for (int i = 0; i < kWeidemanN; ++i) coef.a[i] = (float)a[i];
        for (int i = 0; i < kDawsonNodes; ++i) dawson_coefficients(i / 8.0, coef.dawson + i * kDawsonTerms);
    });
    return coef;
}

cudaError_t launch_voigt(cudaStream_t s, long long n, const float* a, const float* x, float* h)
{
    if (n == 0) return cudaSuccess;
    long long b = (n + 255) / 256;
    if (b > 152LL * 16) b = 152LL * 16;  // two loads of the chip: every CTA fills the table
    k_voigt<<<(unsigned)b, 256, 0, s>>>(voigt_coefficients(), n, a, x, h);
    return cudaGetLastError();
}

}  // namespace dex
