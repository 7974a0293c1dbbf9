// Level populations of a multi-level atom: emissivity/opacity from populations,
// radiative-rate reduction and per-cell statistical equilibrium.
//
//  * k_lte_pops      Boltzmann populations (float64), sum = n_H.
//  * k_atom_eta_chi  Section 2, Eqs. Eta/Chi (complete redistribution) plus a
//                    grey background with Planck source function, float32, per
//                    cell (times the cell size).  One thread per cell, all
//                    wavelengths; the Doppler profile of each line is
//                    renormalised to unit quadrature on the line's samples.
//  * k_rates         Jbar_l = sum_k w_k phi_k J_k per line in float64 (the
//                    profile-weighted mean intensity the radiative rates need).
//  * k_se_solve      rate matrix (radiative + collisional, detailed balance)
//                    and the per-cell statistical-equilibrium solve in float64,
//                    ground row replaced by particle conservation; Gaussian
//                    elimination with partial pivoting.  With rho given, the
//                    downward radiative rate is A rho + B_ul Jbar (the MALI
//                    preconditioned rate, rho = 1 - Psibar, Jbar = Jbar_eff).
//  * k_mali_rates    MALI with same-transition preconditioning and the
//                    diagonal operator of the long-characteristics solve
//                    (Section 4.1, after Rybicki & Hummer 1992): per line and
//                    cell, from the previous populations and their J,
//                      rho      = 1 - Psibar
//                               = sum_k w_k phi_k (E*_k chi_line,k + chi_c,k) / chi_k,
//                      Jbar_eff = sum_k w_k phi_k (J_k - (1 - E*_k) eta_line,k / chi_k)
//                               = sum_k w_k phi_k (Jext_k + (1 - E*_k) eta_c,k / chi_k),
//                    E*_k = 1 - Lambda*_k = sum_d w_d e^{-chi_k l_d}, l_d the
//                    path from the cell centre to its boundary along direction d,
//                    Jext the formal solution with the probe's own-cell emission
//                    left out (J = Jext + (1 - E*) (eta_line + eta_c) / chi).
//                    Both forms avoid a cancellation: 1 - Psibar is not 1 minus a
//                    sum near 1 (the profile has unit quadrature), and Jbar_eff is
//                    not J minus the own-cell term, which in a cell thick at every
//                    sampled frequency is J to float32 precision (that difference
//                    stalled the iteration near 1e-2 in float32).
//  * k_max_rel_change  max over non-empty cells and levels of |new - old| / new.
#include "dex_internal.h"

#include <cmath>

namespace dex {

namespace {

constexpr double kH = 6.62607015e-27;
constexpr double kC = 2.99792458e10;
constexpr double kKB = 1.380649e-16;
constexpr double kAMU = 1.66053906660e-24;
constexpr double kColl = 8.629e-6;
constexpr double kPi = 3.14159265358979323846;
constexpr double kSqrtSteps = 19.217958540583197;  // sqrt(256 / ln 2)

// The kernels of this file are bound by the FP64 pipe (two fused multiply-adds per
// SM and clock), and nearly all of their arithmetic is exponentials.
//
// 2^(y / 256), table-driven (Tang 1989): y = 256 m + j + f with |f| <= 1/2, the
// result 2^m 2^(j/256) (1 + f w(f)), w the series of (2^(f/256) - 1) / f to f^3
// (remainder below 4e-17): 8 FP64 operations and one shared-memory load, within
// about an ulp of the value at y.  Callers form y directly, so the argument needs no
// two-part reduction.  |y| >= 256000 and NaN go to the library's function.
__device__ __forceinline__ double exp2_steps(const double* table, double y)
{
    if ((__double2hiint(y) & 0x7fffffff) >= 0x410f4000) return exp2(y * 0.00390625);
    constexpr double kShift = 6755399441055744.0;  // 1.5 2^52: rounds to an integer
    const double t = y + kShift;
    const int n = __double2loint(t);
    const double f = y - (t - kShift);
    double w = fma(2.239395190875157e-12, f, 3.3083026805413713e-09);
    w = fma(w, f, 3.6655655969101062e-06);
    w = fma(w, f, 0.0027076061740622863);
    const double T = table[n & 255], e = fma(T, f * w, T);
    return __hiloint2double(__double2hiint(e) + ((n >> 8) << 20), __double2loint(e));
}

__device__ __forceinline__ const double* stage_exp(const AtomParams& P)
{
    __shared__ double s_exp[256];
    for (int j = threadIdx.x; j < 256; j += blockDim.x) s_exp[j] = P.exp_table[j];
    __syncthreads();
    return s_exp;
}

// Planck function at sample k: 2 h nu^3 / c^2 / (e^{h nu / k T} - 1).  Below 0.35 the
// difference loses bits and the library's expm1 takes over; above 693 the value is
// below 1e-300 of its prefactor.  The quotient by Newton's iteration on the
// reciprocal, from the 20-bit approximation of the special-function units.
// FINE, for results that stay in double: the rounding of h nu / k T, which the exponential
// multiplies by itself, is carried to first order, and expm1 serves up to 1.04.  Without,
// the error is up to 1.5 times that of plain double arithmetic (mean 10.8 against 7.3
// units of 2^-53 for arguments of 10 to 30), with it at most half (float32 results see
// neither).
template <bool FINE>
__device__ __forceinline__ double planck(const AtomParams& P, const double* table, int k, double T, double inv_T)
{
    const double y = P.by[k] * inv_T;
    const int hi = __double2hiint(y);
    if (hi >= 0x410f4000) return 0.0;
    if (hi < (FINE ? 0x40780000 : 0x40602000)) return P.bc[k] / expm1(P.bx[k] * inv_T);  // y < 384 or 129
    double e = exp2_steps(table, y);
    if constexpr (FINE) {
        const double lo = (fma(-y, T, P.by[k]) + P.by_lo[k]) * inv_T;
        e = fma(e, lo * 0.0027076061740622863, e);  // ln2 / 256
    }
    const double d = e - 1.0;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    return P.bc[k] * r;
}

// sqrt(256 / ln2) / Doppler width (Hz) of line li at temperature T
__device__ __forceinline__ double inv_doppler(const AtomParams& P, int li, double T)
{
    return kSqrtSteps / (P.nu0[li] / kC * sqrt(2.0 * kKB * T / (P.atom.mass_amu * kAMU)));
}

// Gaussian e^{-((nu - nu0) / width)^2} of sample k; the 1 / (sqrt(pi) width) in front
// cancels in the profile's normalisation on the line's samples.
__device__ __forceinline__ double gauss(const AtomParams& P, const double* table, int k, double inv)
{
    const double u = P.off[k] * inv;
    return exp2_steps(table, -u * u);
}

// Values of a line's samples kept between two passes, per thread: the first n_keep
// in shared memory, the rest evaluated again.
constexpr int kMaxKeep = 45;
constexpr int kAtomThreads = 128;

struct LineValues {
    double* s;
    int n_keep;
    __device__ __forceinline__ void put(int q, double v) const
    {
        if (q < n_keep) s[q * kAtomThreads + threadIdx.x] = v;
    }
    __device__ __forceinline__ double get(const AtomParams& P, const double* table, int q, int k, double inv) const
    {
        return q < n_keep ? s[q * kAtomThreads + threadIdx.x] : gauss(P, table, k, inv);
    }
};

// 1 / sum_k w_k e_k of line li (0 if degenerate), the values kept
__device__ __forceinline__ double line_norm(const AtomParams& P, const double* table, int li, double inv,
                                            const LineValues& V)
{
    double s = 0.0;
    for (int q = P.first[li]; q < P.first[li + 1]; ++q) {
        const int k = P.order[q];
        const double e = gauss(P, table, k, inv);
        V.put(q - P.first[li], e);
        s = fma(P.wq[k], e, s);
    }
    return s > 0.0 ? 1.0 / s : 0.0;
}

__global__ void k_lte_pops(const AtomParams P, long long n_cells, const float* __restrict__ T_,
                           const float* __restrict__ nh_, double* __restrict__ pops)
{
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        const double T = T_[c], nh = nh_[c];
        double w[DEX_MAX_LEVELS], s = 0.0;
        for (int i = 0; i < P.atom.n_level; ++i) {
            w[i] = T > 0.0 ? P.atom.g[i] * exp(-P.atom.energy_erg[i] / (kKB * T)) : 0.0;
            s += w[i];
        }
        for (int i = 0; i < P.atom.n_level; ++i) pops[(long long)i * n_cells + c] = s > 0.0 ? w[i] / s * nh : 0.0;
    }
}

// Each line's exponentials are evaluated once, for the norm, and kept for the second
// pass.  With k_rates 512^2 cells, 96 samples: 5.8 -> 1.7 ms.
__global__ void __launch_bounds__(kAtomThreads) k_atom_eta_chi(const AtomParams P, int n_keep, long long n_cells,
                                                               const float* __restrict__ T_,
                                                               const float* __restrict__ ne_,
                                                               const double* __restrict__ pops,
                                                               float* __restrict__ eta, float* __restrict__ chi)
{
    extern __shared__ double s_val[];
    const double* table = stage_exp(P);
    const LineValues V{s_val, n_keep};
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        const double T = T_[c], ne = ne_[c];
        if (!(T > 0.0)) {
            for (int k = 0; k < P.n_lambda; ++k) {
                eta[(long long)k * n_cells + c] = 0.0f;
                chi[(long long)k * n_cells + c] = 0.0f;
            }
            continue;
        }
        const double chi_c = P.atom.background_sigma * ne * P.atom.cell_cm, inv_T = 1.0 / T;
        for (int li = 0; li < P.atom.n_line; ++li) {
            const double inv = inv_doppler(P, li, T);
            const double f = kH / (4.0 * kPi) * P.atom.cell_cm * line_norm(P, table, li, inv, V);
            const double nlo = pops[(long long)P.atom.line_lower[li] * n_cells + c];
            const double nup = pops[(long long)P.atom.line_upper[li] * n_cells + c];
            const double fe = f * nup * P.atom.line_A[li], fx = f * (nlo * P.b_lu[li] - nup * P.b_ul[li]);
            for (int q = P.first[li]; q < P.first[li + 1]; ++q) {
                const int k = P.order[q];
                const double g = V.get(P, table, q - P.first[li], k, inv) * P.nu[k];
                eta[(long long)k * n_cells + c] = (float)fma(g, fe, chi_c * planck<false>(P, table, k, T, inv_T));
                chi[(long long)k * n_cells + c] = (float)fma(g, fx, chi_c);
            }
        }
        for (int q = P.first[P.atom.n_line]; q < P.n_lambda; ++q) {
            const int k = P.order[q];
            eta[(long long)k * n_cells + c] = (float)(chi_c * planck<false>(P, table, k, T, inv_T));
            chi[(long long)k * n_cells + c] = (float)chi_c;
        }
    }
}

// Jbar = sum_k w_k e_k J_k / sum_k w_k e_k: one pass over a line's samples
__global__ void __launch_bounds__(kAtomThreads) k_rates(const AtomParams P, long long n_cells,
                                                        const float* __restrict__ T_, const float* __restrict__ J,
                                                        double* __restrict__ jbar)
{
    const double* table = stage_exp(P);
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        const double T = T_[c];
        for (int li = 0; li < P.atom.n_line; ++li) {
            double jb = 0.0;
            if (T > 0.0) {
                const double inv = inv_doppler(P, li, T);
                double s = 0.0, sj = 0.0;
                for (int q = P.first[li]; q < P.first[li + 1]; ++q) {
                    const int k = P.order[q];
                    const double we = P.wq[k] * gauss(P, table, k, inv);
                    s += we;
                    sj = fma(we, (double)J[(long long)k * n_cells + c], sj);
                }
                jb = s > 0.0 ? sj / s : 0.0;
            }
            jbar[(long long)li * n_cells + c] = jb;
        }
    }
}

__global__ void __launch_bounds__(kAtomThreads) k_mali_rates(const AtomParams P, const OwnCellOperator O, int n_keep,
                                                             long long n_cells, const float* __restrict__ T_,
                                                             const float* __restrict__ ne_,
                                                             const double* __restrict__ pops,
                                                             const float* __restrict__ Jext, double* __restrict__ rho,
                                                             double* __restrict__ jeff)
{
    extern __shared__ double s_val[];
    const double* table = stage_exp(P);
    const LineValues V{s_val, n_keep};
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        const double T = T_[c], ne = ne_[c];
        const double chi_c = P.atom.background_sigma * ne * P.atom.cell_cm;
        for (int li = 0; li < P.atom.n_line; ++li) {
            double r = 0.0, je = 0.0;
            if (T > 0.0) {
                const double inv = inv_doppler(P, li, T), inv_T = 1.0 / T;
                const double norm = line_norm(P, table, li, inv, V);
                const double nlo = pops[(long long)P.atom.line_lower[li] * n_cells + c];
                const double nup = pops[(long long)P.atom.line_upper[li] * n_cells + c];
                const double fx = kH / (4.0 * kPi) * P.atom.cell_cm * (nlo * P.b_lu[li] - nup * P.b_ul[li]);
                for (int q = P.first[li]; q < P.first[li + 1]; ++q) {
                    const int k = P.order[q];
                    const double phi = V.get(P, table, q - P.first[li], k, inv) * norm;
                    const double chi_l = P.nu[k] * phi * fx;
                    const double chi = chi_l + chi_c;
                    if (!(chi > 0.0)) continue;
                    // escape from the own cell, summed over the direction groups
                    const float xf = (float)chi;
                    float es = 0.0f;
                    for (int g = 0; g < O.n; ++g) es = fmaf(O.w[g], expf(-xf * O.ell[g]), es);
                    const double e = (double)es;
                    const double wp = P.wq[k] * phi, inv_chi = 1.0 / chi;
                    const double eta_c = chi_c * planck<true>(P, table, k, T, inv_T);
                    r += wp * ((e * chi_l + chi_c) * inv_chi);
                    je += wp * ((double)Jext[(long long)k * n_cells + c] + (1.0 - e) * (eta_c * inv_chi));
                }
            }
            rho[(long long)li * n_cells + c] = r;
            jeff[(long long)li * n_cells + c] = je;
        }
    }
}

// |new - old| / new maximised over non-empty cells and levels; positive doubles
// order as their bit patterns, so the maximum is an integer atomicMax
__global__ void k_max_rel_change(int n_level, long long n_cells, const float* __restrict__ T_,
                                 const double* __restrict__ old_p, const double* __restrict__ new_p,
                                 unsigned long long* __restrict__ out)
{
    double m = 0.0;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        if (!(T_[c] > 0.0f)) continue;
        for (int i = 0; i < n_level; ++i) {
            const double a = old_p[(long long)i * n_cells + c], b = new_p[(long long)i * n_cells + c];
            const double d = b > 0.0 ? fabs(b - a) / b : (a == b ? 0.0 : __longlong_as_double(0x7ff0000000000000LL));
            m = d > m || d != d ? d : m;   // a NaN propagates
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double v = __shfl_down_sync(0xffffffffu, m, o);
        m = v > m || v != v ? v : m;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

__global__ void k_se_solve(const AtomParams P, long long n_cells, const float* __restrict__ T_,
                           const float* __restrict__ ne_, const float* __restrict__ nh_,
                           const double* __restrict__ jbar, const double* __restrict__ rho,
                           double* __restrict__ pops)
{
    const int nl = P.atom.n_level;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n_cells;
         c += (long long)gridDim.x * blockDim.x) {
        const double T = T_[c], ne = ne_[c], nh = nh_[c];
        if (!(T > 0.0)) {
            for (int i = 0; i < nl; ++i) pops[(long long)i * n_cells + c] = 0.0;
            continue;
        }
        double R[DEX_MAX_LEVELS][DEX_MAX_LEVELS] = {};  // R[i][j]: rate i -> j
        const double sq = sqrt(T);
        for (int i = 0; i < nl; ++i)
            for (int j = i + 1; j < nl; ++j) {
                const double ups = P.atom.upsilon[i][j];
                if (ups <= 0.0) continue;
                const double dE = P.atom.energy_erg[j] - P.atom.energy_erg[i];
                R[i][j] += ne * kColl / (P.atom.g[i] * sq) * ups * exp(-dE / (kKB * T));
                R[j][i] += ne * kColl / (P.atom.g[j] * sq) * ups;
            }
        for (int li = 0; li < P.atom.n_line; ++li) {
            const int lo = P.atom.line_lower[li], up = P.atom.line_upper[li];
            const double jb = jbar[(long long)li * n_cells + c];
            R[lo][up] += P.b_lu[li] * jb;
            R[up][lo] += P.atom.line_A[li] * (rho ? rho[(long long)li * n_cells + c] : 1.0) + P.b_ul[li] * jb;
        }
        // M n = b: row i = inflow - outflow of level i; row 0 = conservation
        double M[DEX_MAX_LEVELS][DEX_MAX_LEVELS + 1];
        for (int i = 0; i < nl; ++i) {
            for (int j = 0; j <= nl; ++j) M[i][j] = 0.0;
            for (int j = 0; j < nl; ++j)
                if (j != i) {
                    M[i][j] += R[j][i];
                    M[i][i] -= R[i][j];
                }
        }
        for (int j = 0; j < nl; ++j) M[0][j] = 1.0;
        M[0][nl] = nh;
        for (int col = 0; col < nl; ++col) {  // elimination with partial pivoting
            int piv = col;
            for (int r = col + 1; r < nl; ++r)
                if (fabs(M[r][col]) > fabs(M[piv][col])) piv = r;
            if (piv != col)
                for (int j = 0; j <= nl; ++j) {
                    const double t = M[col][j];
                    M[col][j] = M[piv][j];
                    M[piv][j] = t;
                }
            const double inv = 1.0 / M[col][col];
            for (int r = col + 1; r < nl; ++r) {
                const double f = M[r][col] * inv;
                for (int j = col; j <= nl; ++j) M[r][j] -= f * M[col][j];
            }
        }
        double n[DEX_MAX_LEVELS];
        for (int i = nl - 1; i >= 0; --i) {
            double s = M[i][nl];
            for (int j = i + 1; j < nl; ++j) s -= M[i][j] * n[j];
            n[i] = s / M[i][i];
        }
        for (int i = 0; i < nl; ++i) pops[(long long)i * n_cells + c] = n[i];
    }
}

unsigned grid_for(long long n, int threads = 256)
{
    long long b = (n + threads - 1) / threads;
    return (unsigned)(b > 152LL * 16 ? 152LL * 16 : (b < 1 ? 1 : b));
}

// samples of the longest line, as many as are kept (with the table 48 KB of shared
// memory)
int kept_values(const AtomParams& P)
{
    int n = 0;
    for (int li = 0; li < P.atom.n_line; ++li) n = max(n, (int)(P.first[li + 1] - P.first[li]));
    return min(n, kMaxKeep);
}

}  // namespace

cudaError_t launch_lte_pops(cudaStream_t s, const AtomParams& P, long long n_cells, const float* T,
                            const float* nh, double* pops)
{
    if (n_cells == 0) return cudaSuccess;
    k_lte_pops<<<grid_for(n_cells), 256, 0, s>>>(P, n_cells, T, nh, pops);
    return cudaGetLastError();
}

cudaError_t launch_atom_eta_chi(cudaStream_t s, const AtomParams& P, long long n_cells, const float* T,
                                const float* ne, const double* pops, float* eta, float* chi)
{
    if (n_cells == 0 || P.n_lambda == 0) return cudaSuccess;
    const int keep = kept_values(P);
    k_atom_eta_chi<<<grid_for(n_cells, kAtomThreads), kAtomThreads, keep * kAtomThreads * sizeof(double), s>>>(
        P, keep, n_cells, T, ne, pops, eta, chi);
    return cudaGetLastError();
}

cudaError_t launch_rates(cudaStream_t s, const AtomParams& P, long long n_cells, const float* T, const float* J,
                         double* jbar)
{
    if (n_cells == 0) return cudaSuccess;
    k_rates<<<grid_for(n_cells, kAtomThreads), kAtomThreads, 0, s>>>(P, n_cells, T, J, jbar);
    return cudaGetLastError();
}

cudaError_t launch_se_solve(cudaStream_t s, const AtomParams& P, long long n_cells, const float* T, const float* ne,
                            const float* nh, const double* jbar, const double* rho, double* pops)
{
    if (n_cells == 0) return cudaSuccess;
    k_se_solve<<<grid_for(n_cells), 128, 0, s>>>(P, n_cells, T, ne, nh, jbar, rho, pops);
    return cudaGetLastError();
}

cudaError_t launch_mali_rates(cudaStream_t s, const AtomParams& P, const OwnCellOperator& O, long long n_cells,
                              const float* T, const float* ne, const double* pops, const float* J, double* rho,
                              double* jeff)
{
    if (n_cells == 0 || P.atom.n_line == 0) return cudaSuccess;
    const int keep = kept_values(P);
    k_mali_rates<<<grid_for(n_cells, kAtomThreads), kAtomThreads, keep * kAtomThreads * sizeof(double), s>>>(
        P, O, keep, n_cells, T, ne, pops, J, rho, jeff);
    return cudaGetLastError();
}

cudaError_t launch_max_rel_change(cudaStream_t s, int n_level, long long n_cells, const float* T, const double* old_p,
                                  const double* new_p, double* out)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
    if (e != cudaSuccess || n_cells == 0) return e;
    k_max_rel_change<<<grid_for(n_cells), 256, 0, s>>>(n_level, n_cells, T, old_p, new_p,
                                                       reinterpret_cast<unsigned long long*>(out));
    return cudaGetLastError();
}

}  // namespace dex
