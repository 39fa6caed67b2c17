// qed_tables.cu -- FP64 construction of the rate and inverse-CDF tables of Sec. 5.1 (W_up, W_down,
// IntF^-1_up/down) and Sec. 5.2 (W_+, W_-, IntG^-1_+/-), from the Bessel forms of App. A.
//
// Every stored number is an exact (to FP64 rounding) value of a defined integral or of the root of a
// monotone equation; the quadrature is only the means:
//   NLC, variable t with u' = t^3 (removes the lambda^{-2/3} infrared behaviour noted in Sec. 4.2):
//       density in t  = w_s(lambda) d lambda/dt,  lambda = 3 chi u'/(2 + 3 chi u'),
//       d lambda/du' = 6 chi / (2 + 3 chi u')^2,  w_s = -IntK13 + kappa K23 + s lambda K13 at u'.
//   NBW, spectrum folded about lambda = 1/2 (it is symmetric), variable t with u~' = 8/(3 chi) + t^2:
//       density in t of one half = w0_s(u~') * 4 / (3 chi u~'^{3/2}), w0_s = IntK13 + rho K23 - s K23,
//       rho = 3 chi u~'/2 - 2; stored scaled by e^{8/(3 chi)}.
// Each row integrates panels of width 1/16 in t with 12-point Gauss-Legendre, sums them into the
// CDF at the panel edges, and inverts the CDF at each r_m by Newton's method inside the bracketing
// panel: NLC on partial integrals by 12-point Gauss-Legendre, NBW on the density's Legendre series
// there (from the panel's 12 nodes).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "qed_bessel.cuh"
#include "qed_fp64.cuh"
#include "qed_internal.h"

namespace qed {

constexpr int kGL = 12;
constexpr double kPanel = 1.0 / 16.0;
__constant__ double c_gl_x[kGL];
__constant__ double c_gl_w[kGL];
__constant__ double c_legendre[kGL][kGL];  // [k][i] = (2k + 1)/2 w_i P_k(x_i): values at the nodes -> coefficients

// Gauss-Legendre nodes and weights on [-1, 1] by Newton's method on the Legendre recurrence.
static void gauss_legendre(int n, double* x, double* w) {
    for (int i = 0; i < n; ++i) {
        double z = std::cos(kPi * (i + 0.75) / (n + 0.5)), dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = 0.0;
            for (int j = 1; j <= n; ++j) {
                const double p2 = p1;
                p1 = p0;
                p0 = ((2.0 * j - 1.0) * z * p1 - (j - 1.0) * p2) / j;
            }
            dp = n * (z * p0 - p1) / (z * z - 1.0);
            const double dz = p0 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

__global__ void bessel_table_kernel(double* tab64, float* tab32) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kBesN) return;
    const double x = exp(log(kBesLo) + kBesH * j);
    double o[3];
    bessel_trapezoid(x, o);
    for (int f = 0; f < 3; ++f) {
        tab64[f * kBesN + j] = o[f];
        tab32[f * kBesN + j] = (float)o[f];
    }
}

// The Bessel polynomials of the step kernels (bessel_poly): one warp per interval evaluates the functions at the
// interval's 9 Chebyshev nodes, the lanes sharing the terms of the trapezoid sums (below 1e-4 the ascending series),
// and turns the values into coefficients with the nodes' inverse Vandermonde matrix.
__constant__ double c_vander[kBpDeg + 1][kBpDeg + 1];  // [power][node]
__constant__ double c_cheb[kBpDeg + 1];

__global__ void __launch_bounds__(128) bessel_poly_kernel(double* tab) {
    __shared__ double val[4][3][kBpDeg + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * 4 + warp;
    if (i >= kBpN) return;
    const double centre = ldexp(1.0 + (i % kBpSub + 0.5) / kBpSub, kBpLoExp + i / kBpSub);
    const double half = ldexp(0.5 / kBpSub, kBpLoExp + i / kBpSub);
    for (int n = 0; n <= kBpDeg; ++n) {
        const double x = fma(half, c_cheb[n], centre);
        double o[3] = {0.0, 0.0, 0.0};
        if (x < kBesLo) {
            bessel_series<double>(x, o);
        } else {
            double T = acosh(1.0 + 46.0 / x);
            T = acosh(1.0 + (46.0 + (2.0 / 3.0) * T) / x);
            const double h = fmin(0.2, 0.6 * rsqrt(x));
            const int steps = (int)ceil(T / h);
            for (int m = 1 + lane; m <= steps; m += 32) {
                const double t = m * h, sh = sinh(0.5 * t), e = exp(-x * (2.0 * sh * sh)), c3 = cosh(t / 3.0);
                o[0] += e * c3;
                o[1] += e * (2.0 * c3 * c3 - 1.0);
                o[2] += e * c3 / cosh(t);
            }
            for (int f = 0; f < 3; ++f) {
                for (int s = 16; s > 0; s >>= 1) o[f] += __shfl_xor_sync(0xffffffffu, o[f], s);
                o[f] = (0.5 + o[f]) * h;
            }
        }
        if (lane < 3) val[warp][lane][n] = lane == 0 ? o[0] : (lane == 1 ? o[1] : o[2]);
    }
    __syncwarp();
    if (lane < kBpRow) {
        const int f = lane / (kBpDeg + 1), k = lane % (kBpDeg + 1);
        double v = 0.0;
        for (int n = 0; n <= kBpDeg; ++n) v += c_vander[k][n] * val[warp][f][n];
        tab[(size_t)i * kBpRow + lane] = v;
    }
}

// NLC rows.  An entry is the value at which Newton's method on the 12-point quadrature, kept inside its bracket,
// stops (a bracket or a step of one part in 1e15).  The learned sampler is trained on differences of two of these
// entries down to 1e-7, and a network follows their last bits: so that networks stay the same from build to build the
// rows keep every bit of that definition, and only the work's distribution is free.  A choice that costs 29 ms (every
// row on the panels' series, as the NBW rows are: 2.2 ms a build, entries within an ulp of these).
__device__ __forceinline__ double nlc_density(const double* __restrict__ bes, double chi, double sigma, double t) {
    double b[3];
    const double up = t * t * t;
    const double den = 2.0 + 3.0 * chi * up;
    const double lam = 3.0 * chi * up / den, one_m = 2.0 / den;
    bessel64(bes, up, b);
    const double kappa = 1.0 / one_m + one_m;
    const double w = exp(-up) * (-b[2] + kappa * b[1] + sigma * lam * b[0]);
    return w * 6.0 * chi / (den * den) * 3.0 * t * t;
}

__device__ __forceinline__ double nlc_integral(const double* bes, double chi, double sigma, double a, double b) {
    const double m = 0.5 * (a + b), r = 0.5 * (b - a);
    double s = 0.0;
#pragma unroll 4
    for (int i = 0; i < kGL; ++i) s += c_gl_w[i] * nlc_density(bes, chi, sigma, m + r * c_gl_x[i]);
    return s * r;
}

constexpr int kNlcThreads = 64, kNlcMaxThreads = 128;
constexpr int kNlcPanels = 70;  // cbrt(80) * 16 = 68.9

// One block per (sign, chi row).  FP64-bound, 13 densities an iteration, and an entry takes 5 to 60 iterations (a
// root approached from the left, where the density falls, is bracketed by bisection): a lane that has finished an
// entry takes the row's next one, so no lane waits for the longest of its warp (256 x 256 entries a sign: 36.5 ms
// with one entry a thread, 29.7 ms so).
__global__ void __launch_bounds__(kNlcMaxThreads) nlc_rows_kernel(const double* __restrict__ bes, qed_table_desc d,
                                                                  double* rates, double* icdf) {
    __shared__ double cum[kNlcPanels + 1];
    __shared__ int next;
    const int n_chi = d.n_chi;
    const int s = blockIdx.x / n_chi, i = blockIdx.x % n_chi;
    const double sigma = s == 0 ? 1.0 : -1.0;
    const double dl = (log(d.chi_max) - log(d.chi_min)) / (n_chi - 1);
    const double chi = exp(log(d.chi_min) + i * dl);
    const double tend = cbrt(80.0);
    const int np = (int)ceil(tend / kPanel);
    for (int p = threadIdx.x; p < np; p += blockDim.x)
        cum[p + 1] = nlc_integral(bes, chi, sigma, p * kPanel, fmin(tend, (p + 1) * kPanel));
    __syncthreads();
    if (threadIdx.x == 0) {
        next = blockDim.x;
        cum[0] = 0.0;
        for (int p = 0; p < np; ++p) cum[p + 1] += cum[p];
        rates[s * n_chi + i] = log(cum[np]);
    }
    __syncthreads();
    const double total = cum[np];
    const double dy = (d.y_hi - d.y_lo) / (d.n_r - 1);
    double* out = icdf + ((size_t)s * n_chi + i) * d.n_r;
    double a = 0.0, target = 0.0, tl = 0.0, th = 0.0, t = 0.0;
    int it = 0, p = 0;
    for (int m = threadIdx.x; m < d.n_r;) {
        if (it == 0) {  // a new entry
            const double r = 1.0 / (1.0 + exp(-(d.y_lo + m * dy)));
            target = r * total;
            // panel with cum[p] <= target < cum[p+1]
            int lo = 0, hi = np - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (cum[mid] <= target) lo = mid; else hi = mid - 1;
            }
            a = lo * kPanel;
            const double b = fmin(tend, (lo + 1) * kPanel);
            p = lo;
            tl = a;
            th = b;
            t = a + (b - a) * (target - cum[p]) / (cum[p + 1] - cum[p]);
        }
        const double F = cum[p] + nlc_integral(bes, chi, sigma, a, t) - target;
        if (F > 0.0) th = t; else tl = t;
        const double dF = nlc_density(bes, chi, sigma, t);
        double tn = t - F / dF;
        if (!(tn > tl && tn < th)) tn = 0.5 * (tl + th);
        const bool done = fabs(tn - t) <= 1e-15 * fmax(t, 1e-300) || th - tl <= 1e-15 * th;
        t = tn;
        if (done || ++it == 100) {
            out[m] = 3.0 * log(t);
            m = atomicAdd(&next, 1);
            it = 0;
        }
    }
}

// NBW rows.  The densities in t at both signs sigma = +1, -1 (they share the Bessel functions and all but one
// product)
__device__ __forceinline__ void nbw_density(const double* __restrict__ besp, double chi, double t, double& dp, double& dm) {
    double b[3];
    const double ut = 8.0 / (3.0 * chi) + t * t;
    bessel_poly(besp, ut, b);
    const double rho = 1.5 * chi * ut - 2.0;
    const double f = exp(-t * t) * 4.0 / (3.0 * chi * ut * sqrt(ut));
    const double w = b[2] + rho * b[1];
    dp = f * (w - b[1]);
    dm = f * (w + b[1]);
}

constexpr int kNbwPanels = 144;  // sqrt(80) * 16 = 143.1

// On a panel [a, a + d] with t = a + d s, x = 2 s - 1 and the density's Legendre coefficients c:
//   dH/ds = d sum_k c_k P_k(x),   H(s) = int_a^t = d s [c_0 + (x - 1) sum_{k>=1} c_k P_k'(x) / (k (k + 1))]
// (int_{-1}^x P_k = (x^2 - 1) P_k'(x) / (k (k + 1))): the factor s in front keeps the relative precision of H
// down to s = 0, where the smallest r_m of a grid lie.
__device__ __forceinline__ void panel_cdf(const double* c, double d, double s, double& H, double& h) {
    const double x = 2.0 * s - 1.0;
    double p0 = 1.0, p1 = x, q0 = 0.0, q1 = 1.0;  // P_k and P_k'
    double f = fma(c[1], p1, c[0]), g = 0.5 * c[1];
#pragma unroll
    for (int k = 2; k < kGL; ++k) {
        const double p = ((2.0 * k - 1.0) / k) * x * p1 - ((k - 1.0) / k) * p0;
        const double q = fma(2.0 * k - 1.0, p1, q0);
        f = fma(c[k], p, f);
        g = fma(c[k] * (1.0 / (k * (k + 1.0))), q, g);
        p0 = p1;
        p1 = p;
        q0 = q1;
        q1 = q;
    }
    h = d * f;
    H = d * s * fma(x - 1.0, g, c[0]);
}

// One block per chi row, both signs.  FP64-bound: the density is evaluated at the panels' nodes, and again only
// where the series has not converged; a Newton step on the series is ~100 fused multiply-adds.  A quadrature and a
// density per step, with a stopping rule of one rounding unit that sent most entries through a bisection, took
// 27 ms for 256 x 256 entries a sign; this kernel takes 0.69 ms (83 % of the FP64 pipe's cycles).
__global__ void __launch_bounds__(256) nbw_rows_kernel(const double* __restrict__ besp, qed_table_desc d, double* rates,
                                                       double* icdf) {
    __shared__ double coef[2][kNbwPanels][kGL];  // density at the nodes, then its Legendre coefficients
    __shared__ double cum[2][kNbwPanels + 1];
    const int n_chi = d.n_chi;
    const int i = blockIdx.x;
    const double dl = (log(d.chi_max) - log(d.chi_min)) / (n_chi - 1);
    const double chi = exp(log(d.chi_min) + i * dl);
    const double tend = sqrt(80.0);
    const int np = (int)ceil(tend / kPanel);
    for (int e = threadIdx.x; e < np * kGL; e += blockDim.x) {
        const int p = e / kGL, k = e % kGL;
        const double a = p * kPanel, b = fmin(tend, (p + 1) * kPanel);
        nbw_density(besp, chi, 0.5 * (a + b) + 0.5 * (b - a) * c_gl_x[k], coef[0][p][k], coef[1][p][k]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * np; e += blockDim.x) {
        const int s = e / np, p = e % np;
        double f[kGL], sum = 0.0;
        for (int k = 0; k < kGL; ++k) {
            f[k] = coef[s][p][k];
            sum += c_gl_w[k] * f[k];
        }
        cum[s][p + 1] = sum * 0.5 * (fmin(tend, (p + 1) * kPanel) - p * kPanel);
        for (int k = 0; k < kGL; ++k) {
            double v = 0.0;
            for (int q = 0; q < kGL; ++q) v += c_legendre[k][q] * f[q];
            coef[s][p][k] = v;
        }
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && threadIdx.x < 64) {  // one warp per sign
        const int s = threadIdx.x >> 5;
        double c = 0.0;
        cum[s][0] = 0.0;
        for (int p = 1; p <= np; ++p) {
            c += cum[s][p];
            cum[s][p] = c;
        }
        rates[2 * n_chi + s * n_chi + i] = log(2.0 * c);
    }
    __syncthreads();
    const double dy = (d.y_hi - d.y_lo) / (d.n_r - 1);
    for (int e = threadIdx.x; e < 2 * d.n_r; e += blockDim.x) {
        const int s = e / d.n_r, m = e % d.n_r;
        const double r = 1.0 / (1.0 + exp(-(d.y_lo + m * dy)));
        const double target = r * cum[s][np];
        // panel with cum[p] <= target < cum[p+1]
        int lo = 0, hi = np - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cum[s][mid] <= target) lo = mid; else hi = mid - 1;
        }
        const double a = lo * kPanel, w = fmin(tend, (lo + 1) * kPanel) - a;
        // The entry is the largest t whose CDF, rounded to FP64, does not exceed the target: half a rounding unit
        // of the target above target - cum (near r = 1, where 1 - r is ~1e-9, that is what the entry hangs on).
        const double ulp = __longlong_as_double(__double_as_longlong(target) + 1ll) - target;
        const double T = (target - cum[s][lo]) + 0.5 * ulp, whole = cum[s][lo + 1] - cum[s][lo];
        double u = whole > 0.0 ? fmin(T / whole, 1.0) : 0.5, ul = 0.0, uh = 1.0;
        if (!(target > 0.0)) u = 0x1.0p-100;  // r below the FP64 range: a finite entry
        else
            for (int it = 0; it < 60; ++it) {
                double H, h;
                panel_cdf(coef[s][lo], w, u, H, h);
                if (H > T) uh = u; else ul = u;
                double un = u - (H - T) / h;
                // a step below 1e-9 of u leaves an error below 1e-17 of it (the convergence is quadratic)
                const bool found = fabs(un - u) <= 1e-9 * u;
                if (!(un >= ul && un <= uh) && !found) un = 0.5 * (ul + uh);
                u = un;
                if (found) break;
            }
        double t = a + w * u;
        // where the series has not converged within its 12 terms (the lowest panels of rows with large chi, whose
        // spectrum varies over t ~ chi^{-1/2}) the root is finished on the quadrature itself, one step from the
        // series' root; where it is no series at all (chi above ~1e5) from the panel's chord, inside a bracket
        const double* c = coef[s][lo];
        const double rest = fabs(c[kGL - 1]) + fabs(c[kGL - 2]);
        if (rest > 2e-14 * fabs(c[0]) && target > 0.0) {
            const bool far = rest > 1e-2 * fabs(c[0]);
            if (far) t = a + w * fmin(T / whole, 1.0);
            double tl = a, th = a + w;
            for (int it = 0; it < 100 && t > a; ++it) {
                double dens[2], sum = 0.0;
                for (int k = 0; k < kGL; ++k) {
                    nbw_density(besp, chi, 0.5 * (a + t) + 0.5 * (t - a) * c_gl_x[k], dens[0], dens[1]);
                    sum += c_gl_w[k] * (s ? dens[1] : dens[0]);
                }
                const double F = sum * 0.5 * (t - a) - T;
                nbw_density(besp, chi, t, dens[0], dens[1]);
                const double tn = t - F / (s ? dens[1] : dens[0]);
                if (fabs(tn - t) <= (far ? 1e-15 : 1e-9) * t && tn >= a && tn <= a + w) {
                    t = tn;
                    break;
                }
                if (F > 0.0) th = t; else tl = t;
                t = tn > tl && tn < th ? tn : 0.5 * (tl + th);
                if (th - tl <= 1e-15 * th) break;
            }
        }
        icdf[((size_t)(2 + s) * n_chi + i) * d.n_r + m] = 2.0 * log(t);
    }
}

__global__ void to_float_kernel(const double* __restrict__ a, float* b, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// a as the unevaluated float sum hi + lo (hi = a rounded to float, lo = the rest rounded to float)
__global__ void split_float_kernel(const double* __restrict__ a, float* hi, float* lo, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float h = (float)a[i];
        hi[i] = h;
        lo[i] = (float)(a[i] - (double)h);
    }
}

// ------------------------------------------------------------------------------------------------
// field-dependent anomalous moment (the one-loop Scorer term of App. A.1; g(chi) of Sec. 8.6.2)
// ------------------------------------------------------------------------------------------------
// Scorer function for z >= 0 from its defining integral pi Gi(z) = Im int_0^inf exp(i(z t + t^3/3)) dt,
// taken along the ray t = e^{i pi/6} s (the integrand is analytic and bounded between the two rays):
//   pi Gi(z) = int_0^inf exp(-s^3/3 - z s/2) sin(sqrt(3) z s/2 + pi/6) ds,
// a decaying integrand with at most ~13 oscillations before the exponential falls below e^-46:
// 40 panels of 12-point Gauss-Legendre on [0, min(5.2, 92/z)], the points shared out over a warp.
__device__ double scorer_gi_warp(double z) {
    const double S = fmin(5.2, 92.0 / fmax(z, 1e-300));
    constexpr int np = 40;
    const double h = S / np, w = 0.86602540378443864676 * z, r = 0.5 * h;
    double acc = 0.0;
    for (int e = threadIdx.x & 31; e < np * kGL; e += 32) {
        const double t = (e / kGL + 0.5) * h + r * c_gl_x[e % kGL];
        acc += c_gl_w[e % kGL] * exp(-t * t * t / 3.0 - 0.5 * z * t) * sin(w * t + kPi / 6.0);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc * r / kPi;
}

// a(chi) = (alpha/chi) int_0^inf du u^2/(1+u)^3 Gi(z)/sqrt(z), z = (u/chi)^{2/3}
// (= (alpha/chi) int_0^1 dlambda lambda Gi(z)/sqrt(z) with u = lambda/(1-lambda)).  With u = chi e^v the factor
// g(v) = Gi(e^{2v/3}) e^{-v/3} does not depend on chi, so it is taken once on nodes in v common to every row:
// panels of width at most 1/4 from v0 = -21 - max(ln chi_max, 0) to v1 = 21 + max(-ln chi_min, 0), 12-point
// Gauss-Legendre in each (2796 nodes for chi in [1e-4, 1e3]).  A row that took the integral on nodes of its own
// evaluated g 2100 times, each 480 exponentials and sines: 36 ms for 256 rows against 0.16 ms for the nodes and
// 0.06 ms for the rows (82-86 % of the FP64 pipe's cycles).
struct AmmGrid {
    double v0, h;
    int panels;
};

static AmmGrid amm_grid(const qed_table_desc& d) {
    AmmGrid g;
    g.v0 = -21.0 - std::max(std::log(d.chi_max), 0.0);
    const double v1 = 21.0 + std::max(-std::log(d.chi_min), 0.0);
    g.panels = (int)std::ceil((v1 - g.v0) * 4.0);
    g.h = (v1 - g.v0) / g.panels;
    return g;
}

__device__ __forceinline__ double amm_node(const AmmGrid& G, int k) {
    return G.v0 + (k / kGL + 0.5) * G.h + 0.5 * G.h * c_gl_x[k % kGL];
}

// one warp per node: g(v) with its quadrature weight
__global__ void __launch_bounds__(128) amm_nodes_kernel(AmmGrid G, double* gv) {
    const int k = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (k >= G.panels * kGL) return;
    const double sz = exp(amm_node(G, k) / 3.0);  // sqrt(z)
    const double gi = scorer_gi_warp(sz * sz);
    if ((threadIdx.x & 31) == 0) gv[k] = c_gl_w[k % kGL] * 0.5 * G.h * gi / sz;
}

// One block per chi node; x = ln u runs over [min(ln chi, 0) - 21, max(ln chi, 0) + 21] (the ends add below
// 1e-17 of the result), summed in a fixed tree order.  Stores ln a.
__global__ void __launch_bounds__(256) amm_table_kernel(qed_table_desc d, AmmGrid G, const double* __restrict__ gv,
                                                        double* amm64, float* amm32) {
    __shared__ double part[256];
    const int i = blockIdx.x;
    const double dl = (log(d.chi_max) - log(d.chi_min)) / (d.n_chi - 1);
    const double lnchi = log(d.chi_min) + i * dl, chi = exp(lnchi);
    const double x0 = fmin(lnchi, 0.0) - 21.0, x1 = fmax(lnchi, 0.0) + 21.0;
    double acc = 0.0;
    for (int k = threadIdx.x; k < G.panels * kGL; k += blockDim.x) {
        const double x = amm_node(G, k) + lnchi;
        if (x < x0 || x > x1) continue;
        const double u = exp(x);
        const double q = 1.0 / (1.0 + u);
        acc += gv[k] * u * u * q * q * q;
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double la = log(kAlpha / chi * part[0]);
        amm64[i] = la;
        amm32[i] = (float)la;
    }
}

}  // namespace qed

using namespace qed;

static void free_tables(qed_tables_s* t) {
    if (!t) return;
    cudaFree(t->rate64);  // the start of the tables' one allocation
    t->magic = 0;
    delete t;
}

extern "C" qed_status qed_tables_build(const qed_table_desc* desc, qed_tables_t* out, void* stream) {
    if (!desc || !out) return QED_ERR_ARG;
    const qed_table_desc d = *desc;
    if (d.n_chi < 2 || d.n_r < 4 || d.n_chi > (1 << 16) || d.n_r > (1 << 16) || !(d.chi_min > 0.0) ||
        !(d.chi_max > d.chi_min) || !(d.y_hi > d.y_lo) || !std::isfinite(d.chi_max) || !std::isfinite(d.y_lo) ||
        !std::isfinite(d.y_hi))
        return QED_ERR_ARG;
    *out = nullptr;
    cudaStream_t st = (cudaStream_t)stream;
    qed_tables_s* t = new qed_tables_s();
    std::memset(t, 0, sizeof(*t));
    t->desc = d;
    cudaGetDevice(&t->device);
    const size_t nr = 4 * (size_t)d.n_chi, ni = 4 * (size_t)d.n_chi * d.n_r;
    const AmmGrid G = amm_grid(d);
    // one allocation for every table and the scratch of the a(chi) nodes (nine took 0.1 ms to make and free)
    size_t bytes = 0;
    auto place = [&bytes](size_t n) {
        const size_t at = bytes;
        bytes += (n + 255) & ~size_t(255);
        return at;
    };
    const size_t at[11] = {place(nr * sizeof(double)),        place(ni * sizeof(double)),
                           place(nr * sizeof(float)),         place(ni * sizeof(float)),
                           place(ni * sizeof(float)),         place(3 * kBesN * sizeof(double)),
                           place(3 * kBesN * sizeof(float)),  place(d.n_chi * sizeof(double)),
                           place(d.n_chi * sizeof(float)),    place((size_t)G.panels * kGL * sizeof(double)),
                           place((size_t)kBpN * kBpRow * sizeof(double))};
    unsigned char* mem = nullptr;
    if (cudaMalloc(&mem, bytes) != cudaSuccess) {
        cudaGetLastError();
        free_tables(t);
        return QED_ERR_NOMEM;
    }
    t->rate64 = (double*)(mem + at[0]);
    t->icdf64 = (double*)(mem + at[1]);
    t->rate32 = (float*)(mem + at[2]);
    t->icdf32 = (float*)(mem + at[3]);
    t->icdf32lo = (float*)(mem + at[4]);
    t->bes64 = (double*)(mem + at[5]);
    t->bes32 = (float*)(mem + at[6]);
    t->amm64 = (double*)(mem + at[7]);
    t->amm32 = (float*)(mem + at[8]);
    double* gv = (double*)(mem + at[9]);
    t->besp = (double*)(mem + at[10]);
    double glx[kGL], glw[kGL], leg[kGL][kGL];
    gauss_legendre(kGL, glx, glw);
    for (int i = 0; i < kGL; ++i) {
        double p0 = 1.0, p1 = glx[i];
        for (int k = 0; k < kGL; ++k) {
            leg[k][i] = (k + 0.5) * glw[i] * p0;
            const double p2 = ((2.0 * k + 3.0) * glx[i] * p1 - (k + 1.0) * p0) / (k + 2.0);
            p0 = p1;
            p1 = p2;
        }
    }
    // Chebyshev nodes, and their inverse Vandermonde matrix through the Chebyshev coefficients
    double cheb[kBpDeg + 1], vander[kBpDeg + 1][kBpDeg + 1] = {};
    {
        constexpr int n = kBpDeg + 1;
        double poly[n][n] = {};  // T_j's coefficients
        poly[0][0] = poly[1][1] = 1.0;
        for (int j = 2; j < n; ++j)
            for (int k = 0; k < n; ++k) poly[j][k] = (k > 0 ? 2.0 * poly[j - 1][k - 1] : 0.0) - poly[j - 2][k];
        for (int i = 0; i < n; ++i) cheb[i] = std::cos(kPi * (i + 0.5) / n);
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j)
                for (int k = 0; k < n; ++k)
                    vander[k][i] += (j == 0 ? 1.0 : 2.0) / n * std::cos(kPi * j * (i + 0.5) / n) * poly[j][k];
    }
    if (cudaMemcpyToSymbolAsync(c_cheb, cheb, sizeof(cheb), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_vander, vander, sizeof(vander), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_gl_x, glx, sizeof(glx), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_gl_w, glw, sizeof(glw), 0, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyToSymbolAsync(c_legendre, leg, sizeof(leg), 0, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        free_tables(t);
        return QED_ERR_CUDA;
    }
    bessel_table_kernel<<<(kBesN + 127) / 128, 128, 0, st>>>(t->bes64, t->bes32);
    int sms = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, t->device);
    // Where every row has an SM of its own, four warps keep its four FP64 pipes busy (2 x 4096 entries a sign: 160 ms
    // with two warps, 91 with four, 92 with eight; 76 x 256: 16.2, 13.2, 12.2); rows that share an SM do better with
    // two, whose last entries hold fewer idle warps (77 x 256: 16.7, 20.4, 19.2; 256 x 256: 31.6, 41.1, 37.7).
    const int nlc_threads = 2 * (int64_t)d.n_chi <= sms ? kNlcMaxThreads : kNlcThreads;
    nlc_rows_kernel<<<2 * d.n_chi, nlc_threads, 0, st>>>(t->bes64, d, t->rate64, t->icdf64);
    bessel_poly_kernel<<<(kBpN + 3) / 4, 128, 0, st>>>(t->besp);
    nbw_rows_kernel<<<d.n_chi, 256, 0, st>>>(t->besp, d, t->rate64, t->icdf64);
    to_float_kernel<<<64, 256, 0, st>>>(t->rate64, t->rate32, nr);
    split_float_kernel<<<256, 256, 0, st>>>(t->icdf64, t->icdf32, t->icdf32lo, ni);
    amm_nodes_kernel<<<(G.panels * kGL + 3) / 4, 128, 0, st>>>(G, gv);
    amm_table_kernel<<<d.n_chi, 256, 0, st>>>(d, G, gv, t->amm64, t->amm32);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
        free_tables(t);
        return QED_ERR_CUDA;
    }
    t->magic = kTablesMagic;
    *out = t;
    return QED_OK;
}

extern "C" qed_status qed_tables_export(qed_tables_t t, double* nlc_rate, double* nbw_rate, double* nlc_icdf,
                                        double* nbw_icdf) {
    if (!valid_tables(t)) return QED_ERR_STATE;
    const size_t nc = t->desc.n_chi, ni = 2 * nc * t->desc.n_r;
    cudaError_t e = cudaSuccess;
    if (nlc_rate && e == cudaSuccess) e = cudaMemcpy(nlc_rate, t->rate64, 2 * nc * sizeof(double), cudaMemcpyDeviceToHost);
    if (nbw_rate && e == cudaSuccess) e = cudaMemcpy(nbw_rate, t->rate64 + 2 * nc, 2 * nc * sizeof(double), cudaMemcpyDeviceToHost);
    if (nlc_icdf && e == cudaSuccess) e = cudaMemcpy(nlc_icdf, t->icdf64, ni * sizeof(double), cudaMemcpyDeviceToHost);
    if (nbw_icdf && e == cudaSuccess) e = cudaMemcpy(nbw_icdf, t->icdf64 + ni, ni * sizeof(double), cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

extern "C" qed_status qed_tables_export_amm(qed_tables_t t, double* ln_a) {
    if (!valid_tables(t)) return QED_ERR_STATE;
    if (!ln_a) return QED_ERR_ARG;
    return cudaMemcpy(ln_a, t->amm64, t->desc.n_chi * sizeof(double), cudaMemcpyDeviceToHost) == cudaSuccess
               ? QED_OK
               : QED_ERR_CUDA;
}

extern "C" qed_status qed_tables_destroy(qed_tables_t t) {
    if (!valid_tables(t)) return QED_ERR_STATE;
    cudaDeviceSynchronize();
    free_tables(t);
    return QED_OK;
}

// ------------------------------------------------------------------------------------------------
// test entry points: the special functions and lookups exactly as the step kernels evaluate them
// ------------------------------------------------------------------------------------------------
namespace qed {
__global__ void bessel_eval_kernel(const double* bes64, const float* bes32, int prec, const double* x, double* out, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (prec == QED_FP64) {
            double o[3];
            bessel64(bes64, x[i], o);
            for (int f = 0; f < 3; ++f) out[3 * i + f] = o[f];
        } else {
            float o[3];
            bessel32(bes32, (float)x[i], o);
            for (int f = 0; f < 3; ++f) out[3 * i + f] = o[f];
        }
    }
}

template <class R>
__global__ void lookup_kernel(TabP<R> T, const double* chi, const double* r, double* out, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const R c = (R)chi[i];
        const R lc = log_(c);
        R Iu, Id, Jp, Jm;
        nlc_rates(T, c, lc, Iu, Id);
        nbw_rates(T, c, lc, Jp, Jm);
        const R rr = (R)r[i];
        const R y = log_(rr) - log_(R(1) - rr);
        double* o = out + QED_LOOKUP_COLS * i;
        o[0] = Iu;
        o[1] = Id;
        o[2] = Jp;
        o[3] = Jm;
        o[4] = icdf_lookup(T, false, 0, lc, y);
        o[5] = icdf_lookup(T, false, 1, lc, y);
        o[6] = icdf_lookup(T, true, 0, lc, y);
        o[7] = icdf_lookup(T, true, 1, lc, y);
        o[8] = amm_lookup(T, c);
    }
}
}  // namespace qed

extern "C" qed_status qed_bessel_eval(qed_tables_t t, int32_t precision, const double* x, double* out, int64_t n,
                                      void* stream) {
    if (!valid_tables(t)) return QED_ERR_STATE;
    if ((precision != QED_FP64 && precision != QED_FP32) || n < 0 || (n > 0 && (!x || !out))) return QED_ERR_ARG;
    if (n == 0) return QED_OK;
    bessel_eval_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, (cudaStream_t)stream>>>(
        t->bes64, t->bes32, precision, x, out, n);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

extern "C" qed_status qed_tables_lookup(qed_tables_t t, int32_t precision, const double* chi, const double* r,
                                        double* out, int64_t n, void* stream) {
    if (!valid_tables(t)) return QED_ERR_STATE;
    if ((precision != QED_FP64 && precision != QED_FP32) || n < 0 || (n > 0 && (!chi || !r || !out))) return QED_ERR_ARG;
    if (n == 0) return QED_OK;
    const unsigned g = (unsigned)std::min<int64_t>((n + 255) / 256, 4096);
    if (precision == QED_FP64)
        lookup_kernel<double><<<g, 256, 0, (cudaStream_t)stream>>>(tab_params<double>(t), chi, r, out, n);
    else
        lookup_kernel<float><<<g, 256, 0, (cudaStream_t)stream>>>(tab_params<float>(t), chi, r, out, n);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}
