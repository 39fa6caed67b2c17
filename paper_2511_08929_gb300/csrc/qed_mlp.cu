// qed_mlp.cu -- the learned sampler: a 3-64-64-64-4 SiLU network standing in for the three-dimensional
// inverse CDF in (chi, r, s_beta) that Sec. 5.1 rejects for its memory.
//
// Target (the map the network learns, computed from the FP64 tables): the exact r-quantile ln u' of the
// NLC spectrum for a continuous spin projection s (w is linear in s: the mixture CDF is the rate-weighted
// blend of the two branch CDFs, each the inverse of its interpolated ICDF row) and the photon Stokes
// vector there (App. A.1, s_i = s beta_hat, final spin summed: xi1 = xi2 = 0, xi3 = F3/F0).  The network
// predicts the correction to the rate-weighted blend of the two branch quantiles (and of xi3 there),
// scaled by 100.
//
// Kernels: target generation (FP64); one training kernel (forward, backward and weight gradients of 128-sample
// tiles on the tensor cores: tcgen05.mma with BF16 operands and FP32 accumulators in TMEM) and AdamW; inference
// (layers 2-4 as tcgen05.mma on 128-sample tiles, bias and SiLU between them applied on the way from TMEM back to
// shared memory), and the CDF check with the table fallback.
#include <cstring>

#include <cuda_bf16.h>

#include "qed_device.cuh"
#include "qed_fp64.cuh"
#include "qed_internal.h"

namespace qed {

// ---- parameter layout (FP32, one array): W1[64][3] b1[64] W2[64][64] b2 W3[64][64] b3 W4[4][64] b4[4]
constexpr int kH = 64;
constexpr int kOffW1 = 0, kOffB1 = 192, kOffW2 = 256, kOffB2 = 4352, kOffW3 = 4416, kOffB3 = 8512, kOffW4 = 8576,
              kOffB4 = 8832, kParams = 8836;
static_assert(kParams == QED_MLP_PARAMS, "parameter count");

constexpr double kLnChiLo = -6.907755278982137, kLnChiHi = 4.605170185988092;  // ln 1e-3, ln 1e2
constexpr double kYClamp = 20.0;
constexpr double kOutScale = 100.0;
constexpr uint64_t kMlpStep = 0xFFFFFFFFFFFFFFFEull;  // reserved Philox step of the training inputs

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float dsilu_f(float z) {
    const float s = 1.0f / (1.0f + expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// ---- the map from (chi, r, s) to the target, FP64 tables -------------------------------------------
template <class R>
struct MixPointT {
    R lnchi, y, s, a;  // a = (1 + s) I_up / ((1 + s) I_up + (1 - s) I_down)
    R qu, qd;          // the two branch quantiles at the logit y
};
using MixPoint = MixPointT<double>;

__device__ inline MixPoint mix_point(const TabP<double>& T, double chi, double r, double s) {
    MixPoint m;
    m.lnchi = log(chi);
    m.y = log(r) - log1p(-r);
    m.s = s;
    double Iu, Id;
    nlc_rates(T, chi, m.lnchi, Iu, Id);
    m.a = (1.0 + s) * Iu / ((1.0 + s) * Iu + (1.0 - s) * Id);
    m.qu = icdf_lookup(T, false, 0, m.lnchi, m.y);
    m.qd = icdf_lookup(T, false, 1, m.lnchi, m.y);
    return m;
}

// the same point on the float tables; the logit from r and 1 - r, each rounded to float once, so that
// neither end of (0, 1) loses its precision
__device__ inline MixPointT<float> mix_point32(const TabP<float>& T, double chi, double r, double s) {
    MixPointT<float> m;
    const float c = (float)chi, sf = (float)s;
    m.lnchi = logf(c);
    m.y = logf((float)r) - logf((float)(1.0 - r));
    m.s = sf;
    float Iu, Id;
    nlc_rates(T, c, m.lnchi, Iu, Id);
    m.a = (1.0f + sf) * Iu / ((1.0f + sf) * Iu + (1.0f - sf) * Id);
    m.qu = icdf_lookup(T, false, 0, m.lnchi, m.y);
    m.qd = icdf_lookup(T, false, 1, m.lnchi, m.y);
    return m;
}

// Root of a monotone increasing g on the bracket [a, c] (g(a) < 0 < g(c)) by regula falsi with the
// Illinois weight (the end that stays put has its value halved, so neither end stalls), started at the
// guess x0; a step outside the bracket falls back to its midpoint.  Stops when the bracket is below
// dx or |g| below dg, after at most ITERS evaluations.
template <int ITERS, class R, class G>
__device__ inline R illinois(G g, R a, R ga, R c, R gc, R x0, R dx, R dg) {
    R x = x0 < a ? a : (x0 > c ? c : x0);
    if (!(x > a && x < c)) x = R(0.5) * (a + c);
    int side = 0;
    for (int it = 0; it < ITERS; ++it) {
        const R f = g(x);
        if ((f < R(0) ? -f : f) <= dg) return x;
        if (f < R(0)) {
            a = x;
            ga = f;
            if (side == -1) gc *= R(0.5);
            side = -1;
        } else {
            c = x;
            gc = f;
            if (side == 1) ga *= R(0.5);
            side = 1;
        }
        if (c - a <= dx) break;
        x = (a * gc - c * ga) / (gc - ga);
        if (!(x > a && x < c)) x = R(0.5) * (a + c);
    }
    return R(0.5) * (a + c);
}

// CDF of one spin branch at ln u' = L: the logit y at which the interpolated ICDF row equals L, mapped
// to r.  The search starts at the mixture point's logit yg, whose quantile qg is known: steps of
// (L - qg)/3 (the slope of ln u' in the logit below the grid; it is smaller above), doubled until the
// sign of ICDF(y) - L changes, bracket the root, and the solver finishes inside the bracket.  A step
// that reaches an end of the grid without the change means L lies beyond the tabulated range: above it
// the CDF is 1, below it the linear asymptote is inverted directly.  In FP64 (R = double) the logit to
// 1e-10, so the CDF to 3e-11; on the float tables the logit to 1e-6 and the CDF to ~3e-7 (the float
// entries' own rounding, ~6e-8 of ln u', adds no more than that).
template <int ITERS, class R>
__device__ inline R branch_cdf(const TabP<R>& T, int b, R lnchi, R L, R yg, R qg) {
    constexpr bool F64 = sizeof(R) == 8;
    const R yhi = T.y_lo + R(T.n_r - 1) / T.inv_dy;
    auto g = [&](R yy) { return icdf_lookup(T, false, b, lnchi, yy) - L; };
    const R g0 = qg - L;
    if (g0 == R(0)) return R(1) / (R(1) + exp_(-yg));
    const bool up = g0 < R(0);  // the root lies above yg
    R x = yg, gx = g0;
    R step = (L - qg) / R(3);
    step = step < R(0) ? -step : step;
    if (step < R(F64 ? 1e-9 : 1e-5)) step = R(F64 ? 1e-9 : 1e-5);
    R a = x, ga = gx, c = x, gc = gx;
    bool found = false;
    for (int k = 0; k < 26 && !found; ++k) {
        R xn = up ? x + step : x - step;
        const bool edge = up ? xn >= yhi : xn <= T.y_lo;
        if (edge) xn = up ? yhi : T.y_lo;
        const R gn = g(xn);
        if (up ? gn >= R(0) : gn <= R(0)) {
            a = up ? x : xn;
            ga = up ? gx : gn;
            c = up ? xn : x;
            gc = up ? gn : gx;
            found = true;
        } else if (edge) {
            if (up) return R(1);                                   // L above the row's last entry
            return R(1) / (R(1) + exp_(-(T.y_lo + (-gn) / R(3))));  // below: y_lo + (L - bottom)/3
        } else {
            x = xn;
            gx = gn;
            step *= R(2);
        }
    }
    if (!found) return R(1) / (R(1) + exp_(-x));  // not reached: 26 doublings span the grid
    const R aL = L < R(0) ? -L : L;
    const R x0 = a - ga * (c - a) / (gc - ga);
    const R y = illinois<ITERS>(g, a, ga, c, gc, x0, R(F64 ? 1e-10 : 1e-6), R(F64 ? 1e-13 : 1e-7) * (aL > R(1) ? aL : R(1)));
    return R(1) / (R(1) + exp_(-y));
}

// the mixture's CDF at L: each branch solved from the mixture point's own logit, near which its root
// lies (at most ITERS evaluations each)
template <int ITERS, class R>
__device__ inline R mix_cdf(const TabP<R>& T, const MixPointT<R>& m, R L) {
    return m.a * branch_cdf<ITERS>(T, 0, m.lnchi, L, m.y, m.qu) +
           (R(1) - m.a) * branch_cdf<ITERS>(T, 1, m.lnchi, L, m.y, m.qd);
}

// the blend of the two branch quantiles (the baseline the network corrects)
template <class R>
__device__ inline R mix_baseline(const TabP<R>& T, const MixPointT<R>& m) {
    return m.a * m.qu + (R(1) - m.a) * m.qd;
}

// the exact mixture quantile: the mixture CDF lies between the branch CDFs, so its quantile lies between
// the branch quantiles; the same solver there, from the blend of the two, until the mixture CDF is
// within 2e-11 of r (the inner solves' own accuracy) or the bracket below 1e-12 in ln u'
template <int OUTER, int INNER>
__device__ inline double mix_quantile(const TabP<double>& T, const MixPoint& m, double r) {
    const double qu = m.qu, qd = m.qd;
    const double lo = fmin(qu, qd) - 1e-9, hi = fmax(qu, qd) + 1e-9;
    auto g = [&](double L) { return mix_cdf<INNER>(T, m, L) - r; };
    const double glo = g(lo), ghi = g(hi);
    if (!(glo < 0.0)) return lo;
    if (!(ghi > 0.0)) return hi;
    return illinois<OUTER>(g, lo, glo, hi, ghi, m.a * qu + (1.0 - m.a) * qd, 1e-12, 2e-11);
}

// xi3 = F3 / F0 at u' for s_i = s beta_hat, s_f = 0 (App. A.1)
__device__ inline double xi3_at(const double* __restrict__ bes_tab, double chi, double L, double s) {
    // a network output outside any physical range (or not finite) never reaches the Bessel evaluation
    if (!(L > -200.0 && L < 50.0)) return nan("");
    const double up = exp(L);
    const double lam = 3.0 * chi * up / (2.0 + 3.0 * chi * up), one_m = 1.0 - lam;
    double b[3];
    bessel64(bes_tab, up, b);
    const double u = lam / one_m, kappa = 1.0 / one_m + one_m;
    return (b[1] + u * s * b[0]) / (-b[2] + kappa * b[1] + lam * s * b[0]);
}

// the same from the float Bessel table
__device__ inline float xi3_at32(const float* __restrict__ bes32, float chi, float L, float s) {
    if (!(L > -85.0f && L < 50.0f)) return __int_as_float(0x7FC00000);  // u' outside the float range
    const float up = expf(L);
    const float den = fmaf(3.0f * chi, up, 2.0f), lam = 3.0f * chi * up / den, one_m = 2.0f / den;
    float b[3];
    bessel32(bes32, up, b);
    const float u = lam / one_m, kappa = 1.0f / one_m + one_m;
    return (b[1] + u * s * b[0]) / (-b[2] + kappa * b[1] + lam * s * b[0]);
}

// ---- the sampler's own solves ------------------------------------------------------------------------
// The sampler's check and fallback take their roots on the float tables first and, where FP64 decides, finish them on
// the FP64 tables by Newton's method: a step is two ICDF rows with their slopes, ~45 FP64 instructions a branch, and
// two steps from the float root leave errors below 1e-13.  (The bracketing solvers above, which the training targets
// use, take ~80 ICDF evaluations for a mixture quantile in FP64, 0.65 ms for one warp; this one takes ~0.03 ms.)

// value and slope (in the logit) of branch b's ICDF at the logit y, rows (i, i + 1) blended with f; inside the grid,
// and below it, where the row continues with slope 3
template <class R>
__device__ __forceinline__ void icdf_slope(const TabP<R>& T, int b, int i, R f, R y, R& q, R& dq) {
    const R y0 = T.y_lo * T.inv_dy, tt = fma_(y, T.inv_dy, -y0);
    if (!(tt > R(0))) {
        const R* row = T.nlc_icdf + ((size_t)b * T.n_chi + i) * T.n_r;
        q = fma_(R(3), y - T.y_lo, fma_(f, row[T.n_r] - row[0], row[0]));
        dq = R(3);
        return;
    }
    const int m = min(max((int)tt, 1), T.n_r - 3);
    const R x = fma_(y, T.inv_dy, -y0 - R(m)), xm = x - R(1);
    const R* row = T.nlc_icdf + ((size_t)b * T.n_chi + i) * T.n_r + m;
    R v[2], d[2];
#pragma unroll
    for (int k = 0; k < 2; ++k, row += T.n_r) {
        const R p0 = row[-1], p1 = row[0], p2 = row[1], p3 = row[2];
        const R d1 = p2 - p1, d2 = R(0.5) * ((p0 - p1) + d1), d3 = fma_(R(-3), d1, p3 - p0) * R(1.0 / 6.0);
        const R e = fma_(x + R(1), d3, d2), c = fma_(xm, e, d1);
        v[k] = fma_(x, c, p1);
        d[k] = fma_(x, fma_(xm, d3, e), c);
    }
    q = fma_(f, v[1] - v[0], v[0]);
    dq = fma_(f, d[1] - d[0], d[0]) * T.inv_dy;
}

// Newton's method for the mixture quantile in (L, y_u, y_d): both branch ICDFs at their logits equal L and the blend
// of the logits' CDFs equals r.  True when a step below `dy` was taken with every logit
// below the grid's upper end.
template <class R>
__device__ inline bool mix_newton(const TabP<R>& T, int i, R f, R a, R r, int iters, R dy, R& L, R& yu, R& yd) {
    const R yhi = T.y_lo + R(T.n_r - 1) / T.inv_dy;
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        if (!(yu < yhi && yd < yhi)) return false;
        R qu, du, qd, dd;
        icdf_slope(T, 0, i, f, yu, qu, du);
        icdf_slope(T, 1, i, f, yd, qd, dd);
        if (!(du > R(0) && dd > R(0))) return false;
        const R iu = rcp_(du), id = rcp_(dd);
        const R su = rcp_(R(1) + exp_(-yu)), sd = rcp_(R(1) + exp_(-yd));
        const R wu = a * su * (R(1) - su) * iu, wd = (R(1) - a) * sd * (R(1) - sd) * id;
        const R res = (r - a * su - (R(1) - a) * sd) - fma_(wu, L - qu, wd * (L - qd));
        if (!(wu + wd > R(0))) return false;
        L = L + div_(res, wu + wd);
        const R eu = (L - qu) * iu, ed = (L - qd) * id;
        yu += eu;
        yd += ed;
        if (fabs(eu) < dy && fabs(ed) < dy) return yu < yhi && yd < yhi;
    }
    return false;
}

// the logit at which branch b's ICDF row equals L, from a root y good to the float tables; false if it leaves the
// grid upwards
__device__ inline bool logit_newton64(const TabP<double>& T, int b, int i, double f, double L, double& y) {
    const double yhi = T.y_lo + (T.n_r - 1) / T.inv_dy;
#pragma unroll 1
    for (int it = 0; it < 4; ++it) {
        if (!(y < yhi)) return false;
        double q, dq;
        icdf_slope(T, b, i, f, y, q, dq);
        if (!(dq > 0.0)) return false;
        const double e = (L - q) / dq;
        y += e;
        if (fabs(e) < 1e-7) return y < yhi;
    }
    return false;
}

// branch_cdf on the float tables, returning the logit (infinite above the row's last entry)
__device__ __noinline__ float branch_logit32(const TabP<float>& T, int b, float lnchi, float L, float yg, float qg) {
    const float yhi = T.y_lo + (float)(T.n_r - 1) / T.inv_dy;
    auto g = [&](float yy) { return icdf_lookup(T, false, b, lnchi, yy) - L; };
    const float g0 = qg - L;
    if (g0 == 0.0f) return yg;
    const bool up = g0 < 0.0f;  // the root lies above yg
    float x = yg, gx = g0;
    float step = (L - qg) / 3.0f;
    step = step < 0.0f ? -step : step;
    if (step < 1e-5f) step = 1e-5f;
    float a = x, ga = gx, c = x, gc = gx;
    bool found = false;
#pragma unroll 1
    for (int k = 0; k < 26 && !found; ++k) {
        float xn = up ? x + step : x - step;
        const bool edge = up ? xn >= yhi : xn <= T.y_lo;
        if (edge) xn = up ? yhi : T.y_lo;
        const float gn = g(xn);
        if (up ? gn >= 0.0f : gn <= 0.0f) {
            a = up ? x : xn;
            ga = up ? gx : gn;
            c = up ? xn : x;
            gc = up ? gn : gx;
            found = true;
        } else if (edge) {
            if (up) return __int_as_float(0x7F800000);  // L above the row's last entry
            return T.y_lo + (-gn) / 3.0f;               // below: y_lo + (L - bottom)/3
        } else {
            x = xn;
            gx = gn;
            step *= 2.0f;
        }
    }
    if (!found) return x;  // not reached: 26 doublings span the grid
    const float aL = L < 0.0f ? -L : L;
    return illinois<30>(g, a, ga, c, gc, a - ga * (c - a) / (gc - ga), 1e-6f, 1e-7f * (aL > 1.0f ? aL : 1.0f));
}

// the mixture's CDF at L on the float tables, with the branches' logits
__device__ inline float mix_cdf32(const TabP<float>& T, const MixPointT<float>& m, float L, float& yu, float& yd) {
    yu = branch_logit32(T, 0, m.lnchi, L, m.y, m.qu);
    yd = branch_logit32(T, 1, m.lnchi, L, m.y, m.qd);
    return m.a * (1.0f / (1.0f + exp_(-yu))) + (1.0f - m.a) * (1.0f / (1.0f + exp_(-yd)));
}

// |C(L) - r| on the FP64 tables, from the float tables' logits (the bracketing solver where a logit lies above the
// grid)
__device__ __noinline__ double mix_error64(const TabP<double>& T, const MixPoint& m, double L, double r, float yu32,
                                           float yd32) {
    int i;
    double f, yu = yu32, yd = yd32;
    chi_coord(T, m.lnchi, i, f);
    if (logit_newton64(T, 0, i, f, L, yu) && logit_newton64(T, 1, i, f, L, yd))
        return fabs(m.a / (1.0 + exp(-yu)) + (1.0 - m.a) / (1.0 + exp(-yd)) - r);
    return fabs(mix_cdf<30>(T, m, L) - r);
}

// the mixture quantile: Newton on the float tables from the blend of the branch quantiles, then on the FP64 tables;
// false where that does not converge below the grid's upper end (there the bracketing solver, mix_quantile, finds it)
__device__ __noinline__ bool mix_quantile_fast(const TabP<double>& T, const TabP<float>& T32, const MixPoint& m, double r,
                                               double& L) {
    int i;
    double f;
    chi_coord(T, m.lnchi, i, f);
    L = mix_baseline(T, m);
    double yu = m.y, yd = m.y;
    float L32 = (float)L, yu32 = (float)m.y, yd32 = (float)m.y;
    if (mix_newton<float>(T32, i, (float)f, (float)m.a, (float)r, 12, 1e-3f, L32, yu32, yd32)) {
        L = L32;
        yu = yu32;
        yd = yd32;
    }
    if (!mix_newton<double>(T, i, f, m.a, r, 8, 1e-7, L, yu, yd)) return false;
    // between the branch quantiles, as the bracketing solver: with |s| > 1 the blend has a negative weight and its root
    // lies beyond them (tested on the high word, since every FP64 instruction counts here)
    if ((__double2hiint(m.s) & 0x7FFFFFFF) >= 0x3FF00000)
        L = fmin(fmax(L, fmin(m.qu, m.qd) - 1e-9), fmax(m.qu, m.qd) + 1e-9);
    return true;
}

// xi3 = F3 / F0 at u' = e^L from the Bessel polynomials (see xi3_at)
__device__ inline double xi3_poly(const double* __restrict__ besp, double chi, double L, double s) {
    if (!(L > -200.0 && L < 50.0)) return nan("");
    const double up = exp(L), u = 1.5 * chi * up, iom = 1.0 + u, one_m = 1.0 / iom;
    double b[3];
    bessel_poly(besp, up, b);
    return fma(u * s, b[0], b[1]) / (fma(iom + one_m, b[1], -b[2]) + u * one_m * s * b[0]);
}

__device__ inline void mlp_features(double chi, double r, double s, float x[3]) {
    const double y = fmin(kYClamp, fmax(-kYClamp, log(r) - log1p(-r)));
    x[0] = (float)((log(chi) - 0.5 * (kLnChiLo + kLnChiHi)) / (0.5 * (kLnChiHi - kLnChiLo)));
    x[1] = (float)(y / 10.0);
    x[2] = (float)s;
}

__global__ void mlp_targets_kernel(TabP<double> T, const double* __restrict__ bes_tab, int64_t n, uint64_t seed,
                                   int64_t first, float* __restrict__ X, float* __restrict__ Y, double* __restrict__ raw) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t id = (uint64_t)(first + i);
        const uint4 w0 = draw(id, seed, kMlpStep, 0), w1 = draw(id, seed, kMlpStep, 1);
        const double lnchi = kLnChiLo + uniform52(w0.x, w0.y) * (kLnChiHi - kLnChiLo);
        const double chi = exp(lnchi), r = uniform52(w0.z, w0.w), s = 2.0 * uniform52(w1.x, w1.y) - 1.0;
        const MixPoint m = mix_point(T, chi, r, s);
        const double Lb = mix_baseline(T, m), L = mix_quantile<44, 32>(T, m, r);
        float x[3];
        mlp_features(chi, r, s, x);
        X[3 * i] = x[0];
        X[3 * i + 1] = x[1];
        X[3 * i + 2] = x[2];
        Y[4 * i] = (float)(kOutScale * (L - Lb));
        Y[4 * i + 1] = 0.0f;
        Y[4 * i + 2] = 0.0f;
        Y[4 * i + 3] = (float)(kOutScale * (xi3_at(bes_tab, chi, L, s) - xi3_at(bes_tab, chi, Lb, s)));
        if (raw) {
            raw[3 * i] = chi;
            raw[3 * i + 1] = r;
            raw[3 * i + 2] = s;
        }
    }
}

// ---- BF16 helpers -------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // .x = lo (lower 16 bits), .y = hi
    return *reinterpret_cast<const uint32_t*>(&v);
}

// ---- AdamW ----------------------------------------------------------------------------------------
__device__ __forceinline__ bool is_weight(int k) {
    return k < kOffB1 || (k >= kOffW2 && k < kOffB2) || (k >= kOffW3 && k < kOffB3) || (k >= kOffW4 && k < kOffB4);
}

// AdamW (decoupled weight decay on weights only); t = step count after this update.  zero (may be NULL): the gradient
// array to clear for the next step's sums (the same as G in the training loop)
__global__ void mlp_adamw_kernel(float* P, float* Mm, float* Vv, const float* G, float lr, float wd, float b1t, float b2t,
                                 float* zero) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kParams) return;
    const float g = G[k];
    const float m = 0.9f * Mm[k] + 0.1f * g;
    const float v = 0.999f * Vv[k] + 0.001f * g * g;
    Mm[k] = m;
    Vv[k] = v;
    const float mh = m / (1.0f - b1t), vh = v / (1.0f - b2t);
    float upd = mh / (sqrtf(vh) + 1e-8f);
    if (is_weight(k)) upd += wd * P[k];
    P[k] -= lr * upd;
    if (zero) zero[k] = 0.0f;
}

// Blocks per SM of the tensor-core kernels: 4 by registers (128 a thread; 39 KB of shared memory and 64 of the SM's 512
// TMEM columns each leave room for more).  The occupancy query answers 1 for a kernel that allocates TMEM; a grid of
// one block per SM took 4.0 ms for 1e6 checked samples, one of four 2.8.
constexpr int kTcPerSm = 4;

// ---- fused inference on the 5th-generation tensor cores ---------------------------------------------
// A block of 128 threads takes 128 samples at a time, one per thread and one per TMEM lane.  Layer 1
// (K = 3) runs in FP32 on the CUDA cores; each thread writes its 64 SiLU outputs as BF16 into the A
// tile in shared memory; one thread issues the 128 x 64 x 64 layer as four tcgen05.mma (K = 16 each)
// with the FP32 accumulator in TMEM and commits them to an mbarrier; every thread then reads its row
// of the accumulator (tcgen05.ld), adds the bias, applies SiLU and writes the next layer's A row.  The
// output layer is padded to 16 rows (the smallest MMA width at M = 128).  Operands are K-major without
// swizzle: core matrices of 8 rows x 16 bytes, 128 bytes apart along K, 8-row groups 1024 bytes apart.
constexpr int kIW = 4;         // warps per block
constexpr int kTR = kIW * 32;  // samples per tile (the MMA's M)
constexpr int kTN4 = 16;       // output layer rows after padding
constexpr uint32_t kTmemCols = 64;
constexpr int kTcWaitLimit = 1 << 24;  // bounded mbarrier polling (~0.1 s) before giving up

struct TcShared {
    alignas(1024) unsigned char a[kTR * kH * 2];  // activations (A operand), 16 KB
    alignas(1024) unsigned char w2[kH * kH * 2];  // W2, W3 as B operands (N = 64 rows of K = 64)
    alignas(1024) unsigned char w3[kH * kH * 2];
    alignas(1024) unsigned char w4[kTN4 * kH * 2];  // W4 padded to 16 rows
    float w1[kOffW2];                               // W1, b1 (FP32)
    float b2[kH], b3[kH], b4[4];
    uint64_t bar;            // MMA completion
    uint32_t tmem;           // TMEM base address of the accumulator
};

// byte offset of element (row r, column k) in a K-major tile with K = 64
__device__ __forceinline__ uint32_t kmaj(int r, int k) {
    return (uint32_t)((r >> 3) * 1024 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint32_t sm_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading (K) and stride (8-row group) byte offsets,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t tc_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTR >> 4) << 24);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// the 16 accumulator columns c0.. of this thread's TMEM lane
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// D = A W^T for the A tile and the B operand w (n rows): thread 0 issues, every thread waits.  Returns
// false (in every thread) if the wait gave up.
__device__ bool tc_layer(TcShared& S, const unsigned char* w, int n, uint32_t& phase) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the A rows written above, to the MMA
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x == 0) {
        const uint32_t id = tc_idesc(n);
#pragma unroll
        for (int ks = 0; ks < kH / 16; ++ks) {
            const uint64_t da = tc_desc(sm_u32(S.a) + 256 * ks), db = tc_desc(sm_u32(w) + 256 * ks);
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(S.tmem),
                "l"(da), "l"(db), "r"(id), "r"((uint32_t)ks)
                : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sm_u32(&S.bar))
                     : "memory");
    }
    bool done = false;
    for (int i = 0; i < kTcWaitLimit && !done; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(sm_u32(&S.bar)), "r"(phase)
            : "memory");
        done = ok != 0;
    }
    phase ^= 1u;
    tc_fence_after();
    return __syncthreads_and(done) != 0;
}

// this thread's 64 activations, bias + SiLU, into its A row as BF16
__device__ __forceinline__ void tc_store_row(TcShared& S, const float v[kH]) {
    const int r = threadIdx.x;
#pragma unroll
    for (int c = 0; c < kH / 8; ++c) {
        uint4 q;
        q.x = pack_bf16(v[8 * c], v[8 * c + 1]);
        q.y = pack_bf16(v[8 * c + 2], v[8 * c + 3]);
        q.z = pack_bf16(v[8 * c + 4], v[8 * c + 5]);
        q.w = pack_bf16(v[8 * c + 6], v[8 * c + 7]);
        *reinterpret_cast<uint4*>(S.a + kmaj(r, 8 * c)) = q;
    }
}

// layers 1-4 for this thread's features x; o = raw outputs.  False if the tensor cores did not answer.
__device__ bool tc_infer(TcShared& S, const float x[3], uint32_t& phase, float o[4]) {
    float v[kH];
#pragma unroll
    for (int k = 0; k < kH; ++k) {
        const float* w = S.w1 + 3 * k;
        v[k] = silu_f(fmaf(w[0], x[0], fmaf(w[1], x[1], fmaf(w[2], x[2], S.w1[kOffB1 + k]))));
    }
    tc_store_row(S, v);
    const uint32_t lane_addr = S.tmem + ((uint32_t)(threadIdx.x & ~31) << 16);
#pragma unroll 1
    for (int layer = 0; layer < 2; ++layer) {
        if (!tc_layer(S, layer == 0 ? S.w2 : S.w3, kH, phase)) return false;
        const float* bias = layer == 0 ? S.b2 : S.b3;
#pragma unroll
        for (int c0 = 0; c0 < kH; c0 += 16) tc_ld16(lane_addr + (uint32_t)c0, v + c0);
#pragma unroll
        for (int k = 0; k < kH; ++k) v[k] = silu_f(v[k] + bias[k]);
        tc_store_row(S, v);
    }
    if (!tc_layer(S, S.w4, kTN4, phase)) return false;
    float u[16];
    tc_ld16(lane_addr, u);
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = u[j] + S.b4[j];
    return true;
}

// weights into shared memory, the mbarrier, and the TMEM accumulator (warp 0)
__device__ void tc_setup(TcShared& S, const float* __restrict__ P) {
    const int tid = threadIdx.x;
    for (int i = tid; i < kOffW2; i += blockDim.x) S.w1[i] = P[i];
    for (int i = tid; i < kH; i += blockDim.x) {
        S.b2[i] = P[kOffB2 + i];
        S.b3[i] = P[kOffB3 + i];
    }
    if (tid < 4) S.b4[tid] = P[kOffB4 + tid];
    for (int i = tid; i < kH * kH; i += blockDim.x) {
        const int r = i / kH, k = i % kH;
        *reinterpret_cast<__nv_bfloat16*>(S.w2 + kmaj(r, k)) = __float2bfloat16_rn(P[kOffW2 + i]);
        *reinterpret_cast<__nv_bfloat16*>(S.w3 + kmaj(r, k)) = __float2bfloat16_rn(P[kOffW3 + i]);
    }
    for (int i = tid; i < kTN4 * kH; i += blockDim.x) {
        const int r = i / kH, k = i % kH;
        *reinterpret_cast<__nv_bfloat16*>(S.w4 + kmaj(r, k)) = __float2bfloat16_rn(r < 4 ? P[kOffW4 + i] : 0.0f);
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sm_u32(&S.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_u32(&S.tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

__device__ void tc_teardown(uint32_t tmem) {
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// ---- training: forward, backward and weight gradients of a tile of 128 samples in one kernel ------------
// A block keeps 128 samples, one per TMEM lane, through the whole pass: nothing of the network's 64-wide activations goes
// to global memory.  Layers 2-4 forward and the input gradients of layers 3 and 2 are
// tcgen05.mma of the sample-major tile (M = samples) with the weights or their transposes; the weight gradients of
// layers 2 and 3 are tcgen05.mma over K = 128 samples (M = output units in the lower 64 rows, the upper 64 zero;
// N = input units) that stay in TMEM over the block's tiles.  As in a GEMM of its own, every operand is rounded to
// BF16 and sums are FP32; biases, layer 1 and the 4-wide layer's gradient are FP32 sums over the warp's lanes.
// TMEM columns: Z2, Z3, a scratch accumulator, dW3, dW2.
// Nine GEMM launches that staged their operands from FP32 arrays in global memory (13-80 us each on 32 blocks) and
// ten elementwise and column-sum launches took 0.34 ms for a batch of 4096; this pass takes 23 us.
constexpr uint32_t kTrainCols = 512;
constexpr uint32_t kColZ2 = 0, kColZ3 = 64, kColT = 128, kColW3 = 192, kColW2 = 256;

struct TrainShared {
    alignas(1024) unsigned char a[kTR * kH * 2];        // A operand: 128 samples x 64
    alignas(1024) unsigned char w2[kH * kH * 2];        // B operands: W2, W3 (N = output units)
    alignas(1024) unsigned char w3[kH * kH * 2];
    alignas(1024) unsigned char w2t[kH * kH * 2];       // their transposes (N = input units)
    alignas(1024) unsigned char w3t[kH * kH * 2];
    alignas(1024) unsigned char w4[kTN4 * kH * 2];      // W4 padded to 16 rows
    alignas(1024) unsigned char h1t[kH * kTR * 2];      // B operands: H1^T, H2^T (64 units x 128 samples)
    alignas(1024) unsigned char h2t[kH * kTR * 2];
    alignas(1024) unsigned char dzt[kTR * kTR * 2];     // A operand: dZ^T (64 units x 128 samples, upper 64 rows zero)
    float w1[kOffW2];                                   // W1, b1 (FP32)
    float b2[kH], b3[kH], b4[4];
    float w4r[4][kH];                                   // W4 rounded to BF16
    uint64_t bar;
    uint32_t tmem;
};

// byte offset of (row r, column k) in a K-major tile with K = 128
__device__ __forceinline__ uint32_t kmaj128(int r, int k) {
    return (uint32_t)((r >> 3) * 2048 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// the float at p of this block's shared memory, in the block of the given rank of the cluster
__device__ __forceinline__ float cluster_ld(const float* p, uint32_t rank) {
    uint32_t addr;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(sm_u32(p)), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// one thread: D (+)= A B^T over ks steps of K = 16; group strides in bytes
__device__ __forceinline__ void tc_issue(uint32_t d, uint32_t a, uint32_t asbo, uint32_t b, uint32_t bsbo, int ks, uint32_t id,
                                         bool acc) {
    for (int k = 0; k < ks; ++k) {
        const uint64_t da = (tc_desc(a + 256 * k) & ~((uint64_t)0x3FFF << 32)) | ((uint64_t)(asbo >> 4) << 32);
        const uint64_t db = (tc_desc(b + 256 * k) & ~((uint64_t)0x3FFF << 32)) | ((uint64_t)(bsbo >> 4) << 32);
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
            "l"(da), "l"(db), "r"(id), "r"((uint32_t)(acc || k > 0))
            : "memory");
    }
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sm_u32(bar)) : "memory");
}

// every thread: the shared-memory operands written so far, to the MMA
__device__ __forceinline__ void tc_publish() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

// every thread: wait for the committed MMAs (bounded); false in every thread if the wait gave up
__device__ __forceinline__ bool tc_await(uint64_t* bar, uint32_t& phase) {
    bool done = false;
    for (int i = 0; i < kTcWaitLimit && !done; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(sm_u32(bar)), "r"(phase)
            : "memory");
        done = ok != 0;
    }
    phase ^= 1u;
    tc_fence_after();
    return __syncthreads_and(done) != 0;
}

// Four threads share a sample, 16 units each (a warp reads the TMEM lanes of its index modulo 4): the elementwise work
// and the column sums are what a pass costs, and one thread per sample left a single warp on each scheduler (61 us a
// pass of 32 tiles against 25 with four; 23 now).
constexpr int kTrainThreads = 4 * kTR;
constexpr int kTU = 16;  // units per thread

// this thread's 16 values as BF16: its part of its row of the sample-major A tile, and of its column of a unit-major
// tile
__device__ __forceinline__ void train_row(unsigned char* a, int c0, const float v[kTU]) {
#pragma unroll
    for (int c = 0; c < kTU / 8; ++c) {
        uint4 q;
        q.x = pack_bf16(v[8 * c], v[8 * c + 1]);
        q.y = pack_bf16(v[8 * c + 2], v[8 * c + 3]);
        q.z = pack_bf16(v[8 * c + 4], v[8 * c + 5]);
        q.w = pack_bf16(v[8 * c + 6], v[8 * c + 7]);
        *reinterpret_cast<uint4*>(a + kmaj(threadIdx.x & (kTR - 1), c0 + 8 * c)) = q;
    }
}
__device__ __forceinline__ void train_column(unsigned char* t, int c0, const float v[kTU]) {
#pragma unroll
    for (int j = 0; j < kTU; ++j)
        *reinterpret_cast<__nv_bfloat16*>(t + kmaj128(c0 + j, threadIdx.x & (kTR - 1))) = __float2bfloat16_rn(v[j]);
}

// sums of 16 columns over the warp's lanes: lanes 2 c and 2 c + 1 get column c's, added to s (v is used up).  At each
// step a lane keeps the half of its columns that its lane bit names and gets its partner's sums of that half: 16
// shuffles for 16 columns.
template <int W>
__device__ __forceinline__ void column_fold(float v[kTU]) {
    const bool upper = threadIdx.x & (2 * W);
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const float send = upper ? v[i] : v[i + W], keep = upper ? v[i + W] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * W);
    }
}
__device__ __forceinline__ void column_sums(float v[kTU], float& s) {
    column_fold<8>(v);
    column_fold<4>(v);
    column_fold<2>(v);
    column_fold<1>(v);
    s += v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// What a block adds up over its warps: per unit b3, b2, b1, the four dW4 and the three dW1 values, then the loss and
// dL/db4.  Four warps hold such sums of the same units, from a quarter of the tile's samples each.
constexpr int kWarpSums = 10 * kH + 5;
__device__ __forceinline__ int warp_sum_index(int e) {  // entry e's parameter (kParams: the loss)
    const int f = e / kH, j = e % kH;
    if (f >= 10) return e == 10 * kH ? kParams : kOffB4 + e - (10 * kH + 1);
    if (f >= 7) return kOffW1 + 3 * j + (f - 7);
    if (f >= 3) return kOffW4 + (f - 3) * kH + j;
    return (f == 0 ? kOffB3 : (f == 1 ? kOffB2 : kOffB1)) + j;
}

// Batches of up to 8 tiles run as one cluster, whose blocks' sums are added in the order of their ranks through
// distributed shared memory: the gradients of such a batch, and networks trained on it, repeat bit for bit.  Larger
// batches add their blocks' sums atomically, in the order they arrive.  (The warps' sums are added in shared memory
// first: 8836 atomic adds a block; 4 x 644 + 8192 of them, uncoalesced, cost 2 us of a step of 4096 samples.)
constexpr int kTrainCluster = 8;

// grad (zeroed by the caller) += dL/dparameters, loss (may be NULL) += L of the n samples (X, Tg)
__global__ void __launch_bounds__(kTrainThreads, 1) mlp_train_kernel(const float* __restrict__ P, const float* __restrict__ X,
                                                           const float* __restrict__ Tg, int64_t n, float* __restrict__ grad,
                                                           float* __restrict__ loss) {
    extern __shared__ __align__(1024) unsigned char train_smem[];
    TrainShared& S = *reinterpret_cast<TrainShared*>(train_smem);
    const int tid = threadIdx.x, lane = tid & 31, c0 = (tid / kTR) * kTU;  // this thread's units c0 .. c0 + 15
    for (int i = tid; i < kOffW2; i += kTrainThreads) S.w1[i] = P[i];
    for (int i = tid; i < kH; i += kTrainThreads) {
        S.b2[i] = P[kOffB2 + i];
        S.b3[i] = P[kOffB3 + i];
    }
    if (tid < 4) S.b4[tid] = P[kOffB4 + tid];
    for (int i = tid; i < kH * kH; i += kTrainThreads) {
        const int r = i / kH, k = i % kH;
        const __nv_bfloat16 a = __float2bfloat16_rn(P[kOffW2 + i]), b = __float2bfloat16_rn(P[kOffW3 + i]);
        *reinterpret_cast<__nv_bfloat16*>(S.w2 + kmaj(r, k)) = a;
        *reinterpret_cast<__nv_bfloat16*>(S.w3 + kmaj(r, k)) = b;
        *reinterpret_cast<__nv_bfloat16*>(S.w2t + kmaj(k, r)) = a;
        *reinterpret_cast<__nv_bfloat16*>(S.w3t + kmaj(k, r)) = b;
    }
    for (int i = tid; i < kTN4 * kH; i += kTrainThreads) {
        const int r = i / kH, k = i % kH;
        const float w = r < 4 ? bf16_round(P[kOffW4 + i]) : 0.0f;
        *reinterpret_cast<__nv_bfloat16*>(S.w4 + kmaj(r, k)) = __float2bfloat16_rn(w);
        if (r < 4) S.w4r[r][k] = w;
    }
    for (int i = tid; i < (int)(sizeof(S.dzt) / 16); i += kTrainThreads) reinterpret_cast<uint4*>(S.dzt)[i] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sm_u32(&S.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_u32(&S.tmem)),
                     "r"(kTrainCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = S.tmem, row = tm + ((uint32_t)(tid & (kTR - 1) & ~31) << 16);
    const uint32_t id64 = tc_idesc(kH), id16 = tc_idesc(kTN4);
    const float inv = 1.0f / (float)n;
    uint32_t phase = 0;
    bool ok = true;
    float lsum = 0.0f, sb4[4] = {0, 0, 0, 0}, sb3 = 0.0f, sb2 = 0.0f, sb1 = 0.0f, sw4[4] = {}, sw1[3] = {};
    bool first = true;
    for (int64_t base = (int64_t)blockIdx.x * kTR; base < n && ok; base += (int64_t)gridDim.x * kTR, first = false) {
        const int64_t i = base + (tid & (kTR - 1));
        const bool have = i < n;
        float x[3] = {0.0f, 0.0f, 0.0f}, v[kTU];
        if (have)
            for (int q = 0; q < 3; ++q) x[q] = X[3 * i + q];
        // forward
#pragma unroll
        for (int k = 0; k < kTU; ++k) {
            const float* w = S.w1 + 3 * (c0 + k);
            v[k] = silu_f(fmaf(w[0], x[0], fmaf(w[1], x[1], fmaf(w[2], x[2], S.w1[kOffB1 + c0 + k]))));
        }
        train_row(S.a, c0, v);
        train_column(S.h1t, c0, v);
        tc_publish();
        if (tid == 0) {
            tc_issue(tm + kColZ2, sm_u32(S.a), 1024, sm_u32(S.w2), 1024, kH / 16, id64, false);
            tc_commit(&S.bar);
        }
        if (!(ok = tc_await(&S.bar, phase))) break;
        tc_ld16(row + kColZ2 + c0, v);
#pragma unroll
        for (int k = 0; k < kTU; ++k) v[k] = silu_f(v[k] + S.b2[c0 + k]);
        train_row(S.a, c0, v);
        train_column(S.h2t, c0, v);
        tc_publish();
        if (tid == 0) {
            tc_issue(tm + kColZ3, sm_u32(S.a), 1024, sm_u32(S.w3), 1024, kH / 16, id64, false);
            tc_commit(&S.bar);
        }
        if (!(ok = tc_await(&S.bar, phase))) break;
        tc_ld16(row + kColZ3 + c0, v);
#pragma unroll
        for (int k = 0; k < kTU; ++k) v[k] = silu_f(v[k] + S.b3[c0 + k]);
        train_row(S.a, c0, v);
        tc_publish();
        if (tid == 0) {
            tc_issue(tm + kColT, sm_u32(S.a), 1024, sm_u32(S.w4), 1024, kH / 16, id16, false);
            tc_commit(&S.bar);
        }
        if (!(ok = tc_await(&S.bar, phase))) break;
        // outputs, loss and their gradient
        float u[16], d[4];
        tc_ld16(row + kColT, u);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float e = have ? u[q] + S.b4[q] - Tg[4 * i + q] : 0.0f;
            lsum = fmaf(e * inv, e, lsum);
            d[q] = 2.0f * e * inv;
            sb4[q] += d[q];
            d[q] = bf16_round(d[q]);
        }
        // layer 4: dW4 (v still holds H3), then dZ3 = (dO W4) silu'(Z3)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float t[kTU];
#pragma unroll
            for (int k = 0; k < kTU; ++k) t[k] = d[q] * bf16_round(v[k]);
            column_sums(t, sw4[q]);
        }
        tc_ld16(row + kColZ3 + c0, v);
#pragma unroll
        for (int k = 0; k < kTU; ++k)
            v[k] = fmaf(d[3], S.w4r[3][c0 + k], fmaf(d[2], S.w4r[2][c0 + k], fmaf(d[1], S.w4r[1][c0 + k], d[0] * S.w4r[0][c0 + k]))) *
                   dsilu_f(v[k] + S.b3[c0 + k]);
        train_row(S.a, c0, v);
        train_column(S.dzt, c0, v);
        tc_publish();
        if (tid == 0) {
            tc_issue(tm + kColT, sm_u32(S.a), 1024, sm_u32(S.w3t), 1024, kH / 16, id64, false);
            tc_issue(tm + kColW3, sm_u32(S.dzt), 2048, sm_u32(S.h2t), 2048, kTR / 16, id64, !first);
            tc_commit(&S.bar);
        }
        column_sums(v, sb3);
        if (!(ok = tc_await(&S.bar, phase))) break;
        // layer 3 -> dZ2
        {
            float z[kTU];
            tc_ld16(row + kColT + c0, v);
            tc_ld16(row + kColZ2 + c0, z);
#pragma unroll
            for (int k = 0; k < kTU; ++k) v[k] *= dsilu_f(z[k] + S.b2[c0 + k]);
        }
        train_row(S.a, c0, v);
        train_column(S.dzt, c0, v);
        tc_publish();
        if (tid == 0) {
            tc_issue(tm + kColT, sm_u32(S.a), 1024, sm_u32(S.w2t), 1024, kH / 16, id64, false);
            tc_issue(tm + kColW2, sm_u32(S.dzt), 2048, sm_u32(S.h1t), 2048, kTR / 16, id64, !first);
            tc_commit(&S.bar);
        }
        column_sums(v, sb2);
        if (!(ok = tc_await(&S.bar, phase))) break;
        // layer 2 -> dZ1, layer 1 (FP32)
        tc_ld16(row + kColT + c0, v);
#pragma unroll
        for (int k = 0; k < kTU; ++k) {
            const float* w = S.w1 + 3 * (c0 + k);
            v[k] *= dsilu_f(fmaf(w[0], x[0], fmaf(w[1], x[1], fmaf(w[2], x[2], S.w1[kOffB1 + c0 + k]))));
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            float t[kTU];
#pragma unroll
            for (int k = 0; k < kTU; ++k) t[k] = v[k] * x[q];
            column_sums(t, sw1[q]);
        }
        column_sums(v, sb1);
    }
    // the block's sums, in the order of the parameters, the loss behind them (over the operand tiles, whose last MMAs
    // have been awaited)
    static_assert(sizeof(S.h1t) + sizeof(S.h2t) + sizeof(S.dzt) >= (kParams + 1) * sizeof(float), "the block's sums");
    static_assert(sizeof(S.a) >= kTR / 32 * kWarpSums * sizeof(float), "the warps' sums");
    float* sums = reinterpret_cast<float*>(S.h1t);
    float* part = reinterpret_cast<float*>(S.a);
    const float bad = __int_as_float(0x7FC00000);
    const int u0 = tid & (kTR - 1);
    if (u0 < kH) {  // (whole warps: the accumulator loads are collective)
        float a[kTU] = {}, b[kTU] = {};
        if (!first) {
            tc_ld16(row + kColW3 + c0, a);
            tc_ld16(row + kColW2 + c0, b);
        }
#pragma unroll
        for (int q = 0; q < kTU; ++q) {
            sums[kOffW3 + u0 * kH + c0 + q] = ok ? a[q] : bad;
            sums[kOffW2 + u0 * kH + c0 + q] = ok ? b[q] : bad;
        }
    }
    float* mine = part + (u0 >> 5) * kWarpSums;
    if (!(lane & 1)) {
        const int j = c0 + (lane >> 1);
        mine[j] = sb3;
        mine[kH + j] = sb2;
        mine[2 * kH + j] = sb1;
#pragma unroll
        for (int q = 0; q < 4; ++q) mine[(3 + q) * kH + j] = sw4[q];
#pragma unroll
        for (int q = 0; q < 3; ++q) mine[(7 + q) * kH + j] = sw1[q];
    }
    if (c0 == 0) {  // one of a sample's four threads
        for (int o = 16; o > 0; o >>= 1) {
            lsum += __shfl_down_sync(0xffffffffu, lsum, o);
#pragma unroll
            for (int q = 0; q < 4; ++q) sb4[q] += __shfl_down_sync(0xffffffffu, sb4[q], o);
        }
        if (lane == 0) {
            mine[10 * kH] = lsum;
#pragma unroll
            for (int q = 0; q < 4; ++q) mine[10 * kH + 1 + q] = sb4[q];
        }
    }
    __syncthreads();
    for (int e = tid; e < kWarpSums; e += kTrainThreads) {
        float v = part[e];
        for (int k = 1; k < kTR / 32; ++k) v += part[k * kWarpSums + e];
        sums[warp_sum_index(e)] = ok ? v : bad;
    }
    uint32_t rank, ranks;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(ranks));
    cluster_sync();  // (a cluster of one where the launch names none)
    if (ranks > 1) {  // the whole batch: one add per address, so their order is of no matter
        for (int i = (int)rank * kTrainThreads + tid; i <= kParams; i += (int)ranks * kTrainThreads) {
            float v = 0.0f;
            for (uint32_t k = 0; k < ranks; ++k) v += cluster_ld(sums + i, k);
            if (i < kParams) atomicAdd(&grad[i], v);
            else if (loss) atomicAdd(loss, v);
        }
        cluster_sync();  // no block leaves while another reads its sums
    } else {
        for (int i = tid; i < kParams; i += kTrainThreads) atomicAdd(&grad[i], sums[i]);
        if (tid == 0 && loss) atomicAdd(loss, sums[kParams]);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(kTrainCols) : "memory");
}

// raw network outputs for feature rows X[n][3] (NaN where the tensor cores did not answer)
__global__ void __launch_bounds__(kTR) mlp_forward_kernel(const float* __restrict__ P, const float* __restrict__ X,
                                                          int64_t n, float* __restrict__ O) {
    __shared__ TcShared S;
    tc_setup(S, P);
    uint32_t phase = 0;
    bool broken = false;  // a wait gave up: the remaining tiles skip the network (the same in every thread)
    for (int64_t base = (int64_t)blockIdx.x * kTR; base < n; base += (int64_t)gridDim.x * kTR) {
        const int64_t i = base + threadIdx.x;
        float x[3] = {0.0f, 0.0f, 0.0f}, o[4];
        if (i < n)
            for (int q = 0; q < 3; ++q) x[q] = X[3 * i + q];
        broken = broken || !tc_infer(S, x, phase, o);
        if (broken)
            for (int j = 0; j < 4; ++j) o[j] = __int_as_float(0x7FC00000);
        if (i < n)
            for (int j = 0; j < 4; ++j) O[4 * i + j] = o[j];
    }
    tc_teardown(S.tmem);
}

// flags bit of the sampling kernel for callers that use ln u' only (the batched step's event pass):
// no Stokes outputs, so neither their check nor xi3 on the table path
constexpr int kLnUpOnly = 4;

// the table path for sample i (the exact mixture quantile, and xi3 there unless ln_up_only): by Newton, or with
// bracket by the bracketing solver; false: Newton does not reach it, nothing is written
__device__ __noinline__ bool table_path(const TabP<double>& T, const TabP<float>& T32, const double* __restrict__ besp,
                                        const double* __restrict__ chi_in, const double* __restrict__ r_in,
                                        const double* __restrict__ s_in, int64_t i, float* __restrict__ out4, bool ln_up_only,
                                        bool bracket) {
    const double chi = chi_in[i], r = r_in[i], s = s_in[i];
    const MixPoint m = mix_point(T, chi, r, s);
    double L;
    if (bracket)
        L = mix_quantile<44, 32>(T, m, r);
    else if (!mix_quantile_fast(T, T32, m, r, L))
        return false;
    out4[4 * i] = (float)L;
    out4[4 * i + 1] = 0.0f;
    out4[4 * i + 2] = 0.0f;
    out4[4 * i + 3] = ln_up_only ? 0.0f : (float)xi3_poly(besp, chi, L, s);
    return true;
}

// The check of a network sample, first on the float tables: the FP32 CDF and xi3 errors are within ~1e-6
// of the FP64 ones, so a sample whose FP32 errors are below tol - kMargin32 passes and one with an error
// above tol + kMargin32 fails without FP64 work; only samples in the band between are checked again on
// the FP64 tables (the FP64 pipe of this GPU runs at 1/64 of the FP32 rate).
constexpr float kMargin32 = 1e-5f;

// The sampler is two kernels.  The first runs the network and leaves its raw outputs in out4; the second checks
// them.  In one kernel the check's warps, which differ in their solves, met at the eight barriers of every 128-sample
// tile of the network, and the two codes together missed the instruction cache (barrier and no-instruction stalls
// were 23 of 33 cycles between issues).  1e6 checked samples of a trained network, 1.1 % of them from the tables: 4.0 ms
// in one kernel with one block per SM, 2.8 ms with four, 0.69 ms in two kernels with the solves above.
constexpr uint32_t kNoNet = 0x7FC0BAD0u;  // o[0] of a tile the tensor cores did not answer for (a NaN of its own)

__global__ void __launch_bounds__(kTR, kTcPerSm) mlp_net_kernel(const float* __restrict__ P,
                                                                const double* __restrict__ chi_in,
                                                                const double* __restrict__ r_in,
                                                                const double* __restrict__ s_in, int64_t n,
                                                                float* __restrict__ out4,
                                                                const unsigned long long* __restrict__ n_dev) {
    __shared__ TcShared S;
    if (n_dev) {  // a count the previous kernel of the stream left on the device
        const int64_t nd = (int64_t)*n_dev;
        if (nd < n) n = nd;
    }
    tc_setup(S, P);
    uint32_t phase = 0;
    bool broken = false;  // a wait gave up: the remaining tiles skip the network (the same in every thread)
    for (int64_t base = (int64_t)blockIdx.x * kTR; base < n; base += (int64_t)gridDim.x * kTR) {
        const int64_t i = base + threadIdx.x;
        float x[3] = {0.0f, 0.0f, 0.0f}, o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (i < n) mlp_features(chi_in[i], r_in[i], s_in[i], x);
        if (!broken) broken = !tc_infer(S, x, phase, o);
        if (broken) o[0] = __uint_as_float(kNoNet);
        if (i < n)
            for (int j = 0; j < 4; ++j) out4[4 * i + j] = o[j];  // (the caller's array need not be aligned to 16 bytes)
    }
    tc_teardown(S.tmem);
}

// The check: samples that pass on the float tables are done; the others wait in a block-wide queue, and a full block
// of them at a time goes through FP64 (the check again for those within kMargin32 of the bound, the table path for
// those that fail it, and for all of them with flags bit 0).  One block of 1024 threads per SM: the queue's last,
// partly filled pass then runs in a few warps of every SM.  The tiles are cut so that every SM has as many samples, and
// few samples get blocks of 128 threads: in tiles of 1024, the FP64 passes of 2000 samples ran on two SMs (551 us at
// a bound of 1e-5, longer than the 502 of the fused kernel's tiles of 128; 105 so).  Samples that need the bracketing solver (a logit above the
// grid: uniforms within 2e-9 of 1) wait in a second queue: it takes ~20 times Newton's instructions, and run in the
// lane that met it, it held that lane's whole warp (4e5 table samples, 1 in 24 of them such: 22.7 ms, with the queue
// 14.8).
constexpr int kCheckThreads = 1024;
constexpr int kCheckFew = 128;  // threads of a block when one tile of that size per SM takes all samples

struct CheckItem {
    int64_t i;
    float L, o3, yu, yd;  // the sample and its logits, where the FP64 check decides (yu NaN: the table path)
};

__global__ void __launch_bounds__(kCheckThreads, 1) mlp_check_kernel(TabP<double> T, TabP<float> T32,
                                                                     const float* __restrict__ bes32,
                                                                     const double* __restrict__ besp,
                                                                     const double* __restrict__ chi_in,
                                                                     const double* __restrict__ r_in,
                                                                     const double* __restrict__ s_in, int64_t n, double tol,
                                                                     int flags, float* __restrict__ out4,
                                                                     uint8_t* __restrict__ fell, float* __restrict__ err_out,
                                                                     unsigned long long* n_fallback,
                                                                     const unsigned long long* __restrict__ n_dev) {
    extern __shared__ __align__(16) unsigned char check_smem[];
    const int threads = blockDim.x;
    CheckItem* queue = reinterpret_cast<CheckItem*>(check_smem);             // [2 blockDim.x]
    int64_t* slow = reinterpret_cast<int64_t*>(queue + 2 * threads);         // [2 blockDim.x]
    __shared__ int queued, n_slow;
    if (n_dev) {
        const int64_t nd = (int64_t)*n_dev;
        if (nd < n) n = nd;
    }
    if (threadIdx.x == 0) queued = n_slow = 0;
    __syncthreads();
    const bool table_only = (flags & 1) != 0, ln_up_only = (flags & kLnUpOnly) != 0;
    const float ftol = (float)tol;
    unsigned nf = 0;  // this thread's fallbacks
    int held = 0;     // queued samples (the same in every thread)
    // a queued sample: the FP64 check decides, then the table path
    auto finish = [&](const CheckItem& q) {
        bool fb = true;
        if (!isnan(q.yu)) {
            const double chi = chi_in[q.i], r = r_in[q.i], s = s_in[q.i];
            const MixPoint m = mix_point(T, chi, r, s);
            const double e64 = mix_error64(T, m, (double)q.L, r, q.yu, q.yd);
            double d64 = 0.0;
            if (!ln_up_only)
                d64 = fabs(xi3_poly(besp, chi, mix_baseline(T, m), s) + (double)q.o3 / kOutScale -
                           xi3_poly(besp, chi, (double)q.L, s));
            if (err_out) err_out[q.i] = (float)e64;
            fb = !(e64 <= tol) || !(d64 <= tol);
        }
        if (fell) fell[q.i] = fb ? 1 : 0;
        if (fb) {
            if (!table_path(T, T32, besp, chi_in, r_in, s_in, q.i, out4, ln_up_only, false))
                slow[atomicAdd(&n_slow, 1)] = q.i;  // at most 2 blockDim.x - 1 entries
            ++nf;
        }
    };
    // tiles of equal size for every block: as many rounds as 1024 samples a block would take, in full warps
    const int64_t most = (int64_t)gridDim.x * threads, rounds = max((int64_t)1, (n + most - 1) / most);
    const int tile = (int)((n + gridDim.x * rounds - 1) / (gridDim.x * rounds) + 31) & ~31;
    for (int64_t base = (int64_t)blockIdx.x * tile; base < n; base += (int64_t)gridDim.x * tile) {
        const int64_t i = base + threadIdx.x;
        bool waits = false;  // this thread's sample went to the queue
        if ((int)threadIdx.x < tile && i < n) {
            CheckItem q{i, 0.0f, 0.0f, __int_as_float(0x7FC00000), 0.0f};
            bool done = false;
            if (table_only) {
                if (err_out) err_out[i] = -1.0f;
            } else {
                const float4 o = make_float4(out4[4 * i], out4[4 * i + 1], out4[4 * i + 2], out4[4 * i + 3]);
                if (__float_as_uint(o.x) == kNoNet) {
                    if (err_out) err_out[i] = -1.0f;
                } else {
                    const double chi = chi_in[i], r = r_in[i], s = s_in[i];
                    // the sample on the float tables: baseline, correction, CDF error (and xi3's)
                    const MixPointT<float> m32 = mix_point32(T32, chi, r, s);
                    const float Lb = mix_baseline(T32, m32);
                    const float L = Lb + o.x / (float)kOutScale;
                    float xi1 = 0.0f, xi2 = 0.0f, xi3 = 0.0f, dxi3 = 0.0f;
                    if (!ln_up_only) {
                        xi1 = o.y / (float)kOutScale;
                        xi2 = o.z / (float)kOutScale;
                        xi3 = xi3_at32(bes32, (float)chi, Lb, (float)s) + o.w / (float)kOutScale;
                        dxi3 = fabsf(xi3 - xi3_at32(bes32, (float)chi, L, (float)s));
                    }
                    float yu, yd;
                    const float err_q = fabsf(mix_cdf32(T32, m32, L, yu, yd) - (float)r);  // the CDF check
                    const bool stokes_ok = fabsf(xi1) <= ftol && fabsf(xi2) <= ftol;
                    const bool pass32 = err_q <= ftol - kMargin32 && dxi3 <= ftol - kMargin32 && stokes_ok;
                    const bool fail32 = !(err_q <= ftol + kMargin32) || !(dxi3 <= ftol + kMargin32) || !stokes_ok;
                    if (err_out) err_out[i] = err_q;
                    done = pass32;
                    if (!fail32) {  // (one that fails leaves its row to the table path)
                        out4[4 * i] = L;
                        out4[4 * i + 1] = xi1;
                        out4[4 * i + 2] = xi2;
                        out4[4 * i + 3] = xi3;
                        if (!pass32) {  // the band around tol: the FP64 check decides
                            q.L = L;
                            q.o3 = o.w;
                            q.yu = yu;
                            q.yd = yd;
                        }
                    }
                }
            }
            if (done) {
                if (fell) fell[i] = 0;
            } else {
                queue[atomicAdd(&queued, 1)] = q;  // at most 2 blockDim.x - 1 entries
                waits = true;
            }
        }
        // The tile's entries are counted by the barrier itself: `queued`, read behind it, could already hold what a
        // faster warp added for the next tile, and the warps would part at the barriers below.
        held += __syncthreads_count(waits);
        if (held >= threads) {
            held -= threads;
            finish(queue[held + threadIdx.x]);
            __syncthreads();
            const int sn = n_slow;  // the same in every thread
            if (sn >= threads)
                table_path(T, T32, besp, chi_in, r_in, s_in, slow[sn - threads + threadIdx.x], out4, ln_up_only, true);
            __syncthreads();
            if (threadIdx.x == 0) {
                queued = held;
                if (sn >= threads) n_slow = sn - threads;
            }
            __syncthreads();
        }
    }
    if ((int)threadIdx.x < held) finish(queue[threadIdx.x]);  // (written before the loop's last barrier)
    __syncthreads();
    for (int k = threadIdx.x; k < n_slow; k += threads)
        table_path(T, T32, besp, chi_in, r_in, s_in, slow[k], out4, ln_up_only, true);
    nf = __reduce_add_sync(0xffffffffu, nf);
    if ((threadIdx.x & 31) == 0 && n_fallback && nf) atomicAdd(n_fallback, (unsigned long long)nf);
}

// The method the network would replace, as the step's event pass runs it (Sec. 5.1): the spin branch
// taken with probability W_down (1 - s)/(2 W_s), the uniform rescaled within the chosen branch (the pair
// gives the mixture w(lambda; s) exactly, reading C4), one row of that branch's ICDF in float-float
// (nlc_up_ff, the FP64 row where u' leaves the float range), and xi3 at the sampled u' from the float
// Bessel table.  out4 = (ln u', 0, 0, xi3).
__global__ void branch_table_kernel(TabP<float> T, TabP<double> T64, const float* __restrict__ bes32,
                                    const double* __restrict__ chi_in, const double* __restrict__ r_in,
                                    const double* __restrict__ s_in, int64_t n, float* __restrict__ out4) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float chi = (float)chi_in[i], s = (float)s_in[i];
        const double r = r_in[i];
        const float lnchi = logf(chi);
        float Iu, Id;
        nlc_rates(T, chi, lnchi, Iu, Id);
        const double wd = (double)Id * (1.0 - s) * 0.5, wu = (double)Iu * (1.0 + s) * 0.5;
        const double pd = wd / (wu + wd);
        const bool down = r < pd;
        double rr = down ? r / pd : (r - pd) / (1.0 - pd);
        rr = fmin(fmax(rr, 0x1.0p-53), 1.0 - 0x1.0p-53);
        uint64_t m = (uint64_t)(rr * 0x1.0p52);
        if (m > (1ull << 52) - 1ull) m = (1ull << 52) - 1ull;
        const uint32_t whi = (uint32_t)(m >> 32) << 12, wlo = (uint32_t)m;
        float up;
        if (!nlc_up_ff(T, down ? 1 : 0, lnchi, whi, wlo, up)) {
            const double u = uniform52(whi, wlo);
            up = (float)exp(icdf_lookup(T64, false, down ? 1 : 0, (double)lnchi, log(u) - log(1.0 - u)));
        }
        const float den = fmaf(3.0f * chi, up, 2.0f), lam = 3.0f * chi * up / den, one_m = 2.0f / den;
        float b[3];
        bessel32(bes32, up, b);
        const float u = lam / one_m, kappa = 1.0f / one_m + one_m;
        out4[4 * i] = logf(up);
        out4[4 * i + 1] = 0.0f;
        out4[4 * i + 2] = 0.0f;
        out4[4 * i + 3] = (b[1] + u * s * b[0]) / (-b[2] + kappa * b[1] + lam * s * b[0]);
    }
}

}  // namespace qed

// ---- host side -------------------------------------------------------------------------------------
using namespace qed;

constexpr uint32_t kMlpMagic = 0x514D4C50u;  // "QMLP"

struct qed_mlp_s {
    uint32_t magic;
    int64_t max_batch;
    float *P, *M, *V, *G;  // parameters, Adam moments, gradients
    float *X, *T;          // training samples of several steps (sample_room of them)
    int64_t sample_room;
    int64_t steps;  // AdamW steps taken
};

static bool valid_mlp(const qed_mlp_s* m) { return m && m->magic == kMlpMagic; }

static int grid_for(int64_t work, int threads) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((work + threads - 1) / threads, 152 * 16));
}

// Samples generated ahead per launch of the training loop.  A batch of 4096 is 128 warps on 608 schedulers, each a
// chain of ~12000 FP64 instructions (0.4 ms however few they are); 65536 samples fill the FP64 pipes (1.36 ms, 0.085
// a batch).
constexpr int64_t kTargetsAhead = 65536;

extern "C" void qed_mlp_destroy(qed_mlp_t m) {
    if (!valid_mlp(m)) return;
    for (float* p : {m->P, m->M, m->V, m->G, m->X, m->T}) cudaFree(p);
    m->magic = 0;
    delete m;
}

extern "C" qed_status qed_mlp_create(int64_t max_batch, const float* init_params, qed_mlp_t* out) {
    if (!out || max_batch < 1 || max_batch > (1ll << 26) || !init_params) return QED_ERR_ARG;
    *out = nullptr;
    qed_mlp_s* m = new qed_mlp_s();
    m->magic = kMlpMagic;
    m->max_batch = max_batch;
    m->sample_room = std::max(max_batch, kTargetsAhead);
    const size_t np = sizeof(float) * kParams, ns = (size_t)m->sample_room;
    const bool ok = cudaMalloc(&m->P, np) == cudaSuccess && cudaMalloc(&m->M, np) == cudaSuccess &&
              cudaMalloc(&m->V, np) == cudaSuccess && cudaMalloc(&m->G, np) == cudaSuccess &&
              cudaMalloc(&m->X, 3 * ns * 4) == cudaSuccess && cudaMalloc(&m->T, 4 * ns * 4) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        qed_mlp_destroy(m);
        return QED_ERR_NOMEM;
    }
    if (cudaMemcpy(m->P, init_params, np, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->M, 0, np) != cudaSuccess || cudaMemset(m->V, 0, np) != cudaSuccess) {
        qed_mlp_destroy(m);
        return QED_ERR_CUDA;
    }
    *out = m;
    return QED_OK;
}

extern "C" qed_status qed_mlp_get_params(qed_mlp_t m, float* host_out) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (!host_out) return QED_ERR_ARG;
    return cudaMemcpy(host_out, m->P, sizeof(float) * kParams, cudaMemcpyDeviceToHost) == cudaSuccess ? QED_OK
                                                                                                    : QED_ERR_CUDA;
}

extern "C" qed_status qed_mlp_set_params(qed_mlp_t m, const float* host_in) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (!host_in) return QED_ERR_ARG;
    if (cudaMemcpy(m->P, host_in, sizeof(float) * kParams, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->M, 0, sizeof(float) * kParams) != cudaSuccess ||
        cudaMemset(m->V, 0, sizeof(float) * kParams) != cudaSuccess)
        return QED_ERR_CUDA;
    m->steps = 0;
    return QED_OK;
}

extern "C" qed_status qed_mlp_targets(qed_tables_t t, int64_t n, uint64_t seed, int64_t first_index, float* x_dev,
                                      float* y_dev, double* raw_dev, void* stream) {
    if (!valid_tables(t)) return QED_ERR_STATE;
    if (n < 0 || first_index < 0 || (n > 0 && (!x_dev || !y_dev))) return QED_ERR_ARG;
    if (n == 0) return QED_OK;
    mlp_targets_kernel<<<grid_for(n, 128), 128, 0, (cudaStream_t)stream>>>(tab_params<double>(t), t->bes64, n, seed,
                                                                         first_index, x_dev, y_dev, raw_dev);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

// forward and backward of one batch (features x, targets y), added to grad (kParams floats) and loss
static qed_status mlp_grad_launch(qed_mlp_s* m, const float* x, const float* y, int64_t n, float* grad, float* loss,
                                  cudaStream_t st) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainShared)) !=
        cudaSuccess)
        return QED_ERR_CUDA;
    const int64_t tiles = (n + kTR - 1) / kTR;
    cudaLaunchConfig_t launch = {};
    launch.gridDim = dim3((unsigned)std::min<int64_t>(tiles, sms));
    launch.blockDim = dim3(kTrainThreads);
    launch.dynamicSmemBytes = sizeof(TrainShared);
    launch.stream = st;
    cudaLaunchAttribute cluster = {};
    if (tiles > 1 && tiles <= kTrainCluster) {  // one cluster (of a power of two blocks; one without a tile adds zeros)
        unsigned blocks = 1;
        while (blocks < tiles) blocks *= 2;
        launch.gridDim.x = blocks;
        cluster.id = cudaLaunchAttributeClusterDimension;
        cluster.val.clusterDim.x = blocks;
        cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
        launch.attrs = &cluster;
        launch.numAttrs = 1;
    }
    if (cudaLaunchKernelEx(&launch, mlp_train_kernel, (const float*)m->P, x, y, n, grad, loss) != cudaSuccess) {
        cudaGetLastError();
        return QED_ERR_CUDA;
    }
    return QED_OK;
}

extern "C" qed_status qed_mlp_grad(qed_mlp_t m, const float* x_dev, const float* y_dev, int64_t n, float* grad_dev,
                                   float* loss_dev, void* stream) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (n < 1 || n > m->max_batch || !x_dev || !y_dev || !grad_dev) return QED_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    cudaMemsetAsync(grad_dev, 0, sizeof(float) * kParams, st);
    if (loss_dev) cudaMemsetAsync(loss_dev, 0, sizeof(float), st);
    const qed_status s = mlp_grad_launch(m, x_dev, y_dev, n, grad_dev, loss_dev, st);
    if (s != QED_OK) return s;
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

static void adamw_launch(qed_mlp_s* m, const float* grad, float lr, float weight_decay, float* zero, cudaStream_t st) {
    m->steps += 1;
    const float b1t = (float)std::pow(0.9, (double)m->steps), b2t = (float)std::pow(0.999, (double)m->steps);
    mlp_adamw_kernel<<<(kParams + 255) / 256, 256, 0, st>>>(m->P, m->M, m->V, grad, lr, weight_decay, b1t, b2t, zero);
}

extern "C" qed_status qed_mlp_adamw(qed_mlp_t m, const float* grad_dev, float lr, float weight_decay, void* stream) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (!grad_dev || !(lr >= 0.0f) || !(weight_decay >= 0.0f)) return QED_ERR_ARG;
    adamw_launch(m, grad_dev, lr, weight_decay, nullptr, (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

extern "C" qed_status qed_mlp_train(qed_mlp_t m, qed_tables_t t, int64_t steps, int64_t batch, uint64_t seed,
                                    int64_t first_index, float lr, float lr_final, float weight_decay,
                                    float* loss_per_step_dev, void* stream) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (!valid_tables(t)) return QED_ERR_STATE;
    if (steps < 0 || batch < 1 || batch > m->max_batch || first_index < 0 || !(lr >= 0.0f) || !(lr_final >= 0.0f))
        return QED_ERR_ARG;
    if (!(weight_decay >= 0.0f) && steps > 0) return QED_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t ahead = m->sample_room / batch;  // whole batches generated per launch
    cudaMemsetAsync(m->G, 0, sizeof(float) * kParams, st);
    if (loss_per_step_dev) cudaMemsetAsync(loss_per_step_dev, 0, sizeof(float) * (size_t)steps, st);
    for (int64_t k = 0; k < steps; ++k) {
        // cosine decay from lr to lr_final
        const double c = steps > 1 ? 0.5 * (1.0 + std::cos(3.141592653589793 * (double)k / (double)(steps - 1))) : 1.0;
        const float lrk = (float)(lr_final + (lr - lr_final) * c);
        const int64_t at = k % ahead;
        if (at == 0) {
            const qed_status s = qed_mlp_targets(t, std::min(ahead, steps - k) * batch, seed, first_index + k * batch, m->X,
                                                 m->T, nullptr, stream);
            if (s != QED_OK) return s;
        }
        const qed_status s = mlp_grad_launch(m, m->X + 3 * at * batch, m->T + 4 * at * batch, batch, m->G,
                                             loss_per_step_dev ? loss_per_step_dev + k : nullptr, st);
        if (s != QED_OK) return s;
        adamw_launch(m, m->G, lrk, weight_decay, m->G, st);
    }
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

// persistent grid for the tensor-core kernels: one resident wave of 128-thread blocks
static int tc_blocks(int64_t n) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + kTR - 1) / kTR, (int64_t)sms * kTcPerSm));
}

extern "C" qed_status qed_mlp_forward(qed_mlp_t m, const float* x_dev, int64_t n, float* out_dev, void* stream) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (n < 0 || (n > 0 && (!x_dev || !out_dev))) return QED_ERR_ARG;
    if (n == 0) return QED_OK;
    mlp_forward_kernel<<<tc_blocks(n), kTR, 0, (cudaStream_t)stream>>>(m->P, x_dev, n,
                                                                                                   out_dev);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

// network (unless flags bit 0) and check of the first min(n, *n_dev) samples; grid: the network kernel's
static qed_status mlp_sample_launch(qed_mlp_t m, const qed_tables_s* t, const double* chi, const double* r, const double* s,
                                    int64_t n, const unsigned long long* n_dev, double tol, int flags, float* out4,
                                    uint8_t* fell_back, float* err_out, unsigned long long* n_fallback, int grid,
                                    cudaStream_t st) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr size_t kPerThread = 2 * (sizeof(CheckItem) + sizeof(int64_t));
    if (cudaFuncSetAttribute(mlp_check_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kCheckThreads * kPerThread)) != cudaSuccess)
        return QED_ERR_CUDA;
    if (!(flags & QED_MLP_ALWAYS_TABLE))
        mlp_net_kernel<<<grid, kTR, 0, st>>>(m->P, chi, r, s, n, out4, n_dev);
    const int blocks = (int)std::min<int64_t>((n + 31) / 32, sms);
    const int threads = n <= (int64_t)kCheckFew * sms ? kCheckFew : kCheckThreads;
    mlp_check_kernel<<<blocks, threads, threads * kPerThread, st>>>(tab_params<double>(t), tab_params<float>(t), t->bes32,
                                                                    t->besp, chi, r, s, n, tol, flags, out4, fell_back,
                                                                    err_out, n_fallback, n_dev);
    return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
}

extern "C" qed_status qed_mlp_sample(qed_mlp_t m, qed_tables_t t, const double* chi, const double* r, const double* s,
                                     int64_t n, double tol, int32_t flags, float* out4, uint8_t* fell_back,
                                     float* err_out, unsigned long long* n_fallback, void* stream) {
    if (!valid_mlp(m)) return QED_ERR_STATE;
    if (!valid_tables(t)) return QED_ERR_STATE;
    if (n < 0 || (n > 0 && (!chi || !r || !s || !out4)) || !(tol >= 0.0) ||
        (flags & ~(QED_MLP_ALWAYS_TABLE | QED_MLP_BRANCH_TABLE)))
        return QED_ERR_ARG;
    if (n == 0) return QED_OK;
    if (flags & QED_MLP_BRANCH_TABLE) {
        const int threads = 256;
        const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 152 * 16);
        branch_table_kernel<<<blocks, threads, 0, (cudaStream_t)stream>>>(tab_params<float>(t), tab_params<double>(t),
                                                                          t->bes32, chi, r, s, n, out4);
        return cudaGetLastError() == cudaSuccess ? QED_OK : QED_ERR_CUDA;
    }
    return mlp_sample_launch(m, t, chi, r, s, n, nullptr, tol, flags, out4, fell_back, err_out, n_fallback, tc_blocks(n),
                             (cudaStream_t)stream);
}

// ---- the sampler inside the batched step (qed_batch.cu) ------------------------------------------------

bool mlp_valid(qed_mlp_t m) { return valid_mlp(m); }

int mlp_listed_grid(int64_t n_max) { return tc_blocks(n_max); }

qed_status mlp_sample_listed(qed_mlp_t m, const qed_tables_s* t, const double* chi, const double* r, const double* s,
                             int64_t n_max, const unsigned long long* n_dev, double tol, float* out4,
                             unsigned long long* n_fallback, int grid, cudaStream_t st) {
    return mlp_sample_launch(m, t, chi, r, s, n_max, n_dev, tol, kLnUpOnly, out4, nullptr, nullptr, n_fallback, grid, st);
}
