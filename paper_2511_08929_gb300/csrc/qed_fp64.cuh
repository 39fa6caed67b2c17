// qed_fp64.cuh -- the FP64 arithmetic of the step kernels: the plain FP64 path (qed_step64.cu) and the events of the
// FP32 path that are taken in FP64 (qed_step32.cuh).
//
// On this GPU an FP64 instruction of a warp holds its scheduler's FP64 pipe for 64 cycles, however many of its lanes
// are active and however independent it is of the one before (measured), so the number of FP64 instructions is the
// cost of every path here.  An IEEE division is ~9 of them, a square root ~8, a reciprocal or reciprocal root ~7, a
// logarithm ~25, an exponential or one of sine and cosine ~18.  Hence: one reciprocal root serves a length, its inverse
// and a direction; quotients that share a denominator take one reciprocal; quantities with a closed form in u' carry no
// division (u = lambda/(1 - lambda) = 3 chi u'/2 for emission, 1/(lambda (1 - lambda)) = 3 chi u~'/2 for pairs); the
// fields of a plane wave carry no products by their zero components; the Bessel functions are polynomials on
// intervals found from the argument's bits (no logarithm).
#pragma once
#include "qed_bessel.cuh"

namespace qed {

using V64 = V3<double>;

// --------------------------------------------------------------------------------------------
// Bessel functions of the steps: e^x (K_1/3, K_2/3, int K_1/3) as polynomials of degree 8 on 16 intervals per octave
// of x in [2^-67, 2^15): 25 FP64 instructions against ~95 for the 8-point Lagrange rule on the grid in ln x.  The
// functions' only singularity is x = 0, 33 half-widths from an interval's centre, so degree 8 leaves 66^-9 ~ 4e-17 of
// relative error beside the nodes' own rounding.
// --------------------------------------------------------------------------------------------
constexpr int kBpDeg = 8;
constexpr int kBpRow = 3 * (kBpDeg + 1);
constexpr int kBpSub = 16;                    // intervals per octave
constexpr int kBpLoExp = -67, kBpHiExp = 15;  // octaves [2^-67, 2^15)
constexpr int kBpN = (kBpHiExp - kBpLoExp) * kBpSub;

static __device__ __noinline__ void bessel_outside(double x, double out[3]) {
    if (x < 1.0) bessel_series<double>(x, out);
    else bessel_trapezoid(x, out);
}

// tab: [kBpN][3][kBpDeg + 1], lowest power first, in t in [-1, 1) across the interval
__device__ __forceinline__ void bessel_poly(const double* __restrict__ tab, double x, double out[3]) {
    const int hi = __double2hiint(x);
    const int i = (hi >> 16) - ((1023 + kBpLoExp) << 4);
    if (i < 0 || i >= kBpN) {
        bessel_outside(x, out);
        return;
    }
    const double m = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, __double2loint(x));  // x's mantissa in [1, 2)
    const double c = __hiloint2double((hi & 0x000F0000) | 0x3FF08000, 0);                  // the interval's centre
    const double t = (m - c) * 32.0;
    const double* r = tab + (size_t)i * kBpRow;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        double v = r[f * (kBpDeg + 1) + kBpDeg];
#pragma unroll
        for (int k = kBpDeg - 1; k >= 0; --k) v = fma(v, t, r[f * (kBpDeg + 1) + k]);
        out[f] = v;
    }
}

// ln of the sampled variable for chi and the logit y (the interpolation of icdf_lookup, with d3/6 as a product)
__device__ __forceinline__ double icdf_row64(const double* __restrict__ row, const TabP<double>& T, double slope, double y) {
    const double y0 = T.y_lo * T.inv_dy;
    const double tt = fma(y, T.inv_dy, -y0);
    if (!(tt > 0.0)) return fma(slope, y - T.y_lo, row[0]);
    if (tt >= (double)(T.n_r - 1)) return row[T.n_r - 1];
    int m = (int)tt;
    if (m < 1) m = 1;
    if (m > T.n_r - 3) m = T.n_r - 3;
    const double x = fma(y, T.inv_dy, -y0 - (double)m);  // keeps the precision of y
    const double a = row[m - 1], b = row[m], c = row[m + 1], d = row[m + 2];
    const double d1 = c - b;
    const double d2 = 0.5 * ((a - b) + d1);
    const double d3 = fma(-3.0, d1, d - a) * (1.0 / 6.0);
    return fma(x, fma(x - 1.0, fma(x + 1.0, d3, d2), d1), b);
}

__device__ __forceinline__ double icdf_lookup64(const TabP<double>& T, bool nbw, int s, double lnchi, double y) {
    const double* base = (nbw ? T.nbw_icdf : T.nlc_icdf) + (size_t)s * T.n_chi * T.n_r;
    int i;
    double f;
    chi_coord(T, lnchi, i, f);
    const double slope = nbw ? 2.0 : 3.0;
    const double v0 = icdf_row64(base + (size_t)i * T.n_r, T, slope, y);
    const double v1 = icdf_row64(base + (size_t)(i + 1) * T.n_r, T, slope, y);
    return fma(f, v1 - v0, v0);
}

// --------------------------------------------------------------------------------------------
// fields and pushers
// --------------------------------------------------------------------------------------------
// a plane wave along +z (the linear and circular lasers) at x: E = (ex, ey, 0), B = z x E = (-ey, ex, 0), |E|
struct Wave64 {
    double ex, ey, mag;
};

__device__ __forceinline__ bool plane_wave(int kind) { return kind == QED_FIELD_LP || kind == QED_FIELD_CP; }

__device__ __forceinline__ Wave64 wave64(const FieldP<double>& f, double ph, double z) {
    const double phi = ph - z;
    Wave64 w{0.0, 0.0, 0.0};
    if (phi < 0.0 || phi > f.phimax) return w;
    const double se = sin(phi * f.inv2n);
    const double a = f.a0 * se * se;
    if (f.kind == QED_FIELD_LP) {
        w.ex = a * cos(phi);
        w.mag = fabs(w.ex);
    } else {
        double s, c;
        sincos(phi, &s, &c);
        w.ex = a * c;
        w.ey = a * s;
        w.mag = fabs(a);
    }
    return w;
}

// the Boris push in such a wave: the rotation of p- by t = (q dt/2) B/gamma- in closed form,
// p+ = c p- + s (p- x t) + s (t.p-) t with s = 2/(1 + t^2), c = s - 1
__device__ __forceinline__ V64 boris_w64(const V64& p, const Wave64& w, double q, double dt) {
    const double h = 0.5 * q * dt;
    const V64 pm{fma(h, w.ex, p.x), fma(h, w.ey, p.y), p.z};
    const double hi = h * rsqrt(1.0 + dot(pm, pm));
    const double tx = -hi * w.ey, ty = hi * w.ex;
    const double sf = 2.0 * (1.0 / fma(tx, tx, fma(ty, ty, 1.0)));
    const double c = sf - 1.0, stp = sf * fma(tx, pm.x, ty * pm.y), sz = sf * pm.z;
    return V64{fma(h, w.ex, fma(c, pm.x, fma(stp, tx, -sz * ty))), fma(h, w.ey, fma(c, pm.y, fma(stp, ty, sz * tx))),
               fma(c, pm.z, sf * fma(pm.x, ty, -pm.y * tx))};
}

__device__ __forceinline__ V64 tbmt_w64(const V64& pb, const Wave64& w, double q, bool paper_form, double ae) {
    const double g2 = 1.0 + dot(pb, pb);
    const double ig = rsqrt(g2), gb = g2 * ig;
    const V64 v = ig * pb;
    const double vB = fma(v.y, w.ex, -v.x * w.ey);
    const double xEx = -v.z * w.ey, xEy = v.z * w.ex, xEz = fma(v.x, w.ey, -v.y * w.ex);  // v x E
    const double r1 = 1.0 / (gb + 1.0);
    const double c1 = ae + ig, m = -(ae * gb * r1 * vB), c3 = paper_form ? c1 : ae + r1;
    return V64{-q * fma(m, v.x, fma(-c3, xEx, -c1 * w.ey)), -q * fma(m, v.y, fma(-c3, xEy, c1 * w.ex)),
               -q * fma(m, v.z, -c3 * xEz)};
}

// rotate s about Omega by |Omega| dt: s + A (Omega x s) + C Omega x (Omega x s), A = sin(th)/|Omega|,
// C = (1 - cos th)/|Omega|^2; for th < 1/4 (a step of a beam in a pulse turns by ~0.03) from their Taylor series in
// th^2, to th^12 (the next term is below 1e-20), without the root and the sine and cosine
__device__ __forceinline__ V64 rotate64(const V64& s, const V64& Om, double dt) {
    const double t2 = dot(Om, Om) * (dt * dt);
    if (!(t2 > 0.0)) return s;
    if (t2 > 0.0625) return rotate(s, Om, dt);
    const double A = dt * fma(t2, fma(t2, fma(t2, fma(t2, fma(t2, fma(t2, 1.0 / 6227020800.0, -1.0 / 39916800.0),
                                                              1.0 / 362880.0), -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
    const double C = dt * dt * fma(t2, fma(t2, fma(t2, fma(t2, fma(t2, fma(t2, 1.0 / 87178291200.0, -1.0 / 479001600.0),
                                                                   1.0 / 3628800.0), -1.0 / 40320.0), 1.0 / 720.0), -1.0 / 24.0), 0.5);
    const V64 c = cross(Om, s);
    return axpy(C, cross(Om, c), axpy(A, c, s));
}

// --------------------------------------------------------------------------------------------
// the classical part of a lepton's step
// --------------------------------------------------------------------------------------------
struct Lep64 {
    V64 x, p, s, E, B, khat, eps, beta;
    double gam, ig, chi;
    bool ok;  // chi and the basis are defined and chi is not below the floor
};

template <bool PW>
__device__ __forceinline__ void lepton_classical64(uint32_t fl, const TabP<double>& T, const FieldP<double>& F, double ph,
                                                   double dt, double chi_floor, double q, const V64& x, const V64& p0,
                                                   const V64& s0, Lep64& st) {
    Wave64 w{0.0, 0.0, 0.0};
    if (PW) {
        w = wave64(F, ph, x.z);
        st.E = V64{w.ex, w.ey, 0.0};
        st.B = V64{-w.ey, w.ex, 0.0};
    } else {
        field_eval(F, ph, 0.0, x, st.E, st.B);
    }
    st.p = p0;
    st.s = s0;
    if (fl & QED_F_PUSH) st.p = PW ? boris_w64(p0, w, q, dt) : boris(p0, st.E, st.B, q, dt);
    if (fl & QED_F_TBMT) {
        const V64 pb = 0.5 * (p0 + st.p);
        const bool paper = (fl & QED_F_TBMT_PAPER) != 0;
        const double ae = tbmt_a(fl, T, F.eta0, pb, st.E, st.B);
        st.s = rotate64(s0, PW ? tbmt_w64(pb, w, q, paper, ae) : tbmt_omega(pb, st.E, st.B, q, paper, ae), dt);
    }
    const double p2 = dot(st.p, st.p), g2 = 1.0 + p2;
    st.ig = rsqrt(g2);
    st.gam = g2 * st.ig;
    st.x = (fl & QED_F_MOVE) ? axpy(dt * st.ig, st.p, x) : x;
    st.chi = 0.0;
    st.ok = false;
    st.khat = st.eps = st.beta = V64{0.0, 0.0, 0.0};
    if (!(fl & QED_F_EMIT) || !(p2 > 0.0)) return;
    const double ipn = rsqrt(p2);
    st.khat = ipn * st.p;
    V64 f;  // E + v x B
    if (PW) {
        // e - p_z without cancellation for a particle moving with the wave
        const double em = st.p.z > 0.0 ? fma(st.p.x, st.p.x, fma(st.p.y, st.p.y, 1.0)) / (st.gam + st.p.z) : st.gam - st.p.z;
        st.chi = F.eta0 * em * w.mag;
        const double g = em * st.ig;
        f = V64{g * w.ex, g * w.ey, st.ig * fma(st.p.x, w.ex, st.p.y * w.ey)};
    } else {
        st.chi = chi_of(F.eta0, st.gam, st.p, st.E, st.B);
        f = axpy(st.ig, cross(st.p, st.B), st.E);
    }
    if (!(st.chi >= chi_floor) || !(st.chi > 0.0)) return;
    const V64 fp = axpy(-dot(f, st.khat), st.khat, f);
    const double n2 = dot(fp, fp);
    if (!(n2 > 0.0)) return;
    st.eps = (-q * rsqrt(n2)) * fp;
    st.beta = cross(st.khat, st.eps);
    st.ok = true;
}

// --------------------------------------------------------------------------------------------
// emission (App. A.1) with u = lambda/(1 - lambda) and kappa = 1/(1 - lambda) + 1 - lambda at hand
// --------------------------------------------------------------------------------------------
__device__ __forceinline__ V64 stokes_to_P64(const double xi[3], const V64& eps, const V64& beta, const V64& k) {
    const double l2 = fma(xi[0], xi[0], xi[2] * xi[2]);
    if (!(l2 > 0.0)) return xi[1] * k;
    const double l = l2 * rsqrt(l2);
    const bool up = xi[2] >= 0.0;  // cos dth is the larger component
    const double q = 0.5 * l * (l + fabs(xi[2]));
    double ib = rsqrt(q);
    if (!up && xi[0] < 0.0) ib = -ib;
    const double big = q * ib, small = 0.5 * l * xi[0] * ib;
    return axpy(up ? small : big, beta, axpy(up ? big : small, eps, xi[1] * k));
}

// The outcome of an emission of energy fraction lam at u' (up): final spin sf and the photon's Stokes vector xi.
// si: the initial spin (zero without QED_F_RESOLVED); s_keep: the spin kept when spin events are off.
__device__ __forceinline__ void nlc_event64(uint32_t fl, const double* __restrict__ besp, double up, double lam, double u,
                                            double kappa, double kappat, const Lep64& st, const V64& si, double r3, double r4,
                                            V64& sf, double xi[3]) {
    sf = st.s;
    xi[0] = xi[1] = xi[2] = 0.0;
    if (!(fl & (QED_F_SPIN_EVENT | QED_F_POL_EVENT))) return;
    double b[3];
    bessel_poly(besp, up, b);
    const double K13 = b[0], K23 = b[1], IK = b[2];
    const double sib = dot(si, st.beta), sik = dot(si, st.khat);
    const double wv = fma(lam * K13, sib, fma(kappa, K23, -IK));
    // g = u K13 beta + (2 K23 - IK) s_i + lambda u (K23 - IK)(s_i.k) k
    const V64 g = axpy(u * K13, st.beta, axpy(fma(2.0, K23, -IK), si, (lam * u * (K23 - IK) * sik) * st.khat));
    V64 sfu{0, 0, 0};
    if (fl & QED_F_SPIN_EVENT) {
        const double g2 = dot(g, g);
        if (fl & QED_F_BETA_BASIS) {  // resolved along +-beta (Sec. 8.3 comparison)
            const double gb = dot(g, st.beta);
            sf = (fl & QED_F_SPIN_COLLAPSE) ? (2.0 * wv * r3 < wv - gb ? -1.0 : 1.0) * st.beta : (gb / wv) * st.beta;
        } else if (fl & QED_F_SPIN_COLLAPSE) {
            const double ig = g2 > 0.0 ? rsqrt(g2) : 0.0;
            sf = (2.0 * wv * r3 < wv - g2 * ig ? -ig : ig) * g;
        } else {
            sf = (1.0 / wv) * g;
        }
        sfu = sf;
    }
    if (fl & QED_F_POL_EVENT) {
        const double sie = dot(si, st.eps), sfe = dot(sfu, st.eps), sfb = dot(sfu, st.beta), sfk = dot(sfu, st.khat);
        const V64 x = cross(sfu, si);
        const double lu2 = 0.5 * lam * u;
        const double F0 = wv + dot(sfu, g);
        const double F1 = fma(-K13, fma(u, sie, lam * sfe),
                              fma(-lu2 * IK, fma(sfe, sib, sfb * sie), 0.5 * kappat * K23 * dot(x, st.khat)));
        const double F2 = fma(0.5 * kappat * K13, dot(x, st.eps), lu2 * K13 * fma(sfk, sib, sfb * sik)) -
                          fma(lam * IK - kappat * K23, sik, (u * IK - kappat * K23) * sfk);
        const double F3 = K23 + fma(fma(u, sib, lam * sfb), K13, -lu2 * IK * fma(sfe, sie, -sfb * sib)) +
                          fma(0.5 * kappa * K23, dot(sfu, si), -lu2 * K23 * sfk * sik);
        const double n2 = fma(F1, F1, fma(F2, F2, F3 * F3));
        double f;
        if (fl & QED_F_POL_COLLAPSE) {
            f = n2 > 0.0 ? rsqrt(n2) : 0.0;
            if (2.0 * F0 * r4 < F0 - n2 * f) f = -f;
        } else {
            f = 1.0 / F0;
        }
        xi[0] = f * F1;
        xi[1] = f * F2;
        xi[2] = f * F3;
    }
}

// --------------------------------------------------------------------------------------------
// pairs (App. A.2) with 1/lambda and 1/(1 - lambda) at hand
// --------------------------------------------------------------------------------------------
// The daughters' spins: the expected ones, or the four correlated states (order --, -+, +-, ++, first sign the
// positron's) along their directions.  The spectrum contracted with xi is bilinear in the two spins,
// G(a Sp, b Se) = A + a P + b Q + a b R, so one evaluation of its four parts serves all states (four evaluations of the
// whole spectrum before).
__device__ __forceinline__ void nbw_event64(uint32_t fl, const double* __restrict__ besp, double ut, double lam, double one_m,
                                            double il, double im, const double xi[3], double r3, const V64& eps,
                                            const V64& beta, const V64& k, V64& se, V64& sp) {
    double b[3];
    bessel_poly(besp, ut, b);
    const double K13 = b[0], K23 = b[1], IK = b[2];
    const double ri = one_m * il, ro = lam * im, rho = ri + ro, rhot = ri - ro;
    const double w0 = fma(rho - xi[2], K23, IK);
    const double lk = fma(rhot, K23, im * IK), lp = fma(-rhot, K23, il * IK);
    const V64 je = axpy(fma(-xi[2], il, im) * K13, beta, axpy(xi[0] * il * K13, eps, (xi[1] * lk) * k));
    const V64 jp = axpy(fma(xi[2], im, -il) * K13, beta, axpy(-xi[0] * im * K13, eps, (xi[1] * lp) * k));
    if (!(fl & QED_F_SPIN_COLLAPSE)) {
        const double iw = 1.0 / w0;
        if (fl & QED_F_BETA_BASIS) {
            se = (iw * dot(je, beta)) * beta;
            sp = (iw * dot(jp, beta)) * beta;
        } else {
            se = iw * je;
            sp = iw * jp;
        }
        return;
    }
    if (fl & QED_F_BETA_BASIS) {  // the G_ab sum to 4 w0 on any axes
        se = sp = beta;
    } else {
        const double e2 = dot(je, je), p2 = dot(jp, jp);
        se = (e2 > 0.0 ? rsqrt(e2) : 0.0) * je;
        sp = (p2 > 0.0 ? rsqrt(p2) : 0.0) * jp;
    }
    const double spe = dot(sp, eps), spb = dot(sp, beta), spk = dot(sp, k);
    const double see = dot(se, eps), seb = dot(se, beta), sek = dot(se, k);
    const V64 pxe = cross(sp, se);
    const double sps = dot(sp, se), kk = spk * sek, hu = 0.5 * (il + im), hr = 0.5 * rhot;
    const double A = w0;
    const double Q = fma(im * seb, K13, fma(xi[0], K13 * il * see, fma(xi[1], lk * sek, -xi[2] * il * seb * K13)));
    const double P = fma(-il * spb, K13, fma(-xi[0], K13 * im * spe, fma(xi[1], lp * spk, xi[2] * im * spb * K13)));
    const double R0 = fma(fma(-2.0, K23, IK), sps, fma(rho, IK - K23, 2.0 * K23) * kk);
    const double R1 = fma(-hu * IK, fma(spe, seb, spb * see), hr * K23 * dot(pxe, k));
    const double R2 = -K13 * fma(hu, dot(pxe, eps), hr * fma(spk, seb, spb * sek));
    const double R3 = fma(-hu * IK, fma(spe, see, -spb * seb), K23 * fma(0.5 * rho, sps, fma(-0.5, rho, 1.0) * kk));
    const double R = fma(xi[0], R1, fma(xi[1], R2, fma(xi[2], R3, R0)));
    const double lim = 4.0 * w0 * r3;
    const double g0 = (A - P) + (R - Q), g1 = g0 + ((A - P) - (R - Q)), g2 = g1 + ((A + P) - (R + Q));
    const int chosen = lim < g0 ? 0 : (lim < g1 ? 1 : (lim < g2 ? 2 : 3));
    if (!(chosen & 2)) sp = -1.0 * sp;
    if (!(chosen & 1)) se = -1.0 * se;
}

}  // namespace qed
