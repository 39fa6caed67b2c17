// qed_step64.cu -- the plain FP64 path: one thread per particle, every operation in double precision.
// Lepton step: Sec. 5.1 (and its flow chart) with the non-emission update of Sec. 6.
// Photon step: Sec. 5.2 (and its flow chart) with the non-pair update of Sec. 6.
//
// Both kernels are bound by the FP64 pipe (64 cycles of its scheduler per warp instruction, see qed_fp64.cuh): what a
// step costs is the FP64 instructions its warps issue.  They are built twice, for a single plane wave (the linear and
// circular lasers, whose chi, basis and push have short forms) and for any field.  Emission is decided by a few lanes
// of nearly every warp, so the lanes that emit hand their state to a queue in shared memory and the emission runs 32
// at a time (in line, 90 % of the warps of a beam in a pulse issued all of it for two or three lanes); a pair is made
// in one warp of a hundred, and stays in line.  Blocks of four warps, one per scheduler, so that a small beam spreads
// over all SMs.  1e4 electrons, 32 steps with their bookkeeping: 3.76 -> 1.98 ms; 1e5 electrons and 1e6 photons, 4 steps:
// 6.37 -> 4.22 ms.
#include "qed_bessel.cuh"
#include "qed_fp64.cuh"
#include "qed_internal.h"
#include "qed_steps.h"

namespace qed {

constexpr int kT64 = 128;  // threads per block
constexpr int kQ64 = 64;   // queued emissions per warp (drained 32 at a time)
// resident blocks per SM = the grid: two or three warps a scheduler keep its FP64 pipe busy, and few warps with many
// tiles each end with few partly filled queues
constexpr int kLepton64PerSm = 2, kPhoton64PerSm = 3;

__device__ __forceinline__ void store_particle64(const PartDev& B, int64_t k, const V64& x, const V64& p, const V64& s,
                                                 double tau, double w, uint64_t id) {
    B.x[k] = x.x; B.y[k] = x.y; B.z[k] = x.z;
    B.px[k] = p.x; B.py[k] = p.y; B.pz[k] = p.z;
    B.sx[k] = s.x; B.sy[k] = s.y; B.sz[k] = s.z;
    B.tau[k] = tau; B.w[k] = w; B.id[k] = id;
}

// a lepton's step: everything but its weight and id
__device__ __forceinline__ void store_lepton64(const PartDev& L, int64_t j, const V64& x, const V64& p, const V64& s,
                                               double tau) {
    L.x[j] = x.x; L.y[j] = x.y; L.z[j] = x.z;
    L.px[j] = p.x; L.py[j] = p.y; L.pz[j] = p.z;
    L.sx[j] = s.x; L.sy[j] = s.y; L.sz[j] = s.z;
    L.tau[j] = tau;
}

__device__ __forceinline__ bool finite3(const V64& a) { return isfinite(a.x) && isfinite(a.y) && isfinite(a.z); }

enum { C_EVENTS, C_STORED, C_DROPPED, C_CLAMPED, C_RENORM, C_BELOW, C_NONFINITE, C_RATE_STEPS, C_BOUND, C_N };

// the row coordinate in ln chi, clamped to the grid
__device__ __forceinline__ void chi_coord64(const TabP<double>& T, double lnchi, int& i, double& f) {
    const double s = fmin(fmax((lnchi - T.lnchi_min) * T.inv_dlnchi, 0.0), (double)(T.n_chi - 1));
    i = min((int)s, T.n_chi - 2);
    f = s - (double)i;
}

// An emitting lepton's state after the classical part of its step, queued per warp.
enum { Q_X, Q_P = 3, Q_S = 6, Q_EPS = 9, Q_IPN = 12, Q_CHI, Q_WS, Q_WDN, Q_TAU, Q_N };
struct Queue64 {
    double v[Q_N][kQ64];
    int64_t j[kQ64];
};

// the emissions of 32 lanes (j < 0: none); warp-collective
__device__ __forceinline__ void emit64(const TabP<double>& T, const double* __restrict__ besp, const StepP& S,
                                       const Queue64& Q, int e, bool have, const PartDev& L, const PartDev& G,
                                       AppendState* A, qed_counters* ctr, unsigned long long* c) {
    const uint32_t fl = S.flags;
    bool want = false;
    Lep64 st;
    V64 k{0, 0, 0}, pf{0, 0, 0}, sf{0, 0, 0}, P{0, 0, 0};
    double tau = 0.0, tau_kept = 0.0, u0a = 0.0;
    uint64_t gid = 0;
    int64_t j = -1;
    if (have) {
        j = Q.j[e];
        st.x = V64{Q.v[Q_X][e], Q.v[Q_X + 1][e], Q.v[Q_X + 2][e]};
        st.p = V64{Q.v[Q_P][e], Q.v[Q_P + 1][e], Q.v[Q_P + 2][e]};
        st.s = V64{Q.v[Q_S][e], Q.v[Q_S + 1][e], Q.v[Q_S + 2][e]};
        st.eps = V64{Q.v[Q_EPS][e], Q.v[Q_EPS + 1][e], Q.v[Q_EPS + 2][e]};
        const double ipn = Q.v[Q_IPN][e], chi = Q.v[Q_CHI][e];
        tau_kept = tau = Q.v[Q_TAU][e];
        st.khat = ipn * st.p;
        st.beta = cross(st.khat, st.eps);
        const uint64_t id = L.id[j];
        const uint4 w0 = draw(id, S.seed, S.step, kSlotTauBranch);
        const uint4 w1 = draw(id, S.seed, S.step, kSlotLambdaSpin);
        const uint4 w2 = draw(id, S.seed, S.step, kSlotStokes);
        const double r3 = uniform52(w1.z, w1.w), r4 = uniform52(w2.x, w2.y);
        u0a = uniform52(w0.x, w0.y);
        double lam, one_m, iom, u, up;  // iom = 1/(1 - lambda), u = lambda/(1 - lambda)
        if (fl & QED_F_REJECT) {        // the accepted candidate lambda = r1^3
            lam = u0a * u0a * u0a;
            one_m = 1.0 - lam;
            iom = 1.0 / one_m;
            u = lam * iom;
            up = u / (1.5 * chi);
        } else {
            const bool down = (fl & QED_F_TAU) ? uniform52(w0.z, w0.w) * Q.v[Q_WS][e] < Q.v[Q_WDN][e]
                                               : u0a < Q.v[Q_WDN][e] * S.dt;
            const double r2 = uniform52(w1.x, w1.y);
            up = exp(icdf_lookup64(T, false, down ? 1 : 0, log(chi), log(r2 / (1.0 - r2))));
            u = 1.5 * chi * up;
            iom = 1.0 + u;
            one_m = 1.0 / iom;
            lam = u * one_m;
        }
        const V64 si = (fl & QED_F_RESOLVED) ? st.s : V64{0.0, 0.0, 0.0};
        double xi[3];
        nlc_event64(fl, besp, up, lam, u, iom + one_m, iom - one_m, st, si, r3, r4, sf, xi);
        k = lam * st.p;
        pf = (fl & QED_F_RECOIL) ? one_m * st.p : st.p;
        P = stokes_to_P64(xi, st.eps, st.beta, st.khat);
        if ((fl & QED_F_TAU) && !(fl & QED_F_REJECT)) tau = -log(u0a);
        if (lam >= S.store_min * ipn) {
            want = true;
            const uint4 wc = draw(id, S.seed, S.step, kSlotChild);
            gid = (uint64_t)wc.x | ((uint64_t)wc.y << 32);
        } else {
            c[C_BELOW]++;
        }
    }
    // the photon's slot: event ev of the call writes base + ev if ev < budget; otherwise the event is not
    // applied (the lepton keeps its pre-event state and its spent optical depth)
    const long long ev = reserve_event(A, want);
    const bool keep = want && A != nullptr && ev < A->budget;
    const bool refused = want && A != nullptr && !keep;
    if (keep) {
        store_particle64(G, A->base[0] + ev, st.x, k, P, birth_tau(gid, S.seed), L.w[j], gid);
        c[C_STORED]++;
    }
    if (refused) {
        c[C_DROPPED]++;
        record_error(ctr, QED_ERR_CAPACITY, j);
    } else if (want && A == nullptr) {
        c[C_DROPPED]++;  // the caller keeps no photons
    }
    if (have) {
        if (!refused) c[C_EVENTS]++;
        store_lepton64(L, j, st.x, refused ? st.p : pf, refused ? st.s : sf, refused ? tau_kept : tau);
    }
}

template <bool PW>
__global__ void __launch_bounds__(kT64, kLepton64PerSm) lepton64_kernel(TabP<double> T, const double* __restrict__ besp, FieldP<double> F,
                                                        StepP S, double q, PartDev L, PartDev G, AppendState* A,
                                                        qed_counters* ctr) {
    __shared__ Queue64 queue[kT64 / 32];
    Queue64& Q = queue[threadIdx.x >> 5];
    const int64_t n = min(L.begin ? *L.begin : *L.count, L.capacity);
    const uint32_t fl = S.flags;
    const double dt = S.dt;
    const bool resolved = (fl & QED_F_RESOLVED) != 0;
    const double pref = kAlpha / (kSqrt3 * kPi * F.eta0);
    unsigned long long c[C_N] = {};
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int qn = 0;  // queued emissions (warp-uniform)
    for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); w0 < n || qn > 0; w0 += stride) {
        const int64_t j = w0 + lane;
        bool event = false;
        Lep64 st;
        double tauf = 0.0, Ws = 0.0, Wdn = 0.0;
        if (j < n) {
            const V64 x{L.x[j], L.y[j], L.z[j]}, p{L.px[j], L.py[j], L.pz[j]}, s{L.sx[j], L.sy[j], L.sz[j]};
            const double tau = L.tau[j];
            if (!(finite3(x) && finite3(p) && finite3(s) && !isnan(tau))) {
                c[C_NONFINITE]++;
                record_error(ctr, QED_ERR_NAN, j);
            } else {
                lepton_classical64<PW>(fl, T, F, S.ph_hi, dt, S.chi_floor, q, x, p, s, st);
                V64 sf = st.s;
                tauf = tau;
                if (st.ok) {
                    const double chi = st.chi;
                    if (chi > T.chi_max) c[C_CLAMPED]++;
                    int i;
                    double f;
                    chi_coord64(T, log(chi), i, f);
                    const double* ru = T.nlc_rate + i;
                    const double* rd = ru + T.n_chi;
                    double Wu = exp(fma(f, ru[1] - ru[0], ru[0])) * (pref * st.ig);
                    double Wd = exp(fma(f, rd[1] - rd[0], rd[0])) * (pref * st.ig);
                    if (chi < T.chi_min) {  // classical: proportional to chi
                        const double sc = chi / T.chi_min;
                        Wu *= sc;
                        Wd *= sc;
                    }
                    const double sb = resolved ? dot(st.s, st.beta) : 0.0;
                    Wdn = 0.5 * Wd * (1.0 - sb);
                    Ws = fma(0.5 * Wu, 1.0 + sb, Wdn);
                    if (fl & QED_F_REJECT) {
                        // table-free (Sec. 4.2): candidate lambda = r1^3, accepted with probability
                        // 3 r1^2 (dW/dlambda) dt, dW/dlambda = pref w(lambda; s.beta) (App. A.1)
                        const uint4 w = draw(L.id[j], S.seed, S.step, kSlotTauBranch);
                        const double r1 = uniform52(w.x, w.y), r2 = uniform52(w.z, w.w);
                        const double lc = r1 * r1 * r1, om = 1.0 - lc;
                        const double rej_up = 2.0 * lc / (3.0 * chi * om);
                        double b[3] = {0.0, 0.0, 0.0};
                        if (rej_up < 700.0) bessel_poly(besp, rej_up, b);  // scaled by e^{u'}; beyond, w ~ 0
                        const double wl = (-b[2] + (1.0 / om + om) * b[1] + lc * sb * b[0]) * exp(-rej_up);
                        const double acc = 3.0 * r1 * r1 * (pref * st.ig) * wl * dt;
                        if (acc > 1.0) c[C_BOUND]++;
                        event = r2 < acc;
                    } else if (fl & QED_F_TAU) {
                        tauf = fma(-Ws, dt, tau);
                        event = tauf <= 0.0;
                    } else {
                        const uint4 w = draw(L.id[j], S.seed, S.step, kSlotTauBranch);
                        event = uniform52(w.x, w.y) < Ws * dt;
                    }
                    if (!event) {
                        if ((fl & QED_F_NONTRANSITION) && resolved) {
                            // Sec. 6: s <- [s (1 - <P> dt) - P_i beta dt] / [1 - (<P> + P_i beta.s) dt]
                            const double W0 = 0.5 * (Wu + Wd), Pi = 0.5 * (Wu - Wd);
                            const double D = fma(-fma(Pi, sb, W0), dt, 1.0);
                            if (D > 0.0) {
                                const double iD = 1.0 / D;
                                sf = axpy(-Pi * dt * iD, st.beta, (fma(-W0, dt, 1.0) * iD) * st.s);
                                const double n2 = dot(sf, sf);
                                if (n2 > 1.0) {
                                    sf = rsqrt(n2) * sf;
                                    c[C_RENORM]++;
                                }
                            }
                        }
                        // the loop's Scorer term (App. A.1): a turn about the rest-frame magnetic field
                        if (fl & QED_F_LOOP)
                            sf = rotate(sf, loop_omega(T, F.eta0, chi, st.gam, st.p, st.E, st.B, q), dt);
                    }
                }
                if (!event) store_lepton64(L, j, st.x, st.p, sf, tauf);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, event);
        if (event) {
            const int e = qn + __popc(m & ((1u << lane) - 1u));
            Q.j[e] = j;
            Q.v[Q_X][e] = st.x.x; Q.v[Q_X + 1][e] = st.x.y; Q.v[Q_X + 2][e] = st.x.z;
            Q.v[Q_P][e] = st.p.x; Q.v[Q_P + 1][e] = st.p.y; Q.v[Q_P + 2][e] = st.p.z;
            Q.v[Q_S][e] = st.s.x; Q.v[Q_S + 1][e] = st.s.y; Q.v[Q_S + 2][e] = st.s.z;
            Q.v[Q_EPS][e] = st.eps.x; Q.v[Q_EPS + 1][e] = st.eps.y; Q.v[Q_EPS + 2][e] = st.eps.z;
            Q.v[Q_IPN][e] = rsqrt(dot(st.p, st.p));
            Q.v[Q_CHI][e] = st.chi;
            Q.v[Q_WS][e] = Ws;
            Q.v[Q_WDN][e] = Wdn;
            Q.v[Q_TAU][e] = tauf;  // spent (optical depth) or unchanged (probability mode)
        }
        qn += __popc(m);
        __syncwarp();
        if (qn >= 32 || (qn > 0 && w0 + stride >= n)) {  // a full set, or what is left after the last tile
            const int cnt = min(qn, 32);
            qn -= cnt;
            emit64(T, besp, S, Q, qn + lane, lane < cnt, L, G, A, ctr, c);
            __syncwarp();
        }
    }
    flush_counters<C_N>(c, &ctr->events);
}

template <bool PW>
__global__ void __launch_bounds__(kT64, kPhoton64PerSm) photon64_kernel(TabP<double> T, const double* __restrict__ besp, FieldP<double> F,
                                                        StepP S, PartDev G, PartDev El, PartDev Po, AppendState* A,
                                                        qed_counters* ctr) {
    const int64_t n = min(G.begin ? *G.begin : *G.count, G.capacity);
    const uint32_t fl = S.flags;
    const double dt = S.dt;
    const bool resolved = (fl & QED_F_RESOLVED) != 0;
    const double pref0 = kAlpha / (kSqrt3 * kPi * F.eta0);
    unsigned long long c[C_N] = {};
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const bool have_daughters = El.count != nullptr && Po.count != nullptr;
    for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); w0 < n; w0 += stride) {
        const int64_t j = w0 + lane;
        bool want = false;
        V64 x{0, 0, 0}, Pf{0, 0, 0}, pe{0, 0, 0}, pp{0, 0, 0}, se{0, 0, 0}, sp{0, 0, 0};
        double tauf = 0.0;
        uint64_t ide = 0, idp = 0;
        bool skip = true;
        if (j < n) {
            x = V64{G.x[j], G.y[j], G.z[j]};
            const V64 k{G.px[j], G.py[j], G.pz[j]}, P{G.sx[j], G.sy[j], G.sz[j]};
            const double tau = G.tau[j];
            if (!(finite3(x) && finite3(k) && finite3(P) && !isnan(tau))) {
                c[C_NONFINITE]++;
                record_error(ctr, QED_ERR_NAN, j);
            } else {
                skip = false;
                Wave64 w{0.0, 0.0, 0.0};
                V64 E{0, 0, 0}, B{0, 0, 0};
                if (PW) w = wave64(F, S.ph_hi, x.z);
                else field_eval(F, S.ph_hi, 0.0, x, E, B);
                const double k2 = dot(k, k), ik = k2 > 0.0 ? rsqrt(k2) : 0.0, en = k2 * ik;
                const V64 khat = ik * k;
                if (fl & QED_F_MOVE) x = axpy(dt, khat, x);
                Pf = P;
                tauf = tau;
                if ((fl & QED_F_EMIT) && en > 0.0) {
                    double chi;
                    V64 f;  // E + khat x B
                    if (PW) {
                        const double em = k.z > 0.0 ? fma(k.x, k.x, k.y * k.y) / (en + k.z) : en - k.z;
                        chi = F.eta0 * em * w.mag;
                        const double g = em * ik;
                        f = V64{g * w.ex, g * w.ey, fma(khat.x, w.ex, khat.y * w.ey)};
                    } else {
                        chi = chi_of(F.eta0, en, k, E, B);
                        f = E + cross(khat, B);
                    }
                    const V64 fp = axpy(-dot(f, khat), khat, f);
                    const double n2 = dot(fp, fp);
                    if (chi >= S.chi_floor && chi > 0.0 && n2 > 0.0) {
                        const V64 eps = rsqrt(n2) * fp, beta = cross(khat, eps);
                        double xi[3] = {0.0, 0.0, 0.0};
                        if (resolved) P_to_stokes(P, eps, beta, khat, xi);
                        if (chi > T.chi_max) c[C_CLAMPED]++;
                        double Wp = 0.0, Wm = 0.0, lnchi = 0.0;
                        const double ichi = 1.0 / chi;
                        if (chi >= T.chi_min) {
                            lnchi = log(chi);
                            int i;
                            double g;
                            chi_coord64(T, lnchi, i, g);
                            const double sub = (8.0 / 3.0) * (chi > T.chi_max ? 1.0 / T.chi_max : ichi);
                            const double* rp = T.nbw_rate + i;
                            const double* rm = rp + T.n_chi;
                            Wp = exp(fma(g, rp[1] - rp[0], rp[0]) - sub) * (pref0 * ik);
                            Wm = exp(fma(g, rm[1] - rm[0], rm[0]) - sub) * (pref0 * ik);
                        }
                        const double Wmp = 0.5 * Wm * (1.0 - xi[2]);
                        const double Wx = fma(0.5 * Wp, 1.0 + xi[2], Wmp);
                        bool event = false, minus = false;
                        double rej_lam = 0.0;
                        const uint64_t id = G.id[j];
                        if (fl & QED_F_REJECT) {
                            // table-free (Sec. 4.2): candidate positron fraction lambda = r1, accepted with
                            // probability (dW/dlambda) dt = pref w0(lambda; xi3) dt (App. A.2)
                            const uint4 wd = draw(id, S.seed, S.step, kSlotTauBranch);
                            const double r1 = uniform52(wd.x, wd.y), r2 = uniform52(wd.z, wd.w);
                            const double om = 1.0 - r1;
                            rej_lam = r1;
                            const double rej_ut = (2.0 / 3.0) * ichi / (r1 * om);
                            double b[3] = {0.0, 0.0, 0.0};
                            if (rej_ut < 700.0) bessel_poly(besp, rej_ut, b);  // scaled by e^{u~'}; beyond, w0 ~ 0
                            const double w0r = (b[2] + (om / r1 + r1 / om) * b[1] - xi[2] * b[1]) * exp(-rej_ut);
                            const double acc = (pref0 * ik) * w0r * dt;
                            if (acc > 1.0) c[C_BOUND]++;
                            event = r2 < acc;
                        } else if (fl & QED_F_TAU) {
                            tauf = fma(-Wx, dt, tau);
                            event = tauf <= 0.0;
                            if (event) {
                                const uint4 wd = draw(id, S.seed, S.step, kSlotTauBranch);
                                minus = uniform52(wd.z, wd.w) * Wx < Wmp;
                            }
                        } else {
                            const uint4 wd = draw(id, S.seed, S.step, kSlotTauBranch);
                            const double r1 = uniform52(wd.x, wd.y);
                            event = r1 < Wx * dt;
                            minus = r1 < Wmp * dt;
                        }
                        if (event && ((fl & QED_F_REJECT) || Wx > 0.0)) {
                            const uint4 w1 = draw(id, S.seed, S.step, kSlotLambdaSpin);
                            const double r = uniform52(w1.x, w1.y), r3 = uniform52(w1.z, w1.w);
                            double ut, lam, one_m, Qv;  // Qv = 1/(lambda (1 - lambda)) = 3 chi u~'/2
                            if (fl & QED_F_REJECT) {
                                lam = rej_lam;
                                one_m = 1.0 - lam;
                                Qv = 1.0 / (lam * one_m);
                                ut = (2.0 / 3.0) * ichi * Qv;
                            } else {
                                const double rf = r < 0.5 ? 1.0 - 2.0 * r : 2.0 * r - 1.0;
                                double xv = 0.0;
                                if (rf > 0.0) xv = exp(icdf_lookup64(T, true, minus ? 1 : 0, lnchi, log(rf / (1.0 - rf))));
                                const double umin = (8.0 / 3.0) * ichi;
                                ut = umin + xv;
                                // mu = (1 - sqrt(x/u~'))/2 without its cancellation near the centre
                                const double iut = 1.0 / ut;
                                const double mu = 0.5 * umin * iut / (1.0 + sqrt(xv * iut));
                                lam = r < 0.5 ? mu : 1.0 - mu;
                                one_m = r < 0.5 ? 1.0 - mu : mu;
                                Qv = 1.5 * chi * ut;
                            }
                            pp = lam * k;
                            pe = one_m * k;
                            if (fl & QED_F_SPIN_EVENT)
                                nbw_event64(fl, besp, ut, lam, one_m, one_m * Qv, lam * Qv, xi, r3, eps, beta, khat, se, sp);
                            const uint4 wc = draw(id, S.seed, S.step, kSlotChild);
                            ide = (uint64_t)wc.x | ((uint64_t)wc.y << 32);
                            idp = (uint64_t)wc.z | ((uint64_t)wc.w << 32);
                            want = true;
                        } else if (!event && (fl & QED_F_NONTRANSITION) && resolved) {
                            const double W0 = 0.5 * (Wp + Wm), Pi = 0.5 * (Wp - Wm);
                            const double D = fma(-fma(Pi, xi[2], W0), dt, 1.0);
                            if (D > 0.0) {
                                const double iD = 1.0 / D, a1 = fma(-W0, dt, 1.0) * iD;
                                double xn[3] = {xi[0] * a1, xi[1] * a1, fma(xi[2], a1, -Pi * dt * iD)};
                                const double n2x = fma(xn[0], xn[0], fma(xn[1], xn[1], xn[2] * xn[2]));
                                if (n2x > 1.0) {
                                    const double in = rsqrt(n2x);
                                    for (int i = 0; i < 3; ++i) xn[i] *= in;
                                    c[C_RENORM]++;
                                }
                                Pf = stokes_to_P64(xn, eps, beta, khat);
                            }
                        }
                    }
                }
            }
        }
        // daughters: one reservation for the pair (electron base[0] + ev, positron base[1] + ev), both or
        // neither
        bool ok = false;
        if (__any_sync(0xffffffffu, want)) {
            if (have_daughters) {
                const long long ev = reserve_event(A, want);
                ok = want && ev < A->budget;
                if (ok) {
                    const double wgt = G.w[j];
                    store_particle64(El, A->base[0] + ev, x, pe, se, birth_tau(ide, S.seed), wgt, ide);
                    store_particle64(Po, A->base[1] + ev, x, pp, sp, birth_tau(idp, S.seed), wgt, idp);
                }
                const long long s_d = reserve_slots(G.n_dead, ok, 1);
                if (ok && s_d < G.capacity) G.dead[s_d] = j;
            }
            if (want) {
                if (ok) {
                    c[C_EVENTS]++;
                    c[C_STORED] += 2;
                } else {
                    c[C_DROPPED]++;
                    if (have_daughters) record_error(ctr, QED_ERR_CAPACITY, j);
                }
            }
        }
        if (j < n && !skip) {
            G.x[j] = x.x; G.y[j] = x.y; G.z[j] = x.z;
            if (ok) {  // converted: inert until compaction
                G.px[j] = 0.0; G.py[j] = 0.0; G.pz[j] = 0.0;
                G.w[j] = 0.0;
            } else {
                G.sx[j] = Pf.x; G.sy[j] = Pf.y; G.sz[j] = Pf.z;
            }
            G.tau[j] = tauf;
        }
    }
    flush_counters<C_N>(c, &ctr->events);
}

}  // namespace qed

void launch_lepton64(const qed_tables_s* t, const qed_field& f, const qed_step_desc& s, const qed_particles* L,
                     const qed_particles* G, qed_counters* ctr, cudaStream_t st) {
    using namespace qed;
    PartDev g{};
    if (G) g = part_dev(G);
    const int blocks = launch_blocks(L->capacity, kT64, kLepton64PerSm);
    // single plane waves take the kernel of their short forms (the general kernel is 7-8 % slower on them: 2.11 against
    // 1.98 ms for 1e4 electrons, 4.60 against 4.22 ms for the coupled species of 1e5)
    auto* kern = f.kind == QED_FIELD_LP || f.kind == QED_FIELD_CP ? lepton64_kernel<true> : lepton64_kernel<false>;
    kern<<<blocks, kT64, 0, st>>>(tab_params<double>(t), t->besp, field_params<double>(f), step_params(s, f), (double)L->charge,
                                  part_dev(L), g, G ? append_state(ctr) : nullptr, ctr);
}

void launch_photon64(const qed_tables_s* t, const qed_field& f, const qed_step_desc& s, const qed_particles* G,
                     const qed_particles* El, const qed_particles* Po, qed_counters* ctr, cudaStream_t st) {
    using namespace qed;
    PartDev e{}, p{};
    if (El && Po) {
        e = part_dev(El);
        p = part_dev(Po);
    }
    const int blocks = launch_blocks(G->capacity, kT64, kPhoton64PerSm);
    auto* kern = f.kind == QED_FIELD_LP || f.kind == QED_FIELD_CP ? photon64_kernel<true> : photon64_kernel<false>;
    kern<<<blocks, kT64, 0, st>>>(tab_params<double>(t), t->besp, field_params<double>(f), step_params(s, f), part_dev(G), e, p,
                                  (El && Po) ? append_state(ctr) : nullptr, ctr);
}
