// Interface constitutive update (Sec. 2.2: the poroelastoplastic interface law with a
// Coulomb yield surface, a tensile cut-off, softening of friction, dilatancy, cohesion
// and tensile strength, damage, opening and contact) integrated by an elastic predictor
// and plastic corrector (Sec. 3.1.1), with the consistent tangent
// C^ep = d(Delta T') / d(Delta delta) of eq. jac_mech.  One thread per collocation point,
// FP64.
//
// The plastic multiplier x is the root of one equation g(x) = 0 per return.  Every
// equation is evaluated with its slope in closed form (two inverse square roots), first in
// FP32 for a guess good to about 1e-6, then in FP64 by Newton's method safeguarded with
// bisection until a step moves x by no more than an ulp.  The tangent is exact within the
// active mode: the derivatives of the return at fixed x and along x in closed form,
// combined by the implicit function theorem, dx/d(dd_j) = -(dg/d(dd_j)) / (dg/dx).
//
// The FP64 pipe of this GPU (1/64 of the FP32 rate) bounds the update, so FP64 operations
// are what counts.  The first form carried dual numbers of one, four and three components
// through every evaluation and iterated until a step vanished: 34,000 instructions a
// Coulomb point, 9.6 ms for 1,000,000 points of a softening joint with the tangent (the
// states move 244 MB: 0.036 ms); see k_iface_return for the present figures.
//
// Branches (the active mode, the maxima of the internal variables) are taken on values,
// so C^ep is the derivative within the active mode.  Two passes: one classifies every
// point and finishes the elastic and open ones, then each kind of return (Coulomb,
// tensile, apex) runs over its own list, so that a warp follows one branch.  The choices the paper leaves open
// are those stated with hm_interface_update in hmat.h.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "common.h"

namespace hm {
namespace {

enum : int32_t { M_ELASTIC = 0, M_COULOMB = 1, M_TENSILE = 2, M_OPEN = 3, M_APEX = 4 };
constexpr int N_MODES = 5;
constexpr int ST_NOROOT = 1;  // a multiplier bracket without a sign change or no convergence

struct Prm {
    double Ks, Kn, fp, fr, psip, dc, cp, sigp, wc, alphaR;
    double iKs, iKn, idc, iwc;  // reciprocals (at most DBL_MAX, so that 0 times one stays 0)
};

// ---------------------------------------------------------------- the law
// v = sqrt(q) and its reciprocal; 0 and 0 for q = 0
__device__ __forceinline__ void root_of(double q, double& v, double& inv) {
    inv = q > 0.0 ? rsqrt(q) : 0.0;
    v = q * inv;
}
__device__ __forceinline__ void root_of(float q, float& v, float& inv) {
    inv = q > 0.f ? rsqrtf(q) : 0.f;
    v = q * inv;
}

// peak W(chi / scale) with W(x) = max(0, 1 - x) (a zero scale is fully softened), and its
// slope in chi
template <class R>
struct Soft {
    R peak, scale, inv;
    __device__ __forceinline__ R operator()(R chi, R& slope) const {
        const R x = chi * inv;
        const bool on = scale > R(0) && !(x >= R(1));
        slope = on ? -peak * inv : R(0);
        return on ? peak * (R(1) - x) : R(0);
    }
    __device__ __forceinline__ R operator()(R chi) const {
        R s;
        return (*this)(chi, s);
    }
};
template <class R>
struct Law {
    R Ks, Kn, fr;
    Soft<R> f, psi, c, st;  // friction above residual, dilatancy, cohesion, tensile strength
    __host__ __device__ __forceinline__ explicit Law(const Prm& P)
        : Ks((R)P.Ks), Kn((R)P.Kn), fr((R)P.fr),
          f{(R)(P.fp - P.fr), (R)P.dc, (R)P.idc}, psi{(R)P.psip, (R)P.dc, (R)P.idc},
          c{(R)P.cp, (R)P.wc, (R)P.iwc}, st{(R)P.sigp, (R)P.wc, (R)P.iwc} {}
};

// state at t^n of one point
struct Pt {
    double T[3], dp[3], chis, chit, wdil;
};

// state at t^(n+1) and C^ep (row-major, row = traction component)
struct Res {
    double T[3], dp[3], chis, chit, wdil;
    double cep[9];
    int32_t mode;
};

// The multiplier equations g(x) = 0 of the returns from the trial traction (t0, t1, tn)
// and the inelastic DD (p0, p1, pn) the return starts from.  eval gives g, its slope in x
// and the quantities the outputs need.
// Coulomb return (flow along s_hat + psi n, shear direction s_hat of the trial kept)
template <class R>
struct CoulombEq {
    R tau, itau, s0, s1, tn, p0, p1, pn, chis, chit;
    struct At {
        R g, gx;
        R a, b, n, cs, ct, psi, f, c, ta, Tn;  // inelastic DD, internal variables, strengths, tractions
        R ics, ict, f1, psi1, c1;           // 1/cs and 1/ct where they grow (else 0); slopes of f, psi, c
    };
    __device__ __forceinline__ At eval(const Law<R>& P, R x) const {
        At o;
        o.a = p0 + x * s0;
        o.b = p1 + x * s1;
        const R q = o.a * o.a + o.b * o.b;
        R v, inv;
        root_of(q, v, inv);
        const bool on = !(chis >= v);
        o.cs = on ? v : chis;
        o.ics = on ? inv : R(0);
        o.psi = P.psi(o.cs, o.psi1);
        o.f = P.f(o.cs, o.f1) + P.fr;
        o.n = pn + x * o.psi;
        root_of(q + o.n * o.n, v, inv);
        const bool ton = !(chit >= v);
        o.ct = ton ? v : chit;
        o.ict = ton ? inv : R(0);
        o.c = P.c(o.ct, o.c1);
        o.ta = tau - P.Ks * x;
        o.Tn = tn - P.Kn * (o.psi * x);
        o.g = o.ta + o.f * o.Tn - o.c;
        o.gx = slope(P, o, x, R(1), o.a * s0 + o.b * s1, -P.Ks, R(0));
        return o;
    }
    // g(0): without slip of its own the point keeps its internal variables, unless the state
    // given breaks chis >= |slip| or chit >= |DD|
    __device__ __forceinline__ R at_zero(const Law<R>& P) const {
        const R q = p0 * p0 + p1 * p1;
        if (!(chis >= R(0) && chit >= R(0) && q <= chis * chis && q + pn * pn <= chit * chit))
            return eval(P, R(0)).g;
        return tau + (P.f(chis) + P.fr) * tn - P.c(chit);
    }
    // directional derivative of g: dx of x, m = a da + b db, dta of tau - Ks x, dtn of tn
    __device__ __forceinline__ R slope(const Law<R>& P, const At& o, R x, R dx, R m, R dta, R dtn) const {
        const R dcs = m * o.ics, dpsi = o.psi1 * dcs;
        const R dn = dx * o.psi + x * dpsi;
        const R dct = (m + o.n * dn) * o.ict;
        return dta + o.f * (dtn - P.Kn * dn) + o.f1 * dcs * o.Tn - o.c1 * dct;
    }
};

// tensile return (flow along n)
template <class R>
struct TensileEq {
    R tn, p0, p1, pn, chit;
    struct At {
        R g, gx, n, ct, ict, Tn;
    };
    __device__ __forceinline__ At eval(const Law<R>& P, R x) const {
        At o;
        o.n = pn + x;
        R v, inv, st1;
        root_of(p0 * p0 + p1 * p1 + o.n * o.n, v, inv);
        const bool ton = !(chit >= v);
        o.ct = ton ? v : chit;
        o.ict = ton ? inv : R(0);
        o.Tn = tn - P.Kn * x;
        o.g = o.Tn - P.st(o.ct, st1);
        o.gx = -P.Kn - st1 * (o.n * o.ict);
        return o;
    }
};

// apex of the Coulomb cone: shear fully inelastic (inelastic DD a, b; friction f there),
// normal increment x
template <class R>
struct ApexEq {
    R tn, a, b, f, pn, chit;
    struct At {
        R g, gx, n, ct, ict, c1, Tn;
    };
    __device__ __forceinline__ At eval(const Law<R>& P, R x) const {
        At o;
        o.n = pn + x;
        R v, inv;
        root_of(a * a + b * b + o.n * o.n, v, inv);
        const bool ton = !(chit >= v);
        o.ct = ton ? v : chit;
        o.ict = ton ? inv : R(0);
        o.Tn = tn - P.Kn * x;
        o.g = f * o.Tn - P.c(o.ct, o.c1);
        o.gx = -f * P.Kn - o.c1 * (o.n * o.ict);
        return o;
    }
};

// A guess of the root in (0, hi): Newton in FP32 kept inside the bracket.  Whatever it
// returns only starts the FP64 iteration.
template <class Eq>
__device__ __forceinline__ float guess_root(const Law<float>& P, const Eq& e, float hi, float x0) {
    float x = x0 > 0.f && x0 < hi ? x0 : 0.5f * hi;
    for (int it = 0; it < 12; ++it) {
        const auto o = e.eval(P, x);
        if (!(o.gx < 0.f)) break;
        float xn = x - o.g / o.gx;
        if (!(xn > 0.f)) xn = 0.5f * x;
        if (!(xn < hi)) xn = 0.5f * (x + hi);
        const float step = fabsf(xn - x);
        x = xn;
        if (step <= 2e-7f * x) break;
    }
    return x;
}

// Root of g on [0, hi] with g0 = g(0) > 0 >= g(hi) (values), 0 when g0 <= 0: Newton from
// x0 (0 when outside the bracket) safeguarded by the bracket -- a bisection step replaces
// the Newton step when that would leave the bracket or would not at least halve the step
// before last (the rule of the safeguarded Newton method of Press et al., Numerical
// Recipes, "rtsafe"); converged when a step is at most an ulp of the iterate, or when g is
// within two ulps of its largest term (gscale), its rounding noise (that last step is
// still taken).
template <class Eq>
__device__ __forceinline__ double find_root(const Law<double>& P, const Eq& e, double g0, double gscale, double hi,
                                            double x0, int* st) {
    if (!(g0 > 0.0)) return 0.0;
    double lo = 0.0, x = 0.0, dx = hi, dxold = hi;
    if (x0 > 0.0 && x0 < hi) x = x0;
    for (int it = 0; it < 200; ++it) {
        const auto o = e.eval(P, x);  // the bracket keeps g(lo) > 0 >= g(hi)
        if (o.g > 0.0) lo = x; else hi = x;
        if (o.g == 0.0) return x;
        const double xn = x - o.g / o.gx;
        const double moved = fabs(x - xn);
        if (o.gx < 0.0 && (moved <= 2.3e-16 * fabs(x) || fabs(o.g) <= 4.5e-16 * gscale))
            return xn >= lo && xn <= hi ? xn : x;
        if (!(o.gx < 0.0) || !(xn > lo && xn < hi) || fabs(2.0 * o.g) > fabs(dxold * o.gx)) {
            dxold = dx;
            dx = 0.5 * (hi - lo);
            x = lo + dx;
            if (x == lo || x == hi) return x;
            if (fabs(dx) <= 1e-16 * fabs(x)) return x;
        } else {
            dxold = dx;
            dx = x - xn;
            x = xn;
        }
        if (!(hi > lo)) return x;
    }
    *st |= ST_NOROOT;
    return x;
}

// a / b to the rounding of a division from r = 1 / b: the residual of a r corrected once
// (Markstein, IBM J. Res. Dev. 34, 1990), for several quotients by one divisor.
__device__ __forceinline__ double quotient(double a, double b, double r) {
    const double q = a * r;
    return fma(fma(-q, b, a), r, q);
}

// 1 / (dg/dx) for dx/d(dd_j) = -g_j / (dg/dx); 0 at x = 0 and where the slope vanishes
// (flagged).  The quotients are corrected: the tangent takes K dx from C, and where a return
// holds a traction the two nearly cancel, so the rounding of a plain product with this
// reciprocal came out several times larger.  (Corrections against divisions: 1,000,000 points of
// a softening joint 0.93 ms with divisions throughout.)
__device__ __forceinline__ double inverse_slope(double x, double gx, int* st) {
    if (!(x > 0.0)) return 0.0;
    if (!(gx != 0.0)) {
        *st |= ST_NOROOT;
        return 0.0;
    }
    return 1.0 / gx;
}

// An internal variable as it leaves the step: where it grew (inv = 1/v is not 0) v = q inv
// carries the rounding of both factors, and one Newton step takes it to that of sqrt(q)
// (1,000,000 points of a softening joint: 24 us more with square roots, 10 with this).
__device__ __forceinline__ double grown(double inv, double q, double v) {
    return inv > 0.0 ? fma(0.5 * inv, fma(-v, v, q), v) : v;
}

// open state: T' = 0, all of dd + C^-1 T'^n inelastic
__device__ __forceinline__ void open_state(const Prm& P, const Pt& p, const double dd[3], Res& r) {
    r.dp[0] = p.dp[0] + p.T[0] * P.iKs + dd[0];
    r.dp[1] = p.dp[1] + p.T[1] * P.iKs + dd[1];
    r.dp[2] = p.dp[2] + p.T[2] * P.iKn + dd[2];
    r.T[0] = r.T[1] = r.T[2] = 0.0;
    const double q = r.dp[0] * r.dp[0] + r.dp[1] * r.dp[1];
    const double s = sqrt(q), t = sqrt(q + r.dp[2] * r.dp[2]);
    r.chis = p.chis >= s ? p.chis : s;
    r.chit = p.chit >= t ? p.chit : t;
    r.wdil = p.wdil;
#pragma unroll
    for (int i = 0; i < 9; ++i) r.cep[i] = 0.0;
    r.mode = M_OPEN;
}

// the Coulomb equation from the trial traction (tau > 0); SIGN: only the sign of g is asked for
template <class R, bool SIGN = false>
__device__ __forceinline__ CoulombEq<R> make_coulomb(R tau, const double* Ttr, const double* dpb, const Pt& p) {
    CoulombEq<R> e;
    e.tau = tau;
    e.itau = R(1) / tau;
    if constexpr (sizeof(R) == 8 && !SIGN) {
        e.s0 = quotient(Ttr[0], tau, e.itau);
        e.s1 = quotient(Ttr[1], tau, e.itau);
    } else {
        e.s0 = (R)Ttr[0] * e.itau;
        e.s1 = (R)Ttr[1] * e.itau;
    }
    e.tn = (R)Ttr[2];
    e.p0 = (R)dpb[0];
    e.p1 = (R)dpb[1];
    e.pn = (R)dpb[2];
    e.chis = (R)p.chis;
    e.chit = (R)p.chit;
    return e;
}

// trial traction with the closed-state reference (damaged) or the plain one
__device__ __forceinline__ void trial(const Prm& P, const Pt& p, const double* dd, double dpn_shift, double* Ttr) {
    Ttr[0] = p.T[0] + P.Ks * dd[0];
    Ttr[1] = p.T[1] + P.Ks * dd[1];
    Ttr[2] = (p.T[2] - P.Kn * dpn_shift) + P.Kn * dd[2];
}

// The active mode at the trial state (values only; reading of the mode rules with
// hm_interface_update in hmat.h): M_ELASTIC, M_COULOMB, M_TENSILE, M_OPEN or M_APEX (a
// Coulomb return without a root before the shear traction vanishes).  dpb: the inelastic
// DD the return starts from (the closed-state normal part of a damaged point); shift:
// its normal change.
// the inelastic DD a return starts from and its normal change (closed-state reference of
// a fully damaged point); true if the point is fully damaged
__device__ __forceinline__ bool start_state(const Prm& P, const Pt& p, double dpb[3], double& shift) {
    const bool damaged = !(P.wc > 0.0) || p.chit >= P.wc;
    dpb[0] = p.dp[0];
    dpb[1] = p.dp[1];
    dpb[2] = p.dp[2];
    shift = 0.0;
    if (damaged) {
        const double wR = P.alphaR * P.wc + p.wdil;
        const double dpn_c = fmin(p.dp[2], wR);
        shift = dpn_c - p.dp[2];
        dpb[2] = dpn_c;
    }
    return damaged;
}

__device__ __forceinline__ int classify(const Prm& P, const Law<double>& W, const Pt& p, const double ddv[3],
                                        double dpb[3], double& shift) {
    const bool damaged = start_state(P, p, dpb, shift);
    double Ttr[3];
    trial(P, p, ddv, shift, Ttr);
    if (damaged && Ttr[2] > 0.0) return M_OPEN;
    const double tau = sqrt(Ttr[0] * Ttr[0] + Ttr[1] * Ttr[1]);
    const double f0 = W.f(p.chis) + W.fr;
    int kind = M_COULOMB;
    if (damaged) {
        if (tau + f0 * Ttr[2] <= 0.0) return M_ELASTIC;  // no cohesion left
    } else {
        const double c0 = W.c(p.chit), st0 = W.st(p.chit);
        const double Fc = tau + f0 * Ttr[2] - c0, Ft = Ttr[2] - st0;
        if (Fc <= 0.0 && Ft <= 0.0) return M_ELASTIC;
        const double a = sqrt(1.0 + f0 * f0) - f0;
        const double h = tau - (c0 - f0 * st0) - a * (Ttr[2] - st0);
        kind = h > 0.0 ? M_COULOMB : M_TENSILE;
    }
    if (kind == M_COULOMB) {
        if (!(tau > 0.0)) return M_APEX;
        // g where the shear traction vanishes: without ta, which is rounding noise there and would
        // decide for a frictionless contact (f = c = 0: g is zero), an apex return that opens it
        const auto o = make_coulomb<double, true>(tau, Ttr, dpb, p).eval(W, tau * P.iKs);
        if (o.f * o.Tn - o.c > 0.0) return M_APEX;
    }
    return kind;
}

__device__ __forceinline__ void finish_coulomb(const Prm& P, const Law<double>& W, const Law<float>& Wf, const Pt& p, const double* Ttr,
                                               const double* dpb, bool want_cep, Res& r, int* st) {
    const double tau = sqrt(Ttr[0] * Ttr[0] + Ttr[1] * Ttr[1]);
    const CoulombEq<double> e = make_coulomb<double>(tau, Ttr, dpb, p);
    const double hi = tau * P.iKs;
    // without softening the multiplier is F_trial / (Ks + f psi Kn)
    const CoulombEq<float> ef = make_coulomb<float>((float)tau, Ttr, dpb, p);
    const float f0 = Wf.f(ef.chis) + Wf.fr;
    const float x0 = (ef.tau + f0 * ef.tn - Wf.c(ef.chit)) / (Wf.Ks + f0 * Wf.psi(ef.chis) * Wf.Kn);
    const float xg = guess_root(Wf, ef, (float)hi, x0);
    const double x = find_root(W, e, e.at_zero(W), tau, hi, (double)xg, st);
    const auto o = e.eval(W, x);
    r.T[0] = o.ta * e.s0;
    r.T[1] = o.ta * e.s1;
    r.T[2] = o.Tn;
    r.dp[0] = o.a;
    r.dp[1] = o.b;
    r.dp[2] = o.n;
    r.chis = grown(o.ics, o.a * o.a + o.b * o.b, o.cs);
    r.chit = grown(o.ict, o.a * o.a + o.b * o.b + o.n * o.n, o.ct);
    r.wdil = p.wdil + o.psi * x;
    r.mode = M_COULOMB;
    if (!want_cep) return;
    // At fixed x a change of the trial shear turns s_hat: ds0 = Ks s1 (s1 d0 - s0 d1) / tau,
    // ds1 = -Ks s0 (s1 d0 - s0 d1) / tau, so a da + b db = x Ks / tau (a s1 - b s0) (s1 d0 - s0 d1)
    // with a s1 - b s0 = p0 s1 - p1 s0.
    const double kt = quotient(P.Ks, tau, e.itau), w = (e.p0 * e.s1 - e.p1 * e.s0) * (kt * x);
    const double ih = inverse_slope(x, o.gx, st);
    const double along = o.a * e.s0 + o.b * e.s1;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double rot = j == 0 ? e.s1 : (j == 1 ? -e.s0 : 0.0);
        const double dtau = j == 0 ? P.Ks * e.s0 : (j == 1 ? P.Ks * e.s1 : 0.0), dtn = j == 2 ? P.Kn : 0.0;
        const double dx = -quotient(e.slope(W, o, x, 0.0, w * rot, dtau, dtn), o.gx, ih);
        const double m = w * rot + dx * along;  // a da + b db of the whole change
        const double dn = dx * o.psi + x * (o.psi1 * (m * o.ics));
        const double dta = dtau - P.Ks * dx;
        r.cep[j] = dta * e.s0 + o.ta * (kt * e.s1 * rot);
        r.cep[3 + j] = dta * e.s1 - o.ta * (kt * e.s0 * rot);
        r.cep[6 + j] = dtn - P.Kn * dn;
    }
}

__device__ __forceinline__ void finish_apex(const Prm& P, const Law<double>& W, const Law<float>& Wf, const Pt& p, const double* Ttr,
                                            const double* dpb, bool want_cep, Res& r, int* st) {
    const bool sheared = Ttr[0] * Ttr[0] + Ttr[1] * Ttr[1] > 0.0;
    ApexEq<double> e;
    e.a = sheared ? dpb[0] + Ttr[0] * P.iKs : dpb[0];
    e.b = sheared ? dpb[1] + Ttr[1] * P.iKs : dpb[1];
    double v, inv, f1;
    root_of(e.a * e.a + e.b * e.b, v, inv);
    const bool on = !(p.chis >= v);
    r.chis = on ? grown(inv, e.a * e.a + e.b * e.b, v) : p.chis;
    e.f = W.f(r.chis, f1) + W.fr;
    e.tn = Ttr[2];
    e.pn = dpb[2];
    e.chit = p.chit;
    const ApexEq<float> ef{(float)e.tn, (float)e.a, (float)e.b, (float)e.f, (float)e.pn, (float)e.chit};
    const double hi = Ttr[2] * P.iKn;
    const float x0 = ef.f > 0.f ? (ef.tn - Wf.c(ef.chit) / ef.f) / Wf.Kn : 0.f;
    const double x = find_root(W, e, e.eval(W, 0.0).g, e.f * e.tn, hi, (double)guess_root(Wf, ef, (float)hi, x0), st);
    const auto o = e.eval(W, x);
    r.T[0] = r.T[1] = 0.0;
    r.T[2] = o.Tn;
    r.dp[0] = e.a;
    r.dp[1] = e.b;
    r.dp[2] = o.n;
    r.chit = grown(o.ict, e.a * e.a + e.b * e.b + o.n * o.n, o.ct);
    r.wdil = p.wdil;
    r.mode = M_APEX;
    if (!want_cep) return;
    const double ih = inverse_slope(x, o.gx, st);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double s = !sheared ? 0.0 : (j == 0 ? e.a : (j == 1 ? e.b : 0.0));  // a da + b db
        const double dtn = j == 2 ? P.Kn : 0.0;
        const double g = (on ? f1 * (s * inv) : 0.0) * o.Tn + e.f * dtn - o.c1 * (s * o.ict);
        r.cep[j] = r.cep[3 + j] = 0.0;
        r.cep[6 + j] = dtn + P.Kn * quotient(g, o.gx, ih);
    }
}

__device__ __forceinline__ void finish_tensile(const Prm& P, const Law<double>& W, const Law<float>& Wf, const Pt& p, const double* Ttr,
                                               const double* dpb, bool want_cep, Res& r, int* st) {
    const TensileEq<double> e{Ttr[2], dpb[0], dpb[1], dpb[2], p.chit};
    const TensileEq<float> ef{(float)e.tn, (float)e.p0, (float)e.p1, (float)e.pn, (float)e.chit};
    const double hi = Ttr[2] * P.iKn;
    const float x0 = (ef.tn - Wf.st(ef.chit)) / Wf.Kn;
    const double x = find_root(W, e, e.eval(W, 0.0).g, e.tn, hi, (double)guess_root(Wf, ef, (float)hi, x0), st);
    const auto o = e.eval(W, x);
    r.T[0] = Ttr[0];
    r.T[1] = Ttr[1];
    r.T[2] = o.Tn;
    r.dp[0] = dpb[0];
    r.dp[1] = dpb[1];
    r.dp[2] = o.n;
    r.chis = p.chis;
    r.chit = grown(o.ict, e.p0 * e.p0 + e.p1 * e.p1 + o.n * o.n, o.ct);
    r.wdil = p.wdil;
    r.mode = M_TENSILE;
    if (!want_cep) return;
#pragma unroll
    for (int i = 0; i < 9; ++i) r.cep[i] = 0.0;
    r.cep[0] = r.cep[4] = P.Ks;
    r.cep[8] = P.Kn + P.Kn * quotient(P.Kn, o.gx, inverse_slope(x, o.gx, st));
}

// The return of the given mode and, with want_cep, its derivative in Delta delta.  KIND is
// the mode (a template argument: each kernel holds the code of its own modes).
template <int KIND>
__device__ __forceinline__ void finish(const Prm& P, const Law<double>& W, const Law<float>& Wf, const Pt& p,
                                       const double ddv[3],
                                       const double dpb[3], double shift, bool want_cep, Res& r, int* st) {
    double Ttr[3];
    trial(P, p, ddv, shift, Ttr);
    if constexpr (KIND == M_OPEN) {
        open_state(P, p, ddv, r);
    } else if constexpr (KIND == M_ELASTIC) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            r.T[i] = Ttr[i];
            r.dp[i] = dpb[i];
        }
        r.chis = p.chis;
        r.chit = p.chit;
        r.wdil = p.wdil;
#pragma unroll
        for (int i = 0; i < 9; ++i) r.cep[i] = 0.0;
        r.cep[0] = r.cep[4] = P.Ks;
        r.cep[8] = P.Kn;
        r.mode = M_ELASTIC;
    } else if constexpr (KIND == M_COULOMB) {
        finish_coulomb(P, W, Wf, p, Ttr, dpb, want_cep, r, st);  // stays in contact whatever the damage
    } else {
        if constexpr (KIND == M_APEX)
            finish_apex(P, W, Wf, p, Ttr, dpb, want_cep, r, st);
        else
            finish_tensile(P, W, Wf, p, Ttr, dpb, want_cep, r, st);
        if (!(P.wc > 0.0) || r.chit >= P.wc) open_state(P, p, ddv, r);  // full damage: open
    }
}

struct IfArgs {
    Prm P;
    Law<float> Wf;  // converted once on the host: a conversion costs as much as an FP64 operation
    int64_t n;
    const double *T, *dp, *chi, *dd;  // the outputs may alias these: a point is read before it is written
    double *T1, *dp1, *chi1, *cep;
    int32_t* mode;
    unsigned long long* counts;  // per mode, then unresolved (or NULL)
    int32_t* list;               // [3][n]: points of the Coulomb, tensile and apex returns
    unsigned int* lcount;        // [3]
};

__device__ __forceinline__ void load_point(const IfArgs& a, int64_t e, Pt& p, double ddv[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        p.T[i] = a.T[3 * e + i];
        p.dp[i] = a.dp[3 * e + i];
        ddv[i] = a.dd[3 * e + i];
    }
    p.chis = a.chi[3 * e];
    p.chit = a.chi[3 * e + 1];
    p.wdil = a.chi[3 * e + 2];
}

__device__ __forceinline__ void store_point(const IfArgs& a, int64_t e, const Res& r, int st,
                                            unsigned int* s_cnt) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        a.T1[3 * e + i] = r.T[i];
        a.dp1[3 * e + i] = r.dp[i];
    }
    a.chi1[3 * e] = r.chis;
    a.chi1[3 * e + 1] = r.chit;
    a.chi1[3 * e + 2] = r.wdil;
    if (a.cep) {
#pragma unroll
        for (int i = 0; i < 9; ++i) a.cep[9 * e + i] = r.cep[i];
    }
    if (a.mode) a.mode[e] = r.mode | (st ? 256 : 0);
    atomicAdd(&s_cnt[r.mode], 1u);
    if (st) atomicAdd(&s_cnt[N_MODES], 1u);
}

__device__ __forceinline__ void flush_counts(const IfArgs& a, unsigned int* s_cnt) {
    __syncthreads();
    if (a.counts && threadIdx.x < N_MODES + 1 && s_cnt[threadIdx.x])
        atomicAdd(&a.counts[threadIdx.x], (unsigned long long)s_cnt[threadIdx.x]);
}

// list slot of each return kind (Coulomb, tensile, apex)
__device__ __forceinline__ int list_of(int kind) {
    return kind == M_COULOMB ? 0 : (kind == M_TENSILE ? 1 : (kind == M_APEX ? 2 : -1));
}

// Pass 1, one thread per point: the mode; elastic and open points are finished here, the
// returns are listed by kind so that pass 2 runs each kind in warps of that kind only
// (a warp over mixed modes would run every branch).
__global__ void __launch_bounds__(128) k_iface_classify(IfArgs a) {
    __shared__ unsigned int s_cnt[N_MODES + 1];
    if (threadIdx.x < N_MODES + 1) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int kind = -1;
    Pt p;
    double ddv[3], dpb[3], shift = 0.0;
    if (e < a.n) {
        const Law<double> W(a.P);
        load_point(a, e, p, ddv);
        kind = classify(a.P, W, p, ddv, dpb, shift);
        if (kind == M_ELASTIC || kind == M_OPEN) {
            int st = 0;
            Res r;
            if (kind == M_ELASTIC)
                finish<M_ELASTIC>(a.P, W, a.Wf, p, ddv, dpb, shift, a.cep != nullptr, r, &st);
            else
                finish<M_OPEN>(a.P, W, a.Wf, p, ddv, dpb, shift, a.cep != nullptr, r, &st);
            store_point(a, e, r, st, s_cnt);
        }
    }
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, list_of(kind) == k);
        if (m == 0u) continue;
        unsigned base = 0;
        if (lane == __ffs(m) - 1) base = atomicAdd(&a.lcount[k], (unsigned)__popc(m));
        base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
        if (list_of(kind) == k) a.list[(int64_t)k * a.n + base + __popc(m & ((1u << lane) - 1u))] = (int32_t)e;
    }
    flush_counts(a, s_cnt);
}

// Pass 2: the listed points of one return kind, grid-stride.  Bound by the FP64 pipe (80 to
// 86 % busy).  Of 1,000,000 points of a softening joint with the tangent, the Coulomb returns
// take 0.49 ms (dual numbers: 7.44), the apex returns 0.15 (1.42), the tensile ones 0.02
// (0.48), the classification 0.20 (0.32); the whole update 0.87 ms (9.56).
template <int KIND>
__global__ void __launch_bounds__(128) k_iface_return(IfArgs a) {
    __shared__ unsigned int s_cnt[N_MODES + 1];
    if (threadIdx.x < N_MODES + 1) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int k = list_of(KIND);
    const Law<double> W(a.P);
    const int64_t cnt = a.lcount[k];
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < cnt; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = a.list[(int64_t)k * a.n + q];
        Pt p;
        double ddv[3], dpb[3], shift = 0.0;
        load_point(a, e, p, ddv);
        start_state(a.P, p, dpb, shift);
        int st = 0;
        Res r;
        finish<KIND>(a.P, W, a.Wf, p, ddv, dpb, shift, a.cep != nullptr, r, &st);
        store_point(a, e, r, st, s_cnt);
    }
    flush_counts(a, s_cnt);
}

bool finite_pos(double x) { return std::isfinite(x) && x > 0.0; }
bool finite_nonneg(double x) { return std::isfinite(x) && x >= 0.0; }

}  // namespace
}  // namespace hm

extern "C" hm_status hm_interface_update(const hm_interface_params* prm, int64_t n, const double* T_dev,
                                         const double* dp_dev, const double* chi_dev, const double* dd_dev,
                                         double* T1_dev, double* dp1_dev, double* chi1_dev, double* cep_dev,
                                         int32_t* mode_dev, int64_t* counts, void* stream) {
    using namespace hm;
    HM_API_BEGIN
    hm::NvtxScope nvtx_("hm_interface_update");
    if (!prm) fail(HM_EINVAL, "interface_update: params is NULL");
    if (n < 0) fail(HM_EINVAL, "interface_update: n < 0");
    const hm_interface_params& q = *prm;
    if (!finite_pos(q.Ks) || !finite_pos(q.Kn)) fail(HM_EINVAL, "interface_update: stiffnesses must be > 0");
    if (!finite_nonneg(q.fp) || !finite_nonneg(q.fr) || !finite_nonneg(q.psip) || !finite_nonneg(q.cp) ||
        !finite_nonneg(q.sigp) || !finite_nonneg(q.wc) || !finite_nonneg(q.alphaR))
        fail(HM_EINVAL, "interface_update: friction, dilatancy, strengths, w_c and alpha_R must be finite and >= 0");
    if (!(q.dc > 0.0) || std::isnan(q.dc)) fail(HM_EINVAL, "interface_update: d_c must be > 0");
    if (n > 0 && (!T_dev || !dp_dev || !chi_dev || !dd_dev || !T1_dev || !dp1_dev || !chi1_dev))
        fail(HM_EINVAL, "interface_update: a state or increment pointer is NULL");
    if (n > INT32_MAX) fail(HM_EINVAL, "interface_update: more than 2^31 - 1 points");
    cudaStream_t st = (cudaStream_t)stream;
    DevBuf<unsigned long long> cnt;
    if (counts) {
        cnt.alloc(N_MODES + 1);
        HM_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes(), st));
    }
    auto inv = [](double x) { return x > 0.0 ? std::min(1.0 / x, DBL_MAX) : 0.0; };
    const Prm P{q.Ks, q.Kn, q.fp, q.fr, q.psip, q.dc, q.cp, q.sigp, q.wc, q.alphaR,
                inv(q.Ks), inv(q.Kn), inv(q.dc), inv(q.wc)};
    if (n > 0) {
        // stream-ordered scratch for the per-kind lists: no device-wide synchronisation
        void* scratch = nullptr;
        const size_t lbytes = (size_t)3 * n * sizeof(int32_t), cbytes = 4 * sizeof(unsigned int);
        HM_CUDA(cudaMallocAsync(&scratch, lbytes + cbytes, st));
        IfArgs a{P, Law<float>(P), n, T_dev, dp_dev, chi_dev, dd_dev, T1_dev, dp1_dev, chi1_dev, cep_dev, mode_dev,
                 counts ? cnt.p : nullptr, (int32_t*)scratch, (unsigned int*)((char*)scratch + lbytes)};
        cudaError_t err = cudaMemsetAsync(a.lcount, 0, cbytes, st);
        if (err == cudaSuccess) {
            k_iface_classify<<<(unsigned)ceil_div(n, 128), 128, 0, st>>>(a);
            int dev = 0, nsm = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            const unsigned g2 = (unsigned)std::min<int64_t>(ceil_div(n, 128), (int64_t)std::max(nsm, 1) * 16);
            k_iface_return<M_COULOMB><<<g2, 128, 0, st>>>(a);
            k_iface_return<M_TENSILE><<<g2, 128, 0, st>>>(a);
            k_iface_return<M_APEX><<<g2, 128, 0, st>>>(a);
            err = cudaGetLastError();
        }
        HM_CUDA(cudaFreeAsync(scratch, st));
        HM_CUDA(err);
    }
    if (counts) {
        unsigned long long h[N_MODES + 1];
        HM_CUDA(cudaMemcpyAsync(h, cnt.p, sizeof(h), cudaMemcpyDeviceToHost, st));
        HM_CUDA(cudaStreamSynchronize(st));
        for (int i = 0; i <= N_MODES; ++i) counts[i] = (int64_t)h[i];
        if (h[N_MODES]) fail(HM_ENOCONV, "interface_update: a plastic multiplier did not converge (" +
                                             std::to_string(h[N_MODES]) + " points)");
    }
    HM_API_END
}
