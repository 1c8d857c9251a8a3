// Pointwise kernels of the right-hand side (one thread per grid node, FP64).
//
//   k_prep  metric reconstruction -> primitive recovery -> densitized Valencia fluxes,
//           stress-energy tensor, radial light-cone speed          (paper: "The Primitive
//           Variable Recovery", "The Conserved Fluxes and Geometric Source Terms")
//   k_rhs   BSSN + gauge right-hand side, Valencia flux divergence + geometric sources,
//           interface penalty, outer-boundary freeze, Runge-Kutta stage combination
//           (paper: "BSSN Evolution Equations", "Gauge Conditions", "Time Integration")
//
// Field arrays are structure-of-arrays double[field][P], P = E*Nr*Nt*Np, phi fastest, so
// consecutive threads of a warp touch consecutive doubles of every field.
#include <math.h>

#include "fp_convert.cuh"
#include "grmhd_internal.h"

namespace gk {

// packed index of the symmetric pair (i, j): 00 01 02 11 12 22 -> 0..5 (a compile-time
// constant inside unrolled loops, so arrays indexed by it stay in registers)
__host__ __device__ constexpr int sym_idx(int i, int j) {
    return i <= j ? i * 3 - i * (i + 1) / 2 + j : j * 3 - j * (j + 1) / 2 + i;
}
#define SI(i, j) sym_idx(i, j)

// --------------------------------------------------------------------------- helpers
// Scalar invariants of the conserved state entering the one-variable master function
// in mu = 1/(h W) (Kastaun, Kalinani & Ciolfi 2021): q = tau/D, r^2 = S^2/D^2,
// bb = B^2/D, rb2 = (S.B)^2/D^3.  For the Gamma law h = 1 + Gamma eps, and the two
// estimates of h/W whose larger one the method takes are equal except where eps is clamped
// to eps_min, where h(eps_min)/W is the larger.  So the function is
//   g(mu) = mu z - 1,  z = h/W + mu rbar^2 = 1 + qbar + (Gamma - 1) eps / W  (eps not clamped),
// with the same sign and root as mu - 1/z and no further division.
template <class T>
struct C2PScal {
    T r2, bb, rb2;
    T c0, c1;       // qbar = c0 - c1 (mu x)^2: q - bb/2 and (bb r^2 - rb2)/2
    T g1, eps_min;  // Gamma - 1
    T v2max;        // r^2 / (1 + r^2), the largest admissible v^2
};

// With x = 1/(1 + mu bb), t = r^2 x^3 + mu x (S.B)^2/D^3 (1 + x + x^2) (r_par^2 + r_perp^2 x^3, split
// along and across the field), the derivatives by mu are those of sums of positive terms,
//   dv^2 = 2 mu t,  d(qbar - mu rbar^2) = -t,
//   dg = h/W + mu t (1 + (Gamma - 1) (mu W - 1)),  below the floor h/W + mu t (2 - h mu W),
// without the mu W where v^2 is clamped: FP32 keeps its accuracy of the slope however strong the
// field (differentiated term by term, x^3 is the difference of terms larger by 1/x: with fields
// of B^2 = 1e4 rho h and more the steps came out wrong, and W with them).
__device__ __forceinline__ float slope_t(float x, float w, float u) {    // w = r^2 x, u = mu x rb2
    return fmaf(w * x, x, u * fmaf(x, x, 1.f + x));
}

// g and its slope in FP32 alone: the search.  The cap on v^2 keeps W finite (at most 4,096: from
// there on FP32 has no digits of 1 - v^2 left, and eps / W, all that W enters by, has no weight)
struct Master32 {
    float g, dg;
};
__device__ __forceinline__ Master32 master32(float mu, const C2PScal<float>& c) {
    Master32 r;
    const float x = __fdividef(1.f, fmaf(mu, c.bb, 1.f)), mx = mu * x, w = c.r2 * x, u = mx * c.rb2;
    const float m1 = mu * fmaf(w, x, fmaf(u, x, u)), mt = mu * slope_t(x, w, u);
    const float qb = c.c0 - c.c1 * mx * mx;
    float v2 = mu * m1;
    const float cap = fminf(c.v2max, 1.f - 0x1p-24f);
    const bool clamped = !(v2 <= cap);
    if (clamped) v2 = cap;
    const float om = 1.f - v2, W = rsqrtf(om), iW = om * W, muW = clamped ? 0.f : mu * W;
    const float e = fmaf(W, 1.f + (qb - m1), -1.f);
    const bool gas = e >= c.eps_min;
    const float h = fmaf(1.f + c.g1, gas ? e : c.eps_min, 1.f);
    const float z = gas ? fmaf(c.g1 * e, iW, 1.f + qb) : fmaf(h, iW, m1);
    r.g = fmaf(mu, z, -1.f);
    r.dg = fmaf(mt, gas ? fmaf(c.g1, muW - 1.f, 1.f) : fmaf(-h, muW, 2.f), h * iW);
    return r;
}

// g in FP64 and the quantities that the primitives are made of
struct Master64 {
    double g, x, v2, m1, q2;     // v2 before the clamp to v2max; q2 = (mu x)^2
    float w, u;                  // r^2 x, mu x rb2
    double W, e;                 // of the clamped v2; eps before its floor
};
__device__ __forceinline__ Master64 master64(double mu, const C2PScal<double>& c) {
    Master64 r;
    r.x = rcp64(fma(mu, c.bb, 1.0));
    const double mx = mu * r.x;
    const double w = c.r2 * r.x, u = mx * c.rb2;
    r.w = d2f_rn(w);
    r.u = d2f_rn(u);
    r.q2 = mx * mx;
    r.m1 = mu * fma(r.x, w, fma(u, r.x, u));
    const double zb = fma(-c.c1, r.q2, 1.0 + c.c0);
    r.v2 = mu * r.m1;
    const double om = 1.0 - (r.v2 <= c.v2max ? r.v2 : c.v2max);
    r.W = rsqrt64(om);
    const double iW = om * r.W;
    r.e = fma(r.W, zb - r.m1, -1.0);
    const double z = r.e >= c.eps_min ? fma(c.g1 * r.e, iW, zb) : fma(fma(1.0 + c.g1, c.eps_min, 1.0), iW, r.m1);
    r.g = fma(mu, z, -1.0);
    return r;
}

// The slope of g where FP64 has evaluated it, in FP32, from the evaluation's own quantities: W (what
// FP32 cannot resolve of 1 - v^2, W enters with W^2 times its relative error), eps, and on which
// side of v2max and of eps_min the point lies (cold gas has v^2 within about eps / W^2 of v2max).
struct Slope32 {
    float dg, t, dv2, de;        // dv2, de: before the clamp and the floor
};
__device__ __forceinline__ Slope32 slope32(float mu, const Master64& f, const C2PScal<double>& c64,
                                           const C2PScal<float>& c) {
    Slope32 r;
    r.t = slope_t(d2f_rn(f.x), f.w, f.u);
    const float mt = mu * r.t;
    r.dv2 = 2.f * mt;
    // W of the evaluation (1 <= W < 2^27), cut to FP32
    const float W = __uint_as_float(__funnelshift_l((uint32_t)__double2loint(f.W), (uint32_t)__double2hiint(f.W) - 0x38000000u, 3));
    const float muW = f.v2 <= c64.v2max ? mu * W : 0.f, e = d2f_rn(f.e);
    r.de = W * r.t * fmaf(muW, 1.f + e, -1.f);
    const bool gas = f.e >= c64.eps_min;
    const float h = fmaf(1.f + c.g1, gas ? e : c.eps_min, 1.f);
    r.dg = fmaf(mt, gas ? fmaf(c.g1, muW - 1.f, 1.f) : fmaf(-h, muW, 2.f), __fdividef(h, W));
    return r;
}

// Primitive recovery at one point: the root of g in the bracket [0, 1] (h >= 1).  FP32 finds
// it to FP32's accuracy from the guess (its pipe is idle: 64 FP32 instructions issue in the
// time of one FP64 instruction); then Newton steps with the residual in FP64 and the slope in
// FP32 to about 1e-6, so that a step leaves that much of the last one's error unless a kink of g
// lies between: two FP64 evaluations of 27 instructions in place of three or four of ~110
// with the derivative carried in FP64.  Safeguarded by bisection throughout.  Returns 1 on
// success without floor, 0 if eps was floored or the iteration did not converge; *mu_o, *x_o,
// *W_o, *iW_o, *eps_o (floored) at the root.
__device__ __forceinline__ int con2prim_root(const C2PScal<double>& c, int maxit, double tol, float guess,
                                             double* mu_o, double* x_o, double* W_o, double* iW_o, double* eps_o) {
    const C2PScal<float> cf = {d2f_rn(c.r2), d2f_rn(c.bb), d2f_rn(c.rb2),     d2f_rn(c.c0),
                               d2f_rn(c.c1), d2f_rn(c.g1), d2f_rn(c.eps_min), d2f_rn(c.v2max)};
    float m = (guess > 0.f && guess < 1.f) ? guess : 0.5f;
    {
        // until the step is within a few units of FP32's noise; else the iterate of least |g|
        float lo = 0.f, hi = 1.f, best = m, gbest = 3e38f;
        for (int it = 0; it < 12; it++) {
            const Master32 f = master32(m, cf);
            if (fabsf(f.g) < gbest) { gbest = fabsf(f.g); best = m; }
            const float mn = m - __fdividef(f.g, f.dg);
            if (fabsf(mn - m) <= 4e-6f * m) {
                best = mn;
                break;
            }
            if (f.g < 0.f) lo = m; else hi = m;
            m = (mn > lo && mn < hi) ? mn : 0.5f * (lo + hi);
        }
        m = best;
    }
    double lo = 0.0, hi = 1.0, mu = f2d(fminf(m, 1.f)), delta = 0.0;
    float dprev = 0.f;
    int conv = 0;
    Master64 f;
    Slope32 s;
    const float tolf = (float)tol;
    // f(0+) < 0 and f(1) >= 0 for every admissible state (h >= 1); a state without a root
    // never converges and is flagged below.  Stop when the Newton step is below tol, or when
    // two consecutive steps d_{k-1} > d_k predict the next one, d_k (d_k / d_{k-1}) for linear
    // convergence, below tol / 100 and the step crosses no kink of g (the slope changes there:
    // for cold gas by a factor of two), or when a step of rounding size leaves the bracket.  The
    // limit counts the FP64 evaluations that a step follows.
    for (int it = 0;; it++) {
        f = master64(mu, c);
        s = slope32(d2f_rn(mu), f, c, cf);
        delta = 0.0;
        if (it >= maxit) break;
        if (f.g == 0.0) { conv = 1; break; }
        if (f.g < 0.0) lo = mu; else hi = mu;
        double mn = fma(-f.g, f2d(__fdividef(1.f, s.dg)), mu);
        // (late steps that do not shrink are rounding noise of g, which a strong field makes large:
        // the bracket is halved instead)
        const bool newton = mn > lo && mn < hi && !(it >= 24 && dprev > 0.f && fabsf(d2f_rn(mn - mu)) > 0.5f * dprev);
        if (!newton) {
            if (fabsf(d2f_rn(mn - mu)) <= 4e-15f * d2f_rn(mu)) { conv = 1; break; }
            mn = 0.5 * (lo + hi);
        }
        delta = mn - mu;
        const float dk = fabsf(d2f_rn(delta)), mf = d2f_rn(mn);
        if (dk <= tolf * mf) { conv = 1; break; }
        if (newton && dprev > dk && dk <= 1e-3f * mf && __fdividef(dk, dprev) * dk <= 0.01f * tolf * mf &&
            fabsf(s.dv2) * dk <= fabsf(d2f_rn(f.v2 - c.v2max)) && fabsf(s.de) * dk <= fabsf(d2f_rn(f.e) - cf.eps_min)) {
            conv = 1;
            break;
        }
        dprev = newton ? dk : 0.f;
        mu = mn;
        if (hi - lo <= tol * hi) {
            conv = 1;
            f = master64(mu, c);
            delta = 0.0;
            break;
        }
    }
    double qm = fma(-c.c1, f.q2, c.c0) - f.m1;    // qbar - mu rbar^2
    if (delta != 0.0) {
        // the last step is not evaluated any more: to first order, or, where tol let it be
        // large, after all
        mu += delta;
        if (fabs(delta) > 1e-10 * mu) {
            f = master64(mu, c);
            qm = fma(-c.c1, f.q2, c.c0) - f.m1;
        } else {
            const float x = d2f_rn(f.x);
            f.x = fma(f2d(__fdividef(x * x - x, d2f_rn(mu))), delta, f.x);    // dx = -bb x^2
            f.v2 = fma(f2d(s.dv2), delta, f.v2);
            qm = fma(f2d(-s.t), delta, qm);
        }
    }
    const double v2 = f.v2 <= c.v2max ? f.v2 : c.v2max;
    const double om = 1.0 - v2, W = rsqrt64(om);
    // eps without the cancellation of W (1 + qm) - 1: W - 1 = W^2 v^2 / (1 + W)
    const double e = fma(W, qm, v2 * W * W * rcp64(1.0 + W));
    *mu_o = mu;
    *x_o = f.x;
    *W_o = W;
    *iW_o = om * W;
    *eps_o = fmax(e, c.eps_min);
    return conv && e >= c.eps_min;
}

// The paper's primitive recovery (Methods, "The Primitive Variable Recovery") as an option
// (opts.c2p_lambda > 0): predicted conserved variables from the current primitives,
// residuals dS_i, dtau, the damped update v^i += lam gamma^ij dS_j / (rho h W^2),
// eps += lam dtau / (rho W^2), rho = D / W, lam halved (and the update retried) while the
// residual grows, stop at ||dS|| + |dtau| < tol D; after maxit updates one Newton-Raphson
// update of eps on the tau residual.  The same sequence of steps and tests as the oracle's
// con2prim_damped (W <= 10, eps >= eps_min after every update), in FP64.
struct DampedResid {
    double dS[3], dtau, nrm;
};

__device__ __forceinline__ double lorentz_w(const double v[3], const double g[3][3]) {
    double v2 = 0.0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) v2 += g[i][j] * v[i] * v[j];
    return 1.0 / sqrt(1.0 - v2);
}

__device__ void damped_resid(double rho, const double v[3], double eps, const double B[3], const double g[3][3],
                             const double gi[3][3], double gam, const double S_d[3], double tau, DampedResid* r) {
    const double W = lorentz_w(v, g);
    const double pr = (gam - 1.0) * rho * eps;
    const double h = 1.0 + eps + pr / rho;
    const double Z = rho * h * W * W;
    double v_d[3], B_d[3];
    for (int i = 0; i < 3; i++) {
        v_d[i] = g[i][0] * v[0] + g[i][1] * v[1] + g[i][2] * v[2];
        B_d[i] = g[i][0] * B[0] + g[i][1] * B[1] + g[i][2] * B[2];
    }
    const double B2 = B_d[0] * B[0] + B_d[1] * B[1] + B_d[2] * B[2];
    const double vB = v_d[0] * B[0] + v_d[1] * B[1] + v_d[2] * B[2];
    for (int i = 0; i < 3; i++) r->dS[i] = S_d[i] - ((Z + B2) * v_d[i] - vB * B_d[i]);
    r->dtau = tau - (Z + B2 - pr - 0.5 * (B2 / (W * W) + vB * vB) - rho * W);
    double q = 0.0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) q += r->dS[i] * gi[i][j] * r->dS[j];
    r->nrm = sqrt(fmax(q, 0.0)) + fabs(r->dtau);
}

__device__ __forceinline__ void damped_clamp(double v[3], double* eps, const double g[3][3], double v2max,
                                             double eps_min) {
    double v2 = 0.0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) v2 += g[i][j] * v[i] * v[j];
    const double f = sqrt(fmin(1.0, v2max / fmax(v2, 1e-300)));
    for (int i = 0; i < 3; i++) v[i] *= f;
    *eps = fmax(*eps, eps_min);
}

// Returns 1 if the residual fell below tol D without the final Newton update and without a
// floor; rho, v, eps hold the starting point on entry.
__device__ int con2prim_damped_point(double D, const double S_d[3], double tau, const double B_u[3],
                                     const double g[3][3], const double gi[3][3], double gam, double eps_min,
                                     int maxit, double tol, double lam0, double* rho, double v[3], double* eps,
                                     double* pr, double* Wout) {
    const double v2max = 1.0 - 1.0 / (10.0 * 10.0);
    damped_clamp(v, eps, g, v2max, eps_min);
    *rho = D / lorentz_w(v, g);
    double lam = lam0;
    bool done = false;
    DampedResid r0;
    for (int it = 0; it < maxit; it++) {
        damped_resid(*rho, v, *eps, B_u, g, gi, gam, S_d, tau, &r0);
        if (r0.nrm < tol * D) { done = true; break; }
        const double W = lorentz_w(v, g);
        const double pr0 = (gam - 1.0) * (*rho) * (*eps);
        const double h = 1.0 + *eps + pr0 / (*rho);
        const double iZ = 1.0 / (*rho * h * W * W);
        double dv[3];
        for (int i = 0; i < 3; i++)
            dv[i] = (gi[i][0] * r0.dS[0] + gi[i][1] * r0.dS[1] + gi[i][2] * r0.dS[2]) * iZ;
        const double de = r0.dtau / (*rho * W * W);
        double tl = lam;
        for (int hv = 0; hv <= 30; hv++) {
            double tv[3] = {v[0] + tl * dv[0], v[1] + tl * dv[1], v[2] + tl * dv[2]};
            double te = *eps + tl * de;
            damped_clamp(tv, &te, g, v2max, eps_min);
            const double tr = D / lorentz_w(tv, g);
            DampedResid r1;
            damped_resid(tr, tv, te, B_u, g, gi, gam, S_d, tau, &r1);
            if (r1.nrm <= r0.nrm || hv == 30) {
                for (int i = 0; i < 3; i++) v[i] = tv[i];
                *eps = te;
                *rho = tr;
                lam = tl;
                break;
            }
            tl *= 0.5;
        }
    }
    if (!done) {
        damped_resid(*rho, v, *eps, B_u, g, gi, gam, S_d, tau, &r0);
        done = r0.nrm < tol * D;
    }
    const double W = lorentz_w(v, g);
    if (!done) *eps += r0.dtau / (*rho * (gam * W * W - gam + 1.0));
    const int ok = done && (*eps >= eps_min);
    *eps = fmax(*eps, eps_min);
    *pr = (gam - 1.0) * (*rho) * (*eps);
    *Wout = W;
    return ok;
}

// --------------------------------------------------------------------------- k_prep
// Densitized fluxes and matter terms of one node in FP64 from the primitives: W b^i and
// the Eulerian projections of T^{mu nu},
//   Z = rho h* W^2, b^i = B^i / W + W (v.B) v^i, E = Z - p* - W^2 (v.B)^2,
//   S_i = Z v_i - W (v.B) b_i, S^ij = Z v^i v^j + p* gamma^ij - b^i b^j,
// with h* = 1 + eps + (p + b^2)/rho, p* = p + b^2/2 (alpha b^0 = W (v.B); the spatial part of
// b_mu is b_i).  The factor sqrt(gamma) goes into the scalars once instead of into every
// flux, F^i_{B^k} is formed from the densitized field and antisymmetric, and no T^{mu nu}
// is built: ~140 FP64 instructions against ~240 for the four-vector form, on a kernel
// that the FP64 pipe bounds.  mat (densitized): E, S_i, E + S, S^ij, Z v_i v_j - b_i b_j (the
// right-hand side needs S_ij only up to multiples of gamma_ij; S = E - rho (1 + eps) + 3 p).
__device__ __forceinline__ void fluxes64(long long p, long long P, double alpha, const double beta[3],
                                         const double gti[6], double e4m, double sqg, double rho, const double v[3],
                                         const double v_d[3], double eps, double pr, double W, double iW,
                                         const double B[3], const double B_d[3], double B2, const double Bs[3],
                                         double* __restrict__ flux, double* __restrict__ mat) {
    double b_u[3], b_d[3], vt[3];
    const double vB = v_d[0] * B[0] + v_d[1] * B[1] + v_d[2] * B[2], WvB = W * vB;
    const double b2 = B2 * (iW * iW) + vB * vB;
    for (int i = 0; i < 3; i++) {
        b_u[i] = B[i] * iW + WvB * v[i];
        b_d[i] = B_d[i] * iW + WvB * v_d[i];
        vt[i] = alpha * v[i] - beta[i];
    }
    const double r1 = rho + rho * eps, ps = pr + 0.5 * b2;
    const double Z = (r1 + pr + b2) * (W * W);
    const double D = sqg * (rho * W), E = sqg * (Z - ps - WvB * WvB), tau = E - D;
    const double sZ = sqg * Z, sp = sqg * ps, aps = alpha * sp, sW = sqg * WvB;
    double S[3], Bw[3];
    const double aw = alpha * iW;
    for (int i = 0; i < 3; i++) {
        S[i] = sZ * v_d[i] - sW * b_d[i];
        Bw[i] = aw * Bs[i];
    }
    for (int i = 0; i < 3; i++) {
        double* F = flux + (long long)(i * 8) * P + p;
        F[0 * P] = D * vt[i];
        for (int j = 0; j < 3; j++) {
            const double f = S[j] * vt[i] - b_d[j] * Bw[i];
            F[(1 + j) * P] = i == j ? f + aps : f;
        }
        F[4 * P] = tau * vt[i] + (aps * v[i] - WvB * Bw[i]);
        F[(5 + i) * P] = 0.0;
    }
    for (int i = 0; i < 3; i++)
        for (int k = i + 1; k < 3; k++) {
            const double f = vt[i] * Bs[k] - vt[k] * Bs[i];
            flux[(long long)(i * 8 + 5 + k) * P + p] = f;
            flux[(long long)(k * 8 + 5 + i) * P + p] = -f;
        }
    mat[0 * P + p] = E;
    for (int i = 0; i < 3; i++) mat[(1 + i) * P + p] = S[i];
    mat[4 * P + p] = 2.0 * E - sqg * (r1 - 3.0 * pr);
    const double spe = sp * e4m;
    double zv[3], zd[3], sb[3], sd[3];
    for (int i = 0; i < 3; i++) {
        zv[i] = sZ * v[i];
        zd[i] = sZ * v_d[i];
        sb[i] = sqg * b_u[i];
        sd[i] = sqg * b_d[i];
    }
    for (int i = 0; i < 3; i++)
        for (int j = i; j < 3; j++) {
            mat[(5 + SI(i, j)) * P + p] = zv[i] * v[j] + (spe * gti[SI(i, j)] - sb[i] * b_u[j]);
            mat[(11 + SI(i, j)) * P + p] = zd[i] * v_d[j] - sd[i] * b_d[j];
        }
}

// What a launch computes: the primitives alone, or also the fluxes and matter terms in FP64
// or FP32.  Bound by the FP64 pipe (87 % busy): 346 FP64 instructions per node against 707
// in FP64, so the launch inside the stepping of 393,216 nodes went from 545 to 281 us (ncu),
// the FP32 form from 384 to 198 us, the recovery of a newly loaded state (grmhd_con2prim,
// whole call) from 807 to 247 us.  Three blocks per SM (168 registers): per step of three
// launches 843 us in FP64 and 586 us in FP32.  Measured when that was chosen, with a slope of a
// few instructions less: 843 and 575 with three, 865 and 580 with four (128 registers, spills of
// 120 B), 972 and 634 with five.
enum { PREP_PRIM = 0, PREP_F64 = 1, PREP_F32 = 2 };

template <int WHAT>
__global__ void __launch_bounds__(128, 3) k_prep(Dims d, PhysParams pp, const double* __restrict__ U,
                                              double* __restrict__ prim, double* __restrict__ flux,
                                              double* __restrict__ tmn, double* __restrict__ lam,
                                              unsigned long long* __restrict__ nfail, double* __restrict__ met) {
    long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long P = d.P;
    int bad = 0;
    if (p < P) {
        // gamma = e^{4phi} gammatilde, gamma^-1 = e^{-4phi} gammatilde^-1, det gamma =
        // e^{12phi} det gammatilde, computed as the right-hand side uses them and kept in met
        // (e^{4phi}, e^{-4phi}, sqrt(gamma), gammatilde^ij) so that k_rhs reads them: GB300's
        // FP64 pipe bounds both kernels
        const double e4 = exp(4.0 * U[V_PHI * P + p]);
        const double e4m = rcp64(e4);
        double gt[6], gti[6];
        for (int q = 0; q < 6; q++) gt[q] = U[(V_GT + q) * P + p];
        const double c00 = gt[3] * gt[5] - gt[4] * gt[4], c01 = gt[2] * gt[4] - gt[1] * gt[5],
                     c02 = gt[1] * gt[4] - gt[2] * gt[3];
        const double detgt = gt[0] * c00 + gt[1] * c01 + gt[2] * c02;
        const double id = rcp64(detgt);
        gti[0] = c00 * id; gti[1] = c01 * id; gti[2] = c02 * id;
        gti[3] = (gt[0] * gt[5] - gt[2] * gt[2]) * id;
        gti[4] = (gt[1] * gt[2] - gt[0] * gt[4]) * id;
        gti[5] = (gt[0] * gt[3] - gt[1] * gt[1]) * id;
        const double detg = e4 * e4 * e4 * detgt;
        const double isq = rsqrt64(detg), sqg = detg * isq;
        double Us[3], Bs[3], B_u[3], B_d[3];
        const double Ud = U[V_D * P + p], Ut = U[V_TAU * P + p];
        for (int i = 0; i < 3; i++) {
            Us[i] = U[(V_S + i) * P + p];
            Bs[i] = U[(V_B + i) * P + p];
            B_u[i] = Bs[i] * isq;
        }
        for (int i = 0; i < 3; i++)
            B_d[i] = e4 * (gt[SI(i, 0)] * B_u[0] + gt[SI(i, 1)] * B_u[1] + gt[SI(i, 2)] * B_u[2]);
        const double B2 = B_d[0] * B_u[0] + B_d[1] * B_u[1] + B_d[2] * B_u[2];
        const double Dc = Ud * isq, tau = Ut * isq;

        double rho, v[3], v_d[3], eps, pr, W, iW;
        int ok;
        const bool gas = Dc > pp.rho_atm && isfinite(Dc) && isfinite(tau);
        if (gas && !(pp.c2p_lambda > 0.0)) {
            // ratios to D straight from the densitized variables
            const double iU = rcp64(Ud), iD = iU * sqg;
            double s[3], su[3];
            for (int i = 0; i < 3; i++) s[i] = Us[i] * iU;
            for (int i = 0; i < 3; i++)
                su[i] = e4m * (gti[SI(i, 0)] * s[0] + gti[SI(i, 1)] * s[1] + gti[SI(i, 2)] * s[2]);
            const double sB = s[0] * B_u[0] + s[1] * B_u[1] + s[2] * B_u[2];
            C2PScal<double> c;
            c.r2 = s[0] * su[0] + s[1] * su[1] + s[2] * su[2];
            c.bb = B2 * iD;
            c.rb2 = sB * sB * iD;
            c.c0 = Ut * iU - 0.5 * c.bb;
            c.c1 = 0.5 * (c.bb * c.r2 - c.rb2);
            c.g1 = pp.gam - 1.0;
            c.eps_min = pp.eps_atm;
            c.v2max = c.r2 * rcp64(1.0 + c.r2);
            if (__double2hiint(c.v2max) >= 0x3FF00000) c.v2max = 1.0 - 0x1p-53;    // r above 1e8: W stays finite
            // guess mu = 1/(h W) from the stored primitives
            const float guess = __fdividef(1.f, (1.f + (float)pp.gam * d2f_rn(prim[4 * P + p])) * d2f_rn(prim[6 * P + p]));
            double mu, x;
            ok = con2prim_root(c, pp.c2p_maxit, pp.c2p_tol, guess, &mu, &x, &W, &iW, &eps);
            rho = Dc * iW;
            pr = c.g1 * rho * eps;
            // v_i = mu x (S_i/D + mu (S.B) B_i / D^2)
            const double mx = mu * x, fac = mu * (sB * iD);
            for (int i = 0; i < 3; i++) {
                v_d[i] = mx * (s[i] + fac * B_d[i]);
                v[i] = mx * (su[i] + fac * B_u[i]);
            }
        } else {
            double g[3][3];
            for (int i = 0; i < 3; i++)
                for (int j = 0; j < 3; j++) g[i][j] = e4 * gt[SI(i, j)];
            if (gas) {
                double gi[3][3], S_d[3];
                for (int i = 0; i < 3; i++) {
                    S_d[i] = Us[i] * isq;
                    for (int j = 0; j < 3; j++) gi[i][j] = e4m * gti[SI(i, j)];
                }
                // the paper's damped iteration from the stored primitives, or (after a reset)
                // from the dust estimates v^i = gamma^ij S_j / (tau + D), eps = (tau + D)/(D W) - 1
                const double Wg = prim[6 * P + p];
                if (Wg >= 1.0 && prim[0 * P + p] > 0.0) {
                    rho = prim[0 * P + p];
                    for (int i = 0; i < 3; i++) v[i] = prim[(1 + i) * P + p];
                    eps = prim[4 * P + p];
                } else {
                    const double ie = 1.0 / (tau + Dc);
                    for (int i = 0; i < 3; i++)
                        v[i] = (gi[i][0] * S_d[0] + gi[i][1] * S_d[1] + gi[i][2] * S_d[2]) * ie;
                    eps = 0.0;
                    damped_clamp(v, &eps, g, 1.0 - 1.0 / (10.0 * 10.0), 0.0);
                    const double W0 = lorentz_w(v, g);
                    eps = fmax((tau + Dc) / (Dc * W0) - 1.0, pp.eps_atm);
                    rho = Dc / W0;
                }
                ok = con2prim_damped_point(Dc, S_d, tau, B_u, g, gi, pp.gam, pp.eps_atm, pp.c2p_maxit, pp.c2p_tol,
                                           pp.c2p_lambda, &rho, v, &eps, &pr, &W);
            } else {
                ok = 0;
                rho = pp.rho_atm; v[0] = v[1] = v[2] = 0.0; eps = pp.eps_atm;
                pr = (pp.gam - 1.0) * rho * eps; W = 1.0;
            }
            iW = 1.0 / W;
            for (int i = 0; i < 3; i++) v_d[i] = g[i][0] * v[0] + g[i][1] * v[1] + g[i][2] * v[2];
        }
        bad = !ok;
        prim[0 * P + p] = rho;
        prim[1 * P + p] = v[0];
        prim[2 * P + p] = v[1];
        prim[3 * P + p] = v[2];
        prim[4 * P + p] = eps;
        prim[5 * P + p] = pr;
        prim[6 * P + p] = W;

        if constexpr (WHAT != PREP_PRIM) {
            met[0 * P + p] = e4;
            met[1 * P + p] = e4m;
            met[2 * P + p] = sqg;
            for (int q = 0; q < 6; q++) met[(3 + q) * P + p] = gti[q];
            const double alpha = U[V_ALPHA * P + p];
            const double beta[3] = {U[V_BETA * P + p], U[(V_BETA + 1) * P + p], U[(V_BETA + 2) * P + p]};
            // the light-cone speed is read at the element ends (interface penalty) only
            const uint32_t ir = ((uint32_t)p / (uint32_t)d.NtNp) % (uint32_t)d.Nr;
            if (ir == 0 || ir == (uint32_t)d.Nr - 1) lam[p] = fabs(beta[0]) + alpha * sqrt(e4m * gti[0]);
            if constexpr (WHAT == PREP_F64) {
                met[9 * P + p] = isq;
                fluxes64(p, P, alpha, beta, gti, e4m, sqg, rho, v, v_d, eps, pr, W, iW, B_u, B_d, B2, Bs, flux, tmn);
            } else {
                using R = float;
                double g[3][3], gi[3][3];
                for (int i = 0; i < 3; i++)
                    for (int j = 0; j < 3; j++) {
                        g[i][j] = e4 * gt[SI(i, j)];
                        gi[i][j] = e4m * gti[SI(i, j)];
                    }
                // ---- four-vectors, fluxes and T^{mu nu} of the mixed modes in FP32 (their consumers,
                // the tensor-core contractions and the FP32 right-hand side, keep about 24 bits); the
                // primitive recovery above stays FP64
                const R alphaR = narrow<R>(alpha), sqgR = narrow<R>(sqg), WR = narrow<R>(W);
                R gR[3][3], betaR[3], vR[3], BR[3];
                for (int i = 0; i < 3; i++) {
                    betaR[i] = narrow<R>(beta[i]);
                    vR[i] = narrow<R>(v[i]);
                    BR[i] = narrow<R>(B_u[i]);
                    for (int j = 0; j < 3; j++) gR[i][j] = narrow<R>(g[i][j]);
                }
                R vR_d[3];
                for (int i = 0; i < 3; i++) vR_d[i] = gR[i][0] * vR[0] + gR[i][1] * vR[1] + gR[i][2] * vR[2];
                R ia = R(1.0) / alphaR;
                R u0 = WR * ia;
                R uu[3];
                for (int i = 0; i < 3; i++) uu[i] = WR * (vR[i] - betaR[i] * ia);
                R b0 = WR * (vR_d[0] * BR[0] + vR_d[1] * BR[1] + vR_d[2] * BR[2]) * ia;
                R iWR = R(1.0) / WR;
                R bu[3];
                for (int i = 0; i < 3; i++) bu[i] = (BR[i] + alphaR * b0 * uu[i]) * iWR;
                R beta_d[3];
                for (int i = 0; i < 3; i++)
                    beta_d[i] = gR[i][0] * betaR[0] + gR[i][1] * betaR[1] + gR[i][2] * betaR[2];
                R bb_ = beta_d[0] * betaR[0] + beta_d[1] * betaR[1] + beta_d[2] * betaR[2];
                R g00 = -alphaR * alphaR + bb_;
                R bd0 = g00 * b0 + beta_d[0] * bu[0] + beta_d[1] * bu[1] + beta_d[2] * bu[2];
                R bd[3];
                for (int i = 0; i < 3; i++)
                    bd[i] = beta_d[i] * b0 + gR[i][0] * bu[0] + gR[i][1] * bu[1] + gR[i][2] * bu[2];
                R b2 = b0 * bd0 + bu[0] * bd[0] + bu[1] * bd[1] + bu[2] * bd[2];
                const R rhoR = narrow<R>(rho), epsR = narrow<R>(eps), prR = narrow<R>(pr);
                R pstar = prR + R(0.5) * b2;
                R rhohs = rhoR * (R(1.0) + epsR) + prR + b2;   // rho h*
                // conserved variables from the primitives (undensitized)
                R Dp = rhoR * WR;
                R Sp[3];
                for (int j = 0; j < 3; j++) Sp[j] = rhohs * WR * WR * vR_d[j] - alphaR * b0 * bd[j];
                // tau = rho h* W^2 - p* - alpha^2 b0^2 - D without its cancellation: with
                // W^2 - 1 = W^2 v^2 and W - 1 = W^2 v^2 / (W + 1),
                // tau = rho W (eps W + W^2 v^2 / (W + 1)) + p W^2 v^2 + b^2 (W^2 - 1/2) - alpha^2 b0^2
                // (tau ~ 1e-3 D for a cold gas: the direct form loses 3 digits, all of FP32's margin)
                const R Wv2 = WR * WR * (vR_d[0] * vR[0] + vR_d[1] * vR[1] + vR_d[2] * vR[2]);
                const R taup = rhoR * WR * (epsR * WR + Wv2 / (WR + R(1.0))) + prR * Wv2 + b2 * (WR * WR - R(0.5)) -
                               alphaR * alphaR * b0 * b0;
                // ---- densitized fluxes [dir][var]
                R vt[3];
                for (int i = 0; i < 3; i++) vt[i] = alphaR * vR[i] - betaR[i];
                for (int i = 0; i < 3; i++) {
                    // kept in FP32, as is T^{mu nu}: half the bytes, no conversion here and in the readers
                    R* F = reinterpret_cast<R*>(flux) + (long long)(i * 8) * P + p;
                    F[0 * P] = sqgR * (Dp * vt[i]);
                    for (int j = 0; j < 3; j++)
                        F[(1 + j) * P] = sqgR * (Sp[j] * vt[i] + (i == j ? alphaR * pstar : R(0.0)) -
                                                 alphaR * bd[j] * BR[i] * iWR);
                    F[4 * P] = sqgR * (taup * vt[i] + alphaR * pstar * vR[i] - alphaR * alphaR * b0 * BR[i] * iWR);
                    for (int k = 0; k < 3; k++) F[(5 + k) * P] = sqgR * (vt[i] * BR[k] - vt[k] * BR[i]);
                }
                // ---- T^{mu nu}
                R ia2 = ia * ia;
                R gu[4][4];
                gu[0][0] = -ia2;
                for (int i = 0; i < 3; i++) gu[0][i + 1] = gu[i + 1][0] = betaR[i] * ia2;
                for (int i = 0; i < 3; i++)
                    for (int j = 0; j < 3; j++) gu[i + 1][j + 1] = narrow<R>(gi[i][j]) - betaR[i] * betaR[j] * ia2;
                R u4[4] = {u0, uu[0], uu[1], uu[2]};
                R b4[4] = {b0, bu[0], bu[1], bu[2]};
                int n = 0;
                for (int m = 0; m < 4; m++)
                    for (int k = m; k < 4; k++, n++)
                        reinterpret_cast<R*>(tmn)[n * P + p] = rhohs * u4[m] * u4[k] + pstar * gu[m][k] - b4[m] * b4[k];
            }
        }
    }
    // warp-aggregated failure count
    unsigned m = __ballot_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(nfail, (unsigned long long)__popc(m));
}

// --------------------------------------------------------------------------- k_rhs
// the 6 second-derivative pairs rr, rth, rph, thth, thph, phph use the same packing
#define c_pair_idx(i, j) sym_idx(i, j)

// The mixed modes' right-hand side (FP32 algebra; FP64 runs k_rhs64 below).  Bound by memory
// and latency, not by arithmetic, so it keeps the four-dimensional form of the matter terms.
// Each variable is written as soon as it is known, as in k_rhs64 (MODE likewise), and two
// blocks per SM have the registers to do it without spills: 393,216 nodes 144 -> 101 us (98 now,
// about 5.7 TB/s of its ~1.4 KB per node); three blocks of 168 registers with 500 B of spills a
// thread take 142 us, four 156 us.
template <int MODE, bool HAM>
__global__ void __launch_bounds__(128, 2) k_rhs(Dims d, PhysParams pp, const double* __restrict__ U0,
                                             const double* __restrict__ Us,
                                             const float* __restrict__ flux,
                                             const float* __restrict__ tmn,
                                             const double* __restrict__ lam,
                                             const double* __restrict__ met,
                                             const float* __restrict__ d1,
                                             const float* __restrict__ d2,
                                             const float* __restrict__ divF,
                                             const float* __restrict__ divB,
                                             const double* __restrict__ r_scale,
                                             const double* __restrict__ dt_dev, RKCoef co,
                                             double* __restrict__ out, double* __restrict__ acc,
                                             double* __restrict__ ham) {
    using R = float;
    long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long P = d.P;
    if (p >= P) return;
    const R PI = R(3.141592653589793);
    const R third = R(1.0 / 3.0), sixth = R(1.0 / 6.0), two3 = R(2.0 / 3.0);
    const int elem_id = (int)((uint32_t)p / (uint32_t)d.elem);
    const uint32_t ir = ((uint32_t)p / (uint32_t)d.NtNp) % (uint32_t)d.Nr;
    // frozen outer boundary node of each instance
    const bool frozen = ir == (uint32_t)d.Nr - 1 && !d.iface_next[elem_id];
    const double dt = MODE == 0 ? 0.0 : dt_dev[d.elem_inst[elem_id]];
    // a variable is written as soon as its right-hand side is known
    const auto emit = [&](int v, R r) {
        const long long ix = v * P + p;
        const double L = frozen ? 0.0 : widen(r);
        if (MODE == 0) { out[ix] = L; return; }
        double o;
        if (MODE == 1) o = Us[ix] + dt * L;
        else if (MODE == 2) o = co.a * U0[ix] + co.b * (Us[ix] + dt * L);
        else {
            // RK4: next stage input U0 + c dt L, accumulator acc (+)= w dt L;
            // final stage (acc_mode 3): U0 + acc + w dt L
            const double wl = co.w * dt * L;
            if (co.acc_mode == 1) { acc[ix] = wl; o = U0[ix] + co.c * dt * L; }
            else if (co.acc_mode == 2) { acc[ix] += wl; o = U0[ix] + co.c * dt * L; }
            else { o = U0[ix] + (acc[ix] + wl); }
        }
        out[ix] = o;
    };

    // ------------------------------------------------------------ state and metric
    R gt[3][3], At[3][3];
    double gt64[3][3];
    for (int i = 0; i < 3; i++)
        for (int j = i; j < 3; j++) {
            gt64[i][j] = gt64[j][i] = Us[(V_GT + SI(i, j)) * P + p];
            gt[i][j] = gt[j][i] = narrow<R>(gt64[i][j]);
            At[i][j] = At[j][i] = narrow<R>(Us[(V_AT + SI(i, j)) * P + p]);
        }
    const R K = narrow<R>(Us[V_K * P + p]);
    const R alpha = narrow<R>(Us[V_ALPHA * P + p]);
    R Gam[3], beta[3], Bg[3];
    for (int i = 0; i < 3; i++) {
        Gam[i] = narrow<R>(Us[(V_GAM + i) * P + p]);
        beta[i] = narrow<R>(Us[(V_BETA + i) * P + p]);
        Bg[i] = narrow<R>(Us[(V_BG + i) * P + p]);
    }
    // conformal factor, physical metric, its determinant and inverse, conformal inverse:
    // FP64 in every mode; the algebra below runs in R.  e^{4phi}, e^{-4phi}, sqrt(gamma)
    // and gammatilde^ij come from k_prep's met (the same formulas on the same state);
    // gamma = e^{4phi} gammatilde, gamma^{-1} = e^{-4phi} gammatilde^{-1}
    const double e4 = met[0 * P + p], e4m = met[1 * P + p];
    const R e4r = narrow<R>(e4), e4mr = narrow<R>(e4m);
    double g64[3][3], gi64[3][3], gti64[3][3];
    for (int i = 0; i < 3; i++)
        for (int j = i; j < 3; j++) gti64[i][j] = gti64[j][i] = met[(3 + SI(i, j)) * P + p];
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            g64[i][j] = e4 * gt64[i][j];
            gi64[i][j] = e4m * gti64[i][j];
        }
    const R sqg = narrow<R>(met[2 * P + p]);
    R g[3][3], gi[3][3], gti[3][3];
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            g[i][j] = narrow<R>(g64[i][j]);
            gi[i][j] = narrow<R>(gi64[i][j]);
            gti[i][j] = narrow<R>(gti64[i][j]);
        }

    // first derivatives: field f, direction dd -> d1[(f*3+dd)*P + p]
#define D1(f, dd) ((R)d1[((long long)(f) * 3 + (dd)) * P + p])
    R dgt[3][3][3], dAt[3][3][3], dphi[3], dK[3], dGam[3][3], dal[3], dbe[3][3];
    for (int k = 0; k < 3; k++) {
        for (int i = 0; i < 3; i++)
            for (int j = i; j < 3; j++) {
                dgt[k][i][j] = dgt[k][j][i] = D1(V_GT + SI(i, j), k);
                dAt[k][i][j] = dAt[k][j][i] = D1(V_AT + SI(i, j), k);
            }
        dphi[k] = D1(V_PHI, k);
        dK[k] = D1(V_K, k);
        dal[k] = D1(V_ALPHA, k);
        for (int i = 0; i < 3; i++) {
            dGam[k][i] = D1(V_GAM + i, k);
            dbe[k][i] = D1(V_BETA + i, k);
        }
    }
#undef D1

    // ------------------------------------------------------------ Valencia
    {
        R rv[NV_MAX - V_D];
        R T00 = tmn[0 * P + p];
        R T0i[3] = {tmn[1 * P + p], tmn[2 * P + p], tmn[3 * P + p]};
        R Tij[3][3];
        Tij[0][0] = tmn[4 * P + p]; Tij[0][1] = Tij[1][0] = tmn[5 * P + p];
        Tij[0][2] = Tij[2][0] = tmn[6 * P + p]; Tij[1][1] = tmn[7 * P + p];
        Tij[1][2] = Tij[2][1] = tmn[8 * P + p]; Tij[2][2] = tmn[9 * P + p];
        R beta_d[3];
        for (int i = 0; i < 3; i++)
            beta_d[i] = g[i][0] * beta[0] + g[i][1] * beta[1] + g[i][2] * beta[2];
        R T0_d[3];
        for (int i = 0; i < 3; i++)
            T0_d[i] = beta_d[i] * T00 + g[i][0] * T0i[0] + g[i][1] * T0i[1] + g[i][2] * T0i[2];
        const R K3 = K * third;
        R Kij[3][3];
        for (int i = 0; i < 3; i++)
            for (int j = i; j < 3; j++) Kij[i][j] = Kij[j][i] = e4r * (At[i][j] + gt[i][j] * K3);
        R asg = alpha * sqg;
        // symmetric weights w_kl (1 on the diagonal, 2 off it) folded into the contracted
        // tensors: bbw = w beta^k beta^l, tbw = w (T^{0k} beta^l)_(kl), Tw = w T^{kl}
        R bbw[6], tbw[6], Tw[6], gtw[3] = {R(0.0), R(0.0), R(0.0)};
        for (int k = 0; k < 3; k++)
            for (int l = k; l < 3; l++) {
                const int q = SI(k, l);
                const R w = k == l ? R(1.0) : R(2.0);
                bbw[q] = w * beta[k] * beta[l];
                tbw[q] = R(0.5) * w * (T0i[k] * beta[l] + T0i[l] * beta[k]);
                Tw[q] = w * Tij[k][l];
                gtw[0] += bbw[q] * gt[k][l];
                gtw[1] += tbw[q] * gt[k][l];
                gtw[2] += Tw[q] * gt[k][l];
            }
        for (int jd = 0; jd < 3; jd++) {
            // d_j gamma_kl = e^{4phi} (d_j gammatilde_kl + 4 gammatilde_kl d_j phi)
            R sb = R(0.0), st = R(0.0), sT = R(0.0);
            for (int k = 0; k < 3; k++)
                for (int l = k; l < 3; l++) {
                    const int q = SI(k, l);
                    sb += bbw[q] * dgt[jd][k][l];
                    st += tbw[q] * dgt[jd][k][l];
                    sT += Tw[q] * dgt[jd][k][l];
                }
            const R f4 = R(4.0) * dphi[jd];
            const R bbdg = e4r * (sb + f4 * gtw[0]);
            const R t0dg = e4r * (st + f4 * gtw[1]);
            const R tdg = e4r * (sT + f4 * gtw[2]);
            R t0db = T0_d[0] * dbe[jd][0] + T0_d[1] * dbe[jd][1] + T0_d[2] * dbe[jd][2];
            R SS = T00 * (R(0.5) * bbdg - alpha * dal[jd]) + t0dg + t0db + R(0.5) * tdg;
            rv[V_S - V_D + jd] = -(R)divF[(1 + jd) * P + p] + asg * SS;
        }
        R bbK = R(0.0), TK = R(0.0), t0 = R(0.0);
        for (int k = 0; k < 3; k++)
            for (int l = k; l < 3; l++) {
                bbK += bbw[SI(k, l)] * Kij[k][l];
                TK += Tw[SI(k, l)] * Kij[k][l];
            }
        for (int i = 0; i < 3; i++) {
            const R bK = beta[0] * Kij[i][0] + beta[1] * Kij[i][1] + beta[2] * Kij[i][2];
            t0 += T0i[i] * (R(2.0) * bK - dal[i]);
        }
        R bda = beta[0] * dal[0] + beta[1] * dal[1] + beta[2] * dal[2];
        R Stau = T00 * (bbK - bda) + t0 + TK;
        rv[0] = -(R)divF[0 * P + p];
        rv[V_TAU - V_D] = -(R)divF[4 * P + p] + asg * Stau;
        for (int k = 0; k < 3; k++) rv[V_B - V_D + k] = -(R)divF[(5 + k) * P + p];
        // GLM cleaning: d_t psi = alpha (-c_h^2 D_i B^i - psi / tau) with the covariant
        // divergence d_i(sqrt(gamma) B^i) / sqrt(gamma); field source -alpha sqrt(gamma)
        // gamma^ij d_j psi (d psi: d1 field N_D1)
        if (pp.glm) {
            const R psi = narrow<R>(Us[(long long)V_PSI * P + p]);
            R dpsi[3];
            for (int k = 0; k < 3; k++) dpsi[k] = (R)d1[((long long)N_D1 * 3 + k) * P + p];
            rv[V_PSI - V_D] = alpha * (-narrow<R>(pp.glm_ch2) * (R)divB[p] / sqg - psi * narrow<R>(pp.glm_itau));
            for (int i = 0; i < 3; i++)
                rv[V_B - V_D + i] -= asg * (gi[i][0] * dpsi[0] + gi[i][1] * dpsi[1] + gi[i][2] * dpsi[2]);
        }

        // interface penalty (Rusanov flux, strong form) at duplicated element-end nodes
        const long long shell = d.NtNp;
        const int e = elem_id;
        int side = 0;
        if (ir == (uint32_t)d.Nr - 1 && d.iface_next[e]) side = +1;
        if (ir == 0 && e > 0 && d.iface_next[e - 1]) side = -1;
        if (side != 0) {
            long long pl = side > 0 ? p : p - shell;
            long long pr_ = side > 0 ? p + shell : p;
            double lmax = fmax(lam[pl], lam[pr_]);
            double J = 1.0 / r_scale[e];
            double fac = 1.0 / (pp.w_end * J);
            for (int v = 0; v < 8; v++) {
                double FL = widen(flux[(0 * 8 + v) * P + pl]);
                double FR = widen(flux[(0 * 8 + v) * P + pr_]);
                double UL = Us[(V_D + v) * P + pl];
                double UR = Us[(V_D + v) * P + pr_];
                double Fs = 0.5 * (FL + FR) - 0.5 * lmax * (UR - UL);
                if (side > 0) rv[v] += narrow<R>((FL - Fs) * fac);
                else rv[v] -= narrow<R>((FR - Fs) * fac);
            }
        }

#pragma unroll
        for (int v = 0; v < 8; v++) emit(V_D + v, pp.evolve_fluid ? rv[v] : R(0));
        if (pp.glm) emit(V_PSI, pp.evolve_fluid ? rv[V_PSI - V_D] : R(0));

        // matter terms for BSSN: rho = alpha^2 T^00, S_i = alpha T^0_i,
        // S_ij = g_{i mu} g_{j nu} T^{mu nu}
        if (pp.evolve_metric) {
            R rho_m = alpha * alpha * T00;
            R S_i[3];
            for (int i = 0; i < 3; i++) S_i[i] = alpha * T0_d[i];
            R Sij[3][3], Str = R(0.0);
            R gT[3][3];  // gamma_ik T^{kj}
            for (int i = 0; i < 3; i++)
                for (int j = 0; j < 3; j++)
                    gT[i][j] = g[i][0] * Tij[0][j] + g[i][1] * Tij[1][j] + g[i][2] * Tij[2][j];
            R gT0[3];
            for (int i = 0; i < 3; i++) gT0[i] = g[i][0] * T0i[0] + g[i][1] * T0i[1] + g[i][2] * T0i[2];
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    R s = beta_d[i] * beta_d[j] * T00 + beta_d[i] * gT0[j] + beta_d[j] * gT0[i] +
                               gT[i][0] * g[0][j] + gT[i][1] * g[1][j] + gT[i][2] * g[2][j];
                    Sij[i][j] = Sij[j][i] = s;
                    Str += (i == j ? R(1.0) : R(2.0)) * gi[i][j] * s;
                }

            // -------------------------------------------------------- BSSN
#define D2(f, q) ((R)d2[((long long)(f) * 6 + (q)) * P + p])
            // Christoffels of gammatilde: lower Cl[k][i][j] = Gamma_{k ij}, upper Cu[k][i][j]
            R Cl[3][3][3], Cu[3][3][3];
            for (int k = 0; k < 3; k++)
                for (int i = 0; i < 3; i++)
                    for (int j = i; j < 3; j++)
                        Cl[k][i][j] = Cl[k][j][i] =
                            R(0.5) * (dgt[i][k][j] + dgt[j][k][i] - dgt[k][i][j]);
            for (int k = 0; k < 3; k++)
                for (int i = 0; i < 3; i++)
                    for (int j = i; j < 3; j++)
                        Cu[k][i][j] = Cu[k][j][i] =
                            gti[k][0] * Cl[0][i][j] + gti[k][1] * Cl[1][i][j] + gti[k][2] * Cl[2][i][j];
            // gammatilde^{jk} with the symmetric weights (contractions with symmetric tensors)
            R gw[6];
            for (int j = 0; j < 3; j++)
                for (int k = j; k < 3; k++) gw[SI(j, k)] = (j == k ? R(1.0) : R(2.0)) * gti[j][k];
            R Gd[3];
            for (int i = 0; i < 3; i++) {
                R s = R(0.0);
                for (int j = 0; j < 3; j++)
                    for (int k = j; k < 3; k++) s += gw[SI(j, k)] * Cu[i][j][k];
                Gd[i] = s;
            }
            R divb = dbe[0][0] + dbe[1][1] + dbe[2][2];
            // Bt[k][j][m] = gti^{lm} Gamma_{k l j}.  The quadratic Christoffel part of the
            // Ricci tensor, gti^{lm} (Gamma^k_{li} Gamma_{jkm} + Gamma^k_{lj} Gamma_{ikm} +
            // Gamma^k_{im} Gamma_{klj}), is Pq_ij + Pq_ji + Qq_ij with
            // Pq_ij = Gamma^k_{li} Bt[j][k][l] and the symmetric Qq_ij = Gamma^k_{im} Bt[k][j][m].
            R Bt[3][3][3];
            for (int k = 0; k < 3; k++)
                for (int i = 0; i < 3; i++)
                    for (int m = 0; m < 3; m++)
                        Bt[k][i][m] = gti[0][m] * Cl[k][0][i] + gti[1][m] * Cl[k][1][i] + gti[2][m] * Cl[k][2][i];
            R Pq[3][3];
            for (int i = 0; i < 3; i++)
                for (int j = 0; j < 3; j++) {
                    R t = R(0.0);
                    for (int k = 0; k < 3; k++)
                        for (int l = 0; l < 3; l++) t += Cu[k][l][i] * Bt[j][k][l];
                    Pq[i][j] = t;
                }
            R ddphi[3][3], ddal[3][3];
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    int q = c_pair_idx(i, j);
                    ddphi[i][j] = ddphi[j][i] = D2(6, q);
                    ddal[i][j] = ddal[j][i] = D2(7, q);
                }
            R DDphi[3][3], DDal[3][3];
            R gdphi2 = R(0.0);
            R gradphi_u[3];
            for (int k = 0; k < 3; k++)
                gradphi_u[k] = gti[k][0] * dphi[0] + gti[k][1] * dphi[1] + gti[k][2] * dphi[2];
            gdphi2 = gradphi_u[0] * dphi[0] + gradphi_u[1] * dphi[1] + gradphi_u[2] * dphi[2];
            R gdphida = gradphi_u[0] * dal[0] + gradphi_u[1] * dal[1] + gradphi_u[2] * dal[2];
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    R cp = Cu[0][i][j] * dphi[0] + Cu[1][i][j] * dphi[1] + Cu[2][i][j] * dphi[2];
                    R ca = Cu[0][i][j] * dal[0] + Cu[1][i][j] * dal[1] + Cu[2][i][j] * dal[2];
                    DDphi[i][j] = DDphi[j][i] = ddphi[i][j] - cp;
                    // physical Christoffels: + 2(d_i a d_j phi + d_j a d_i phi - gt_ij gt^kl d_l phi d_k a)
                    R cphys = ca + R(2.0) * (dal[i] * dphi[j] + dal[j] * dphi[i] - gt[i][j] * gdphida);
                    DDal[i][j] = DDal[j][i] = ddal[i][j] - cphys;
                }
            R lapphi = R(0.0), trDDal = R(0.0);
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    lapphi += gw[SI(i, j)] * DDphi[i][j];
                    trDDal += gw[SI(i, j)] * DDal[i][j];
                }
            trDDal *= e4mr;
            // Atilde with raised indices
            R Aud[3][3], Auu[3][3];
            for (int k = 0; k < 3; k++)
                for (int j = 0; j < 3; j++)
                    Aud[k][j] = gti[k][0] * At[0][j] + gti[k][1] * At[1][j] + gti[k][2] * At[2][j];
            R AA = R(0.0);
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    Auu[i][j] = Auu[j][i] = Aud[i][0] * gti[0][j] + Aud[i][1] * gti[1][j] + Aud[i][2] * gti[2][j];
                    AA += (i == j ? R(1.0) : R(2.0)) * At[i][j] * Auu[i][j];
                }

            // X_ij = -D_i D_j alpha + alpha (R_ij - 8 pi S_ij)
            R X[3][3];
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    int sij = SI(i, j);
                    R lapg = R(0.0);
                    for (int l = 0; l < 3; l++)
                        for (int m = l; m < 3; m++) lapg += gw[SI(l, m)] * D2(sij, c_pair_idx(l, m));
                    R Ric = -R(0.5) * lapg;
                    for (int k = 0; k < 3; k++)
                        Ric += R(0.5) * (gt[k][i] * dGam[j][k] + gt[k][j] * dGam[i][k]) +
                               R(0.5) * Gd[k] * (Cl[i][j][k] + Cl[j][i][k]);
                    R t = Pq[i][j] + Pq[j][i];
                    for (int k = 0; k < 3; k++)
                        for (int m = 0; m < 3; m++) t += Cu[k][i][m] * Bt[k][j][m];
                    Ric += t;
                    Ric += -R(2.0) * DDphi[i][j] - R(2.0) * gt[i][j] * lapphi + R(4.0) * dphi[i] * dphi[j] -
                           R(4.0) * gt[i][j] * gdphi2;
                    X[i][j] = X[j][i] = -DDal[i][j] + alpha * (Ric - R(8.0) * PI * Sij[i][j]);
                }
            R trX = R(0.0);
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) trX += gw[SI(i, j)] * X[i][j];
            const R trX3 = trX * third;
            for (int i = 0; i < 3; i++)
                for (int j = i; j < 3; j++) {
                    int sij = SI(i, j);
                    R adv_g = beta[0] * dgt[0][i][j] + beta[1] * dgt[1][i][j] + beta[2] * dgt[2][i][j];
                    R adv_a = beta[0] * dAt[0][i][j] + beta[1] * dAt[1][i][j] + beta[2] * dAt[2][i][j];
                    R lg = R(0.0), la = R(0.0), AAd = R(0.0);
                    for (int k = 0; k < 3; k++) {
                        lg += gt[i][k] * dbe[j][k] + gt[j][k] * dbe[i][k];
                        la += At[i][k] * dbe[j][k] + At[j][k] * dbe[i][k];
                        AAd += At[i][k] * Aud[k][j];
                    }
                    emit(V_GT + sij, -R(2.0) * alpha * At[i][j] + adv_g + lg - two3 * gt[i][j] * divb);
                    R XTF = X[i][j] - gt[i][j] * trX3;
                    emit(V_AT + sij, e4mr * XTF + alpha * (K * At[i][j] - R(2.0) * AAd) + adv_a + la -
                                      two3 * At[i][j] * divb);
                }
            emit(V_PHI, -alpha * K * sixth + (beta[0] * dphi[0] + beta[1] * dphi[1] + beta[2] * dphi[2]) +
                         divb * sixth);
            // diagnostics only: the Hamiltonian constraint R + (2/3) K^2 - Atilde.Atilde - 16 pi rho,
            // with R = gamma^ij R_ij = (e^{-4 phi} trX + trDDal) / alpha + 8 pi S (trX, trDDal
            // as above: the same Ricci tensor, no extra derivative)
            // (a separate instance, HAM = true, so that the stepping kernel carries none of it)
            if constexpr (HAM)
                ham[p] = widen((e4mr * trX + trDDal) / alpha + R(8.0) * PI * Str + two3 * K * K - AA -
                               R(16.0) * PI * rho_m);
            emit(V_K, -trDDal + alpha * (AA + K * K3) + R(4.0) * PI * alpha * (rho_m + Str) +
                       (beta[0] * dK[0] + beta[1] * dK[1] + beta[2] * dK[2]));
            // Gammatilde
            R ddb[3][3][3];  // [q pair via j,k][i]
            for (int j = 0; j < 3; j++)
                for (int k = j; k < 3; k++)
                    for (int i = 0; i < 3; i++)
                        ddb[j][k][i] = ddb[k][j][i] = D2(7 + 1 + i, c_pair_idx(j, k));
            R ddbk[3];  // d_j d_k beta^k
            for (int j = 0; j < 3; j++) ddbk[j] = ddb[j][0][0] + ddb[j][1][1] + ddb[j][2][2];
            for (int i = 0; i < 3; i++) {
                R s = R(0.0);
                for (int j = 0; j < 3; j++)
                    for (int k = j; k < 3; k++) s += gw[SI(j, k)] * ddb[j][k][i];
                R s2 = gti[i][0] * ddbk[0] + gti[i][1] * ddbk[1] + gti[i][2] * ddbk[2];
                R adv = beta[0] * dGam[0][i] + beta[1] * dGam[1][i] + beta[2] * dGam[2][i];
                R gdb = Gam[0] * dbe[0][i] + Gam[1] * dbe[1][i] + Gam[2] * dbe[2][i];
                R Ada = Auu[i][0] * dal[0] + Auu[i][1] * dal[1] + Auu[i][2] * dal[2];
                R CA = R(0.0);
                for (int j = 0; j < 3; j++)
                    for (int k = j; k < 3; k++) CA += (j == k ? R(1.0) : R(2.0)) * Cu[i][j][k] * Auu[j][k];
                R Adp = Auu[i][0] * dphi[0] + Auu[i][1] * dphi[1] + Auu[i][2] * dphi[2];
                R gdK = gti[i][0] * dK[0] + gti[i][1] * dK[1] + gti[i][2] * dK[2];
                R gS = gti[i][0] * S_i[0] + gti[i][1] * S_i[1] + gti[i][2] * S_i[2];
                const R rg = s + s2 * third + adv - gdb + two3 * Gam[i] * divb - R(2.0) * Ada +
                                 R(2.0) * alpha * (CA + R(6.0) * Adp - two3 * gdK) -
                                 R(16.0) * PI * alpha * gS;
                emit(V_GAM + i, rg);
                emit(V_BG + i, pp.gauge == 0 ? rg - narrow<R>(pp.eta) * Bg[i] : R(0.0));
            }
#undef D2
            if (pp.gauge == 0) {
                emit(V_ALPHA, -R(2.0) * alpha * K + beta[0] * dal[0] + beta[1] * dal[1] + beta[2] * dal[2]);
                for (int i = 0; i < 3; i++) emit(V_BETA + i, R(0.75) * Bg[i]);
            } else {
                emit(V_ALPHA, R(0.0));
                for (int i = 0; i < 3; i++) emit(V_BETA + i, R(0.0));
            }
        } else {
            for (int v = 0; v < N_BSSN; v++) emit(v, R(0.0));
        }
    }
}

// --------------------------------------------------------------------------- k_rhs64
// The FP64 right-hand side.  GB300's FP64 pipe (2 instructions per SM clock) bounds it, so
// the algebra is arranged for the fewest FP64 instructions (~950 per node and stage, 1,567
// in the form of k_rhs below; the arrangement is the same system of equations):
//   * matter as densitized Eulerian projections (see k_prep): the Valencia sources contract
//     S^ij alone, 1/2 S^ij d_k gamma_ij + S_i d_k beta^i - E d_k alpha (T^00 beta beta +
//     2 T^0i beta + T^ij is S^ij), and S_ij needs no lowering;
//   * C_kij = 2 Gammatilde_kij from d_i gammatilde_jk: nine of its 18 components are single
//     derivatives (C_iij = d_j gammatilde_ii), the others take 1 or 2 operations;
//   * Gammatilde^k d_k gammatilde_ij replaces Gammatilde^k (Gammatilde_ijk + Gammatilde_jik);
//   * only the trace-free part of X_ij is used, so its terms proportional to gammatilde_ij
//     (Laplacian of phi, (d phi)^2, d phi . d alpha, the pressure) are left out;
//   * - 2/3 div beta goes into the diagonal of d_j beta^k, alpha (K/2 - Atilde) beside it;
//   * every gammatilde^ij v_j term of the Gammatilde equation shares one product.
// A variable is written as soon as its right-hand side is known (no array of 33 in local
// memory: 254 registers without spills, against 904 B of spills per thread).  Measured on
// 393,216 nodes, per launch: 1.085 -> 0.603 ms.  MODE: 0 the plain right-hand side, 1 the first SSP-RK3 stage Us + dt L, 2 the
// others a U0 + b (Us + dt L), 3 RK4 stages.  DIVP: parts of divF to add (1, or 3 on small grids).
//
// PART: the variables that an instance writes; what only the others need drops out.  One
// thread per node cannot run faster than ~950 FP64 instructions in turn, 64 clocks each on
// an SM quarter (30 us), so grids of few nodes, which leave most quarters idle, give a node
// to two threads: RHS_A Atilde_ij (the Ricci tensor), RHS_B the rest, with the bits of
// RHS_ALL.  4,608 nodes: 35.9 -> 22.8 us.
enum { RHS_A = 1, RHS_B = 2, RHS_ALL = 3 };

template <int MODE, int PART>
struct Emit {
    const double *U0, *Us;
    double *out, *acc;
    long long P, p;
    double a, b, bdt, cdt, wdt;
    int acc_mode;
    bool frozen;
    __device__ __forceinline__ void operator()(int v, double L) const {
        if (!((v >= V_AT && v < V_AT + 6 ? RHS_A : RHS_B) & PART)) return;
        const long long ix = v * P + p;
        if (frozen) L = 0.0;
        if (MODE == 0) out[ix] = L;
        else if (MODE == 1) out[ix] = fma(bdt, L, Us[ix]);
        else if (MODE == 2) out[ix] = fma(bdt, L, fma(b, Us[ix], a * U0[ix]));
        else {
            // next stage input U0 + c dt L, accumulator acc (+)= w dt L; final stage U0 + acc + w dt L
            const double u0 = U0[ix];
            if (acc_mode == 1) { acc[ix] = wdt * L; out[ix] = fma(cdt, L, u0); }
            else if (acc_mode == 2) { acc[ix] = fma(wdt, L, acc[ix]); out[ix] = fma(cdt, L, u0); }
            else out[ix] = u0 + fma(wdt, L, acc[ix]);
        }
    }
};

template <int MODE, bool HAM, int DIVP, int PART>
__device__ __forceinline__ void rhs64_node(long long p, const Dims& d, const PhysParams& pp,
                                           const double* __restrict__ U0, const double* __restrict__ Us,
                                           const double* __restrict__ flux, const double* __restrict__ mat,
                                           const double* __restrict__ lam, const double* __restrict__ met,
                                           const double* __restrict__ d1, const double* __restrict__ d2,
                                           const double* __restrict__ divF, const double* __restrict__ divB,
                                           const double* __restrict__ r_scale, const double* __restrict__ dt_dev,
                                           const RKCoef& co, double* __restrict__ out, double* __restrict__ acc,
                                           double* __restrict__ ham) {
    const long long P = d.P;
    const int e = (int)(p / d.elem);
    const long long ir = (p / d.NtNp) % d.Nr;
    const double dt = MODE == 0 ? 0.0 : dt_dev[d.elem_inst[e]];
    // the outer boundary node of each instance is frozen
    const Emit<MODE, PART> emit = {U0, Us, out, acc, P, p, co.a, co.b, co.b * dt, co.c * dt, co.w * dt, co.acc_mode,
                             ir == d.Nr - 1 && !d.iface_next[e]};
#define LD(a, k) __ldg((a) + (long long)(k) * P + p)
#define D1(f, dd) LD(d1, (f) * 3 + (dd))
#define D2(f, q) LD(d2, (f) * 6 + (q))
    const double alpha = LD(Us, V_ALPHA), K = LD(Us, V_K);
    double beta[3], gt[6], At[6], gti[6], dgt[3][6], dphi[3], dal[3], dbe[3][3];
#pragma unroll
    for (int q = 0; q < 6; q++) {
        gt[q] = LD(Us, V_GT + q);
        At[q] = LD(Us, V_AT + q);
        gti[q] = LD(met, 3 + q);
    }
#pragma unroll
    for (int k = 0; k < 3; k++) {
        beta[k] = LD(Us, V_BETA + k);
        dphi[k] = D1(V_PHI, k);
        dal[k] = D1(V_ALPHA, k);
#pragma unroll
        for (int q = 0; q < 6; q++) dgt[k][q] = D1(V_GT + q, k);
#pragma unroll
        for (int i = 0; i < 3; i++) dbe[k][i] = D1(V_BETA + i, k);
    }
    const double e4m = LD(met, 1);
    const double third = 1.0 / 3.0;

    // ------------------------------------------------------------ Valencia
    // mat: sqrt(gamma) times E, S_i, E + S, S^ij, Z v_i v_j - b_i b_j
    double S_u[3];  // sqrt(gamma) gammatilde^ij S_j
    {
        double S_d[3];
#pragma unroll
        for (int i = 0; i < 3; i++) S_d[i] = LD(mat, 1 + i);
#pragma unroll
        for (int i = 0; i < 3; i++)
            S_u[i] = gti[SI(i, 0)] * S_d[0] + gti[SI(i, 1)] * S_d[1] + gti[SI(i, 2)] * S_d[2];
        if (!(PART & RHS_B)) {
        } else if (pp.evolve_fluid) {
            double r[8];
#pragma unroll
            for (int v = 0; v < 8; v++)
                r[v] = DIVP == 1 ? -LD(divF, v) : -(LD(divF, v) + LD(divF, 8 + v) + LD(divF, 16 + v));
            // V^ij = 1/2 alpha e^{4phi} S^ij, twice that off the diagonal (symmetric sums)
            const double ae = alpha * LD(met, 0), hae = 0.5 * ae;
            double V[6], tr = 0.0, VA = 0.0;
#pragma unroll
            for (int i = 0; i < 3; i++)
#pragma unroll
                for (int j = i; j < 3; j++) {
                    const int q = SI(i, j);
                    V[q] = (i == j ? hae : ae) * LD(mat, 5 + q);
                    tr = fma(V[q], gt[q], tr);
                    VA = fma(V[q], At[q], VA);
                }
            const double E = LD(mat, 0), f4 = 4.0 * tr;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                // d_k gamma_ij = e^{4phi} (d_k gammatilde_ij + 4 gammatilde_ij d_k phi)
                double s = r[1 + k];
#pragma unroll
                for (int q = 0; q < 6; q++) s = fma(V[q], dgt[k][q], s);
                s = fma(f4, dphi[k], s);
#pragma unroll
                for (int i = 0; i < 3; i++) s = fma(S_d[i], dbe[k][i], s);
                r[1 + k] = fma(-E, dal[k], s);
            }
            // alpha S^ij K_ij - S^i d_i alpha, K_ij = e^{4phi} (Atilde_ij + gammatilde_ij K / 3)
            r[4] = fma(2.0, fma(K * third, tr, VA), r[4]);
            r[4] = fma(-e4m, S_u[0] * dal[0] + S_u[1] * dal[1] + S_u[2] * dal[2], r[4]);
            if (pp.glm) {
                // GLM cleaning: see k_rhs
                double dpsi[3];
#pragma unroll
                for (int k = 0; k < 3; k++) dpsi[k] = D1(N_D1, k);
                const double as = alpha * LD(met, 2) * e4m;
#pragma unroll
                for (int i = 0; i < 3; i++)
                    r[5 + i] -= as * (gti[SI(i, 0)] * dpsi[0] + gti[SI(i, 1)] * dpsi[1] + gti[SI(i, 2)] * dpsi[2]);
                emit(V_PSI, -alpha * fma(pp.glm_ch2 * divB[p], LD(met, 9), LD(Us, V_PSI) * pp.glm_itau));
            }
            // interface penalty (Rusanov flux, strong form) at duplicated element-end nodes
            int side = 0;
            if (ir == d.Nr - 1 && d.iface_next[e]) side = +1;
            if (ir == 0 && e > 0 && d.iface_next[e - 1]) side = -1;
            if (side != 0) {
                const long long pl = side > 0 ? p : p - d.NtNp, pr = pl + d.NtNp;
                const double hl = 0.5 * fmax(lam[pl], lam[pr]);
                const double fac = r_scale[e] / pp.w_end;
#pragma unroll
                for (int v = 0; v < 8; v++) {
                    const double FL = flux[v * P + pl], FR = flux[v * P + pr];
                    const double UL = Us[(V_D + v) * P + pl], UR = Us[(V_D + v) * P + pr];
                    const double Fs = 0.5 * (FL + FR) - hl * (UR - UL);
                    r[v] = side > 0 ? fma(FL - Fs, fac, r[v]) : fma(Fs - FR, fac, r[v]);
                }
            }
#pragma unroll
            for (int v = 0; v < 8; v++) emit(V_D + v, r[v]);
        } else {
            for (int v = V_D; v < NV + pp.glm; v++) emit(v, 0.0);
        }
    }
    if (!pp.evolve_metric) {
        for (int v = 0; v < N_BSSN; v++) emit(v, 0.0);
        return;
    }

    // ------------------------------------------------------------ gammatilde, phi, lapse, shift
    const double bdal = beta[0] * dal[0] + beta[1] * dal[1] + beta[2] * dal[2];
    const double aK = alpha * K;
    const double divb = dbe[0][0] + dbe[1][1] + dbe[2][2], db3 = divb * third;
    emit(V_PHI, fma(-1.0 / 6.0, aK, fma(0.5, db3, beta[0] * dphi[0] + beta[1] * dphi[1] + beta[2] * dphi[2])));
    if (pp.gauge == 0) {
        emit(V_ALPHA, fma(-2.0, aK, bdal));
#pragma unroll
        for (int i = 0; i < 3; i++) emit(V_BETA + i, 0.75 * LD(Us, V_BG + i));
    } else {
        emit(V_ALPHA, 0.0);
#pragma unroll
        for (int i = 0; i < 3; i++) emit(V_BETA + i, 0.0);
    }
    // trace-free d_j beta^k: carries the -2/3 div beta terms of the conformal tensors
#pragma unroll
    for (int i = 0; i < 3; i++) dbe[i][i] -= db3;
    const double m2a = -2.0 * alpha;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            const int q = SI(i, j);
            double s = m2a * At[q];
#pragma unroll
            for (int k = 0; k < 3; k++) s = fma(beta[k], dgt[k][q], s);
            if (i == j) {
                s = fma(2.0, gt[SI(i, 0)] * dbe[i][0] + gt[SI(i, 1)] * dbe[i][1] + gt[SI(i, 2)] * dbe[i][2], s);
            } else {
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    s = fma(gt[SI(i, k)], dbe[j][k], s);
                    s = fma(gt[SI(j, k)], dbe[i][k], s);
                }
            }
            emit(V_GT + q, s);
        }

    // ------------------------------------------------------------ Christoffel symbols, Ricci tensor
    double Cu[3][6], Gd[3], R2[6], gw[6];  // Gammatilde^k_ij, its trace, 2 Rtilde_ij, weighted inverse
    {
        double C[3][6];
#pragma unroll
        for (int k = 0; k < 3; k++)
#pragma unroll
            for (int i = 0; i < 3; i++)
#pragma unroll
                for (int j = i; j < 3; j++) {
                    const int q = SI(i, j);
                    if (k == i) C[k][q] = dgt[j][SI(i, i)];
                    else if (k == j) C[k][q] = dgt[i][SI(j, j)];
                    else if (i == j) C[k][q] = fma(2.0, dgt[i][SI(k, i)], -dgt[k][q]);
                    else C[k][q] = dgt[i][SI(k, j)] + dgt[j][SI(k, i)] - dgt[k][q];
                }
        double hg[6];
#pragma unroll
        for (int q = 0; q < 6; q++) hg[q] = 0.5 * gti[q];
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++) gw[SI(i, j)] = i == j ? gti[SI(i, j)] : gti[SI(i, j)] + gti[SI(i, j)];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < 6; q++) {
                Cu[k][q] = hg[SI(k, 0)] * C[0][q] + hg[SI(k, 1)] * C[1][q] + hg[SI(k, 2)] * C[2][q];
                s = q == 0 ? gw[0] * Cu[k][0] : fma(gw[q], Cu[k][q], s);
            }
            Gd[k] = s;
        }
#pragma unroll
        for (int q = 0; q < 6; q++) R2[q] = Gd[0] * dgt[0][q] + Gd[1] * dgt[1][q] + Gd[2] * dgt[2][q];
        // the quadratic part, gti^lm (Gamma^k_li Gamma_jkm + Gamma^k_lj Gamma_ikm + Gamma^k_im Gamma_klj)
        // twice: P_ij + P_ji + Q_ij with T_i^km = Gamma^k_il gti^lm, P_ij = T_i^km C_jkm (T
        // symmetrised: C is symmetric there), Q_ij = T_i^km C_kmj (symmetric in i, j)
#pragma unroll
        for (int i = 0; i < 3; i++) {
            double T[3][3];
#pragma unroll
            for (int k = 0; k < 3; k++)
#pragma unroll
                for (int m = 0; m < 3; m++)
                    T[k][m] = Cu[k][SI(i, 0)] * gti[SI(0, m)] + Cu[k][SI(i, 1)] * gti[SI(1, m)] +
                              Cu[k][SI(i, 2)] * gti[SI(2, m)];
            const double t01 = T[0][1] + T[1][0], t02 = T[0][2] + T[2][0], t12 = T[1][2] + T[2][1];
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const int q = SI(i, j);
                const double* c = C[j];
                if (i == j) {
                    const double s = T[0][0] * c[0] + t01 * c[1] + t02 * c[2] + T[1][1] * c[3] + t12 * c[4] + T[2][2] * c[5];
                    R2[q] = fma(2.0, s, R2[q]);
                } else {
                    R2[q] = fma(T[0][0], c[0], R2[q]);
                    R2[q] = fma(t01, c[1], R2[q]);
                    R2[q] = fma(t02, c[2], R2[q]);
                    R2[q] = fma(T[1][1], c[3], R2[q]);
                    R2[q] = fma(t12, c[4], R2[q]);
                    R2[q] = fma(T[2][2], c[5], R2[q]);
                }
                if (j >= i)
#pragma unroll
                    for (int k = 0; k < 3; k++)
#pragma unroll
                        for (int m = 0; m < 3; m++) R2[q] = fma(T[k][m], C[k][SI(m, j)], R2[q]);
            }
        }
    }
    double dGam[3][3];
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int i = 0; i < 3; i++) dGam[k][i] = D1(V_GAM + i, k);

    // ------------------------------------------------------------ X_ij, trace-free part
    // X_ij = -D_i D_j alpha + alpha (R_ij - 8 pi S_ij) up to multiples of gammatilde_ij:
    // -d_i d_j alpha - 2 alpha d_i d_j phi + Gamma^k_ij (d_k alpha + 2 alpha d_k phi)
    // + 2 d_i phi (d_j alpha + alpha d_j phi) + (i <-> j) + alpha (Rtilde_ij - 8 pi S_ij)
    const double m8 = 8.0 * 3.141592653589793 * alpha * LD(met, 9);
    double X[6], trX = 0.0, ddal_tr = 0.0, ddphi_tr = 0.0;
    {
        const double ha = 0.5 * alpha;
        double qv[3], pv[3], tv[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            qv[k] = fma(-m2a, dphi[k], dal[k]);
            tv[k] = fma(alpha, dphi[k], dal[k]);
            pv[k] = 2.0 * dphi[k];
        }
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++) {
                const int q = SI(i, j);
                double R = R2[q];
#pragma unroll
                for (int l = 0; l < 6; l++) R = fma(-gw[l], D2(q, l), R);
                if (i == j) {
                    R = fma(2.0, gt[SI(i, 0)] * dGam[i][0] + gt[SI(i, 1)] * dGam[i][1] + gt[SI(i, 2)] * dGam[i][2], R);
                } else {
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        R = fma(gt[SI(k, i)], dGam[j][k], R);
                        R = fma(gt[SI(k, j)], dGam[i][k], R);
                    }
                }
                const double dda = D2(7, q), ddp = D2(6, q);
                ddal_tr = fma(gw[q], dda, ddal_tr);
                if (HAM) ddphi_tr = fma(gw[q], ddp, ddphi_tr);
                double s = fma(m2a, ddp, -dda);
#pragma unroll
                for (int k = 0; k < 3; k++) s = fma(Cu[k][q], qv[k], s);
                s = fma(pv[i], tv[j], s);
                s = fma(pv[j], tv[i], s);
                s = fma(ha, R, s);
                X[q] = fma(-m8, LD(mat, 11 + q), s);
                trX = fma(gw[q], X[q], trX);
            }
    }
    // gammatilde^ij d_i phi d_j alpha; D^i D_i alpha
    double dphi_u[3];
#pragma unroll
    for (int k = 0; k < 3; k++)
        dphi_u[k] = gti[SI(k, 0)] * dphi[0] + gti[SI(k, 1)] * dphi[1] + gti[SI(k, 2)] * dphi[2];
    const double gpa = dphi_u[0] * dal[0] + dphi_u[1] * dal[1] + dphi_u[2] * dal[2];
    double lap = fma(2.0, gpa, ddal_tr);
#pragma unroll
    for (int k = 0; k < 3; k++) lap = fma(-Gd[k], dal[k], lap);
    lap *= e4m;

    // ------------------------------------------------------------ Atilde, K
    double Aud[3][3], Auu[6], AA = 0.0;  // Atilde^k_j; Atilde^ij (twice off the diagonal below)
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int j = 0; j < 3; j++)
            Aud[k][j] = gti[SI(k, 0)] * At[SI(0, j)] + gti[SI(k, 1)] * At[SI(1, j)] + gti[SI(k, 2)] * At[SI(2, j)];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++)
            Auu[SI(i, j)] = Aud[i][0] * gti[SI(0, j)] + Aud[i][1] * gti[SI(1, j)] + Aud[i][2] * gti[SI(2, j)];
    // 2 alpha (Atilde^ij (6 d_j phi) ) - 2 Atilde^ij d_j alpha
    double rG[3];
    {
        double w[3];
        const double a12 = 12.0 * alpha;
#pragma unroll
        for (int k = 0; k < 3; k++) w[k] = fma(a12, dphi[k], -2.0 * dal[k]);
#pragma unroll
        for (int i = 0; i < 3; i++) rG[i] = Auu[SI(i, 0)] * w[0] + Auu[SI(i, 1)] * w[1] + Auu[SI(i, 2)] * w[2];
    }
    Auu[1] += Auu[1];
    Auu[2] += Auu[2];
    Auu[4] += Auu[4];
#pragma unroll
    for (int q = 0; q < 6; q++) AA = fma(At[q], Auu[q], AA);
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 6; q++) s = q == 0 ? Cu[i][0] * Auu[0] : fma(Cu[i][q], Auu[q], s);
        rG[i] = fma(-m2a, s, rG[i]);
    }
    double dK[3];
#pragma unroll
    for (int k = 0; k < 3; k++) dK[k] = D1(V_K, k);
    {
        double s = fma(alpha, fma(K * third, K, AA), -lap);
        s = fma(0.5 * m8, LD(mat, 4), s);
#pragma unroll
        for (int k = 0; k < 3; k++) s = fma(beta[k], dK[k], s);
        emit(V_K, s);
    }
    if (HAM) {
        // Hamiltonian constraint R + (2/3) K^2 - Atilde.Atilde - 16 pi E with e^{4phi} R =
        // gammatilde^ij R_ij: trX holds alpha (its part without the gammatilde_ij terms) minus
        // the lapse and matter terms, which are taken out again
        double gdp2 = dphi_u[0] * dphi[0] + dphi_u[1] * dphi[1] + dphi_u[2] * dphi[2];
        double lapphi = ddphi_tr, pl = ddal_tr, mt = 0.0;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            lapphi = fma(-Gd[k], dphi[k], lapphi);
            pl = fma(-Gd[k], dal[k], pl);
        }
#pragma unroll
        for (int q = 0; q < 6; q++) mt = fma(gw[q], LD(mat, 11 + q), mt);
        const double trR = (trX + pl - 4.0 * gpa + m8 * mt) / alpha - 6.0 * lapphi - 12.0 * gdp2;
        ham[p] = e4m * trR + 2.0 * third * K * K - AA - 16.0 * 3.141592653589793 * LD(mat, 0) * LD(met, 9);
    }
    {
        const double c1 = -(e4m * trX) * third, hk = 0.5 * aK;
        // d_j beta^k - alpha Atilde^k_j + 1/2 alpha K delta: the Lie, quadratic and K terms of Atilde
        double H[3][3];
#pragma unroll
        for (int j = 0; j < 3; j++)
#pragma unroll
            for (int k = 0; k < 3; k++) {
                H[j][k] = fma(-alpha, Aud[k][j], dbe[j][k]);
                if (j == k) H[j][k] += hk;
            }
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = i; j < 3; j++) {
                const int q = SI(i, j);
                double s = fma(e4m, X[q], c1 * gt[q]);
#pragma unroll
                for (int k = 0; k < 3; k++) s = fma(beta[k], D1(V_AT + q, k), s);
                if (i == j) {
                    s = fma(2.0, At[SI(i, 0)] * H[i][0] + At[SI(i, 1)] * H[i][1] + At[SI(i, 2)] * H[i][2], s);
                } else {
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        s = fma(At[SI(i, k)], H[j][k], s);
                        s = fma(At[SI(j, k)], H[i][k], s);
                    }
                }
                emit(V_AT + q, s);
            }
    }

    // ------------------------------------------------------------ Gammatilde, driver
    {
        const double a43 = -4.0 * third * alpha;
        double v[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            // d_j d_k beta^k
            const double t = D2(8, SI(j, 0)) + D2(9, SI(j, 1)) + D2(10, SI(j, 2));
            v[j] = fma(a43, dK[j], t * third);
        }
#pragma unroll
        for (int i = 0; i < 3; i++) {
            double s = fma(-2.0 * m8, S_u[i], rG[i]);
#pragma unroll
            for (int q = 0; q < 6; q++) s = fma(gw[q], D2(8 + i, q), s);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                s = fma(gti[SI(i, k)], v[k], s);
                s = fma(beta[k], dGam[k][i], s);
                s = fma(-LD(Us, V_GAM + k), dbe[k][i], s);
            }
            s = fma(db3, LD(Us, V_GAM + i), s);
            emit(V_GAM + i, s);
            emit(V_BG + i, pp.gauge == 0 ? fma(-pp.eta, LD(Us, V_BG + i), s) : 0.0);
        }
    }
#undef LD
#undef D1
#undef D2
}

// SPLIT: blockIdx.y = 0 Atilde, 1 the rest; else all
template <int MODE, bool HAM, int DIVP, bool SPLIT>
__global__ void __launch_bounds__(128) k_rhs64(Dims d, PhysParams pp, const double* __restrict__ U0,
                                               const double* __restrict__ Us, const double* __restrict__ flux,
                                               const double* __restrict__ mat, const double* __restrict__ lam,
                                               const double* __restrict__ met, const double* __restrict__ d1,
                                               const double* __restrict__ d2, const double* __restrict__ divF,
                                               const double* __restrict__ divB, const double* __restrict__ r_scale,
                                               const double* __restrict__ dt_dev, RKCoef co,
                                               double* __restrict__ out, double* __restrict__ acc,
                                               double* __restrict__ ham) {
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= d.P) return;
#define NODE_ARGS p, d, pp, U0, Us, flux, mat, lam, met, d1, d2, divF, divB, r_scale, dt_dev, co, out, acc, ham
    if constexpr (SPLIT) {
        if (blockIdx.y == 0) rhs64_node<MODE, HAM, DIVP, RHS_A>(NODE_ARGS);
        else rhs64_node<MODE, HAM, DIVP, RHS_B>(NODE_ARGS);
    } else {
        rhs64_node<MODE, HAM, DIVP, RHS_ALL>(NODE_ARGS);
    }
#undef NODE_ARGS
}

// --------------------------------------------------------------------------- launchers
cudaError_t launch_prep(const Dims& d, const PhysParams& pp, const double* U, double* prim,
                        double* flux, double* tmn, double* lam, unsigned long long* nfail, double* met,
                        cudaStream_t s, int fp32_algebra) {
    int bs = 128;
    long long nb = (d.P + bs - 1) / bs;
    if (fp32_algebra) k_prep<PREP_F32><<<(unsigned)nb, bs, 0, s>>>(d, pp, U, prim, flux, tmn, lam, nfail, met);
    else k_prep<PREP_F64><<<(unsigned)nb, bs, 0, s>>>(d, pp, U, prim, flux, tmn, lam, nfail, met);
    return cudaGetLastError();
}

cudaError_t launch_con2prim(const Dims& d, const PhysParams& pp, const double* U, double* prim,
                            unsigned long long* nfail, cudaStream_t s) {
    int bs = 128;
    long long nb = (d.P + bs - 1) / bs;
    k_prep<PREP_PRIM><<<(unsigned)nb, bs, 0, s>>>(d, pp, U, prim, nullptr, nullptr, nullptr, nfail, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_rhs(const Dims& d, const PhysParams& pp, const double* U0, const double* Us,
                       const double* flux, const double* tmn, const double* lam, const double* met,
                       const void* d1, const void* d2, const void* divF, const void* divB, int deriv_fp32,
                       const double* r_scale_dev, const double* dt_dev, RKCoef co, double* out, double* acc, cudaStream_t s,
                       double* ham, int div_parts) {
    int bs = 128;
    long long nb = (d.P + bs - 1) / bs;
#define RHS_ARGS d, pp, U0, Us, (const float*)flux, (const float*)tmn, lam, met, (const float*)d1, (const float*)d2, (const float*)divF, \
                    (const float*)divB, r_scale_dev, dt_dev, co, out, acc, ham
    if (deriv_fp32) {
        const unsigned g = (unsigned)nb;
        if (ham) k_rhs<0, true><<<g, bs, 0, s>>>(RHS_ARGS);
        else if (co.acc_mode < 0) k_rhs<0, false><<<g, bs, 0, s>>>(RHS_ARGS);
        else if (co.acc_mode > 0) k_rhs<3, false><<<g, bs, 0, s>>>(RHS_ARGS);
        else if (co.a == 0.0 && co.b == 1.0) k_rhs<1, false><<<g, bs, 0, s>>>(RHS_ARGS);
        else k_rhs<2, false><<<g, bs, 0, s>>>(RHS_ARGS);
    } else {
        // two threads per node while that still leaves every SM quarter at most one warp
        int dev = 0, nsm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const bool split = div_parts == 3 && d.P * 2 <= 32LL * 4 * nsm;
        if (split) {   // 32 threads a block: a warp per SM quarter
            bs = 32;
            nb = (d.P + bs - 1) / bs;
        }
        const auto run = [&](auto k, unsigned y) {
            k<<<dim3((unsigned)nb, y), bs, 0, s>>>(d, pp, U0, Us, flux, tmn, lam, met, (const double*)d1, (const double*)d2,
                                                   (const double*)divF, (const double*)divB, r_scale_dev, dt_dev, co, out,
                                                   acc, ham);
        };
        // (a runtime branch on div_parts cost 4 %: the additions were issued either way)
#define RHS64_RUN(MODE) \
        split ? run(k_rhs64<MODE, false, 3, true>, 2) \
              : (div_parts == 3 ? run(k_rhs64<MODE, false, 3, false>, 1) : run(k_rhs64<MODE, false, 1, false>, 1))
        if (ham) div_parts == 3 ? run(k_rhs64<0, true, 3, false>, 1) : run(k_rhs64<0, true, 1, false>, 1);
        else if (co.acc_mode < 0) RHS64_RUN(0);
        else if (co.acc_mode > 0) RHS64_RUN(3);
        else if (co.a == 0.0 && co.b == 1.0) RHS64_RUN(1);
        else RHS64_RUN(2);
#undef RHS64_RUN
    }
#undef RHS_ARGS
    return cudaGetLastError();
}

}  // namespace gk
