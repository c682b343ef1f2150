// gcb_ks.cu -- the covariant coupled step in Kerr-Schild spacetime
// (Sec. 2.3 GREOM, Sec. 2.4 GRGCA, Sec. 3.2 coupling), geometrized units
// c = G = M = 1.  Arithmetic and metric in FP64; field records FP32 or FP64
// (interpolated in their own precision).  Same tile structure as the flat
// push: ballot compaction of each tile into [GCA ..., Boris ..., frozen].
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <climits>

#include "gcb.h"
#include "gcb_internal.h"
#include "real64.cuh"

namespace gcb {
namespace ks {

constexpr int TPB = 128;
constexpr int NWARP = TPB / 32;

// The kernel is bound by the FP64 pipe (86% busy; GB300 issues 2 FP64 lanes
// per SM and clock, and comparisons, conversions and roundings take the same
// slots), so everything below is arranged for the fewest FP64 operations: the
// helpers of real64.cuh, closed forms that share their factors, and in the
// guiding-center iterations the metric's derivative along b only.  Measured
// (GB300, 2^20 particles, FP32 records, local-frame kicks): 1391 -> 1017 pipe
// slots a particle-step, 3.17 -> 2.32 ms (2.27 without counters); 100003 particles, FP64 records,
// global-basis kicks: 382 -> 285 us.

// Kerr-Schild 3+1 quantities (M = 1) at a point:
//   rho^2 = r^2 + a^2 cos^2, z = 2r / rho^2, alpha = (1+z)^-1/2, beta^r = z/(1+z),
//   gamma^{rr} = (r^2 + a^2)/rho^2 - beta^r, gamma^{r phi} = a/rho^2,
//   gamma^{th th} = 1/rho^2, gamma^{ph ph} = 1/(rho^2 sin^2),
//   sqrt(gamma) = rho^2 sin sqrt(1+z); lower() for gamma_ij.
struct Metric {
    double s, c, r, s2, is2;            // sin, cos, r, sin^2, 1/sin^2
    double ra2, rho2, irho2, onez, alpha, beta;   // r^2 + a^2, rho^2, 1/rho^2, 1 + z
    double grr, grp, gpp;               // gamma^{rr}, gamma^{r phi}, gamma^{ph ph}
};

// sin theta, cos theta and log r of a point
struct TrigLog {
    double s, c, lr;
};

__device__ __forceinline__ void trig_log(double r, double th, TrigLog &t)
{
    sincos(th, &t.s, &t.c);
    t.lr = log(r);
}

// The same at (r, th) near a point (r0, th0) whose values t0 are known
// (ir0 = 1/r0): sin and cos by the angle-addition formula with the Maclaurin
// series of sin d and cos d (d = th - th0, through d^7 and d^6), log r =
// log r0 + log(1 + e) (e = r/r0 - 1) by the Mercator series through e^9.  For
// |d| <= 0.02 and |e| <= 0.01 the truncation errors are below 1e-18; farther
// away, or within sin th0 <= 0.05 of a pole (where sin th would lose relative
// precision), the library functions.
__device__ __forceinline__ void trig_log_near(const TrigLog &t0, double r0, double ir0, double th0,
                                              double r, double th, TrigLog &t)
{
    const double d = th - th0;
    const double e = (r - r0) * ir0;
    if (gt_nonneg(fabs(d), 0.02) || gt_nonneg(fabs(e), 0.01) || !gt_nonneg(fabs(t0.s), 0.05)) {
        trig_log(r, th, t);
        return;
    }
    const double d2 = d * d;
    const double sd = fma(d * d2, fma(d2, fma(d2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), d);
    const double cd = fma(d2, fma(d2, fma(d2, -1.0 / 720.0, 1.0 / 24.0), -0.5), 1.0);
    t.s = fma(t0.s, cd, t0.c * sd);
    t.c = fma(t0.c, cd, -t0.s * sd);
    double q = 1.0 / 9.0;
    q = fma(-e, q, 1.0 / 8.0);
    q = fma(-e, q, 1.0 / 7.0);
    q = fma(-e, q, 1.0 / 6.0);
    q = fma(-e, q, 1.0 / 5.0);
    q = fma(-e, q, 0.25);
    q = fma(-e, q, 1.0 / 3.0);
    q = fma(-e, q, 0.5);
    q = fma(-e, q, 1.0);
    t.lr = fma(e, q, t0.lr);
}

// (t: sin and cos of th)
__device__ __forceinline__ void ks_metric(double a, double r, const TrigLog &t, Metric &m)
{
    m.s = t.s;
    m.c = t.c;
    m.r = r;
    m.s2 = t.s * t.s;
    m.is2 = rcp64(m.s2);
    const double r2 = r * r, ac = a * t.c;
    m.ra2 = fma(a, a, r2);
    m.rho2 = fma(ac, ac, r2);
    m.irho2 = rcp64(m.rho2);
    const double z = (r + r) * m.irho2;
    m.onez = 1.0 + z;
    m.alpha = rsqrt64(m.onez);
    m.beta = z * (m.alpha * m.alpha);
    m.grr = fma(m.ra2, m.irho2, -m.beta);
    m.grp = a * m.irho2;
    m.gpp = m.irho2 * m.is2;
}

__device__ __forceinline__ double sqrt_gamma(const Metric &m)
{
    return (m.rho2 * m.s) * (m.onez * m.alpha);
}

// gamma^{ij} u_j for covariant u (indices r, theta, phi)
__device__ __forceinline__ void raise(const Metric &m, const double u[3], double v[3])
{
    v[0] = fma(m.grr, u[0], m.grp * u[2]);
    v[1] = m.irho2 * u[1];
    v[2] = fma(m.grp, u[0], m.gpp * u[2]);
}
// gamma_ij v^j: gamma_rr = 1+z, gamma_rph = -a (1+z) sin^2, gamma_thth = rho^2,
// gamma_phph = (rho^2 + a^2 (1+z) sin^2) sin^2
__device__ __forceinline__ void lower(double a, const Metric &m, const double v[3], double u[3])
{
    u[0] = m.onez * fma(-a * m.s2, v[2], v[0]);
    u[1] = m.rho2 * v[1];
    u[2] = m.s2 * fma(-a, u[0], m.rho2 * v[2]);
}

__device__ __forceinline__ double dot(const double a[3], const double b[3])
{
    return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}

// Local frame of the normal observer: gamma^{ij} = L L^T with L lower
// triangular; for this metric L has L10 = L21 = 0.  Frame components of a
// covariant vector: u^ = L^T u; of a contravariant one: F^ = L^{-1} F.
// (i00, i11, i22: reciprocals of the diagonal, so no conversion divides)
struct Tri {
    double l00, l20, l11, l22, i00, i11, i22;
};
__device__ __forceinline__ void make_tri(const Metric &m, Tri &t)
{
    t.i00 = rsqrt64(m.grr);
    t.l00 = m.grr * t.i00;
    t.l20 = m.grp * t.i00;
    t.i11 = rsqrt64(m.irho2);
    t.l11 = m.irho2 * t.i11;
    const double d22 = fma(-t.l20, t.l20, m.gpp);
    t.i22 = rsqrt64(d22);
    t.l22 = d22 * t.i22;
}
__device__ __forceinline__ void cov_to_frame(const Tri &t, const double u[3], double h[3])
{
    h[0] = t.l00 * u[0] + t.l20 * u[2];
    h[1] = t.l11 * u[1];
    h[2] = t.l22 * u[2];
}
__device__ __forceinline__ void frame_to_cov(const Tri &t, const double h[3], double u[3])
{
    u[2] = h[2] * t.i22;
    u[1] = h[1] * t.i11;
    u[0] = (h[0] - t.l20 * u[2]) * t.i00;
}
__device__ __forceinline__ void con_to_frame(const Tri &t, const double F[3], double h[3])
{
    h[0] = F[0] * t.i00;
    h[1] = F[1] * t.i11;
    h[2] = (F[2] - t.l20 * h[0]) * t.i22;
}

struct StepCfg {
    double a, dt, f_rho, f_E2, r_in, r_out, tol;
    int max_iter, fixed_iters, force, mu_mode, basis;
};

template <typename FT>
struct KsGrid {
    const FT *rec;
    int stride, nr, nth;
    double logr0, inv_dlogr, inv_dth;
    const double *dl;
};

// Cell of coordinate s (in cells), clamped to [0, n - 1], and the position in
// it (points just outside extrapolate the edge cell).
__device__ __forceinline__ void ks_axis(double s, int n, int &i, double &t)
{
    double f = floor64(s, INT_MAX, i);
    if ((unsigned)i >= (unsigned)n) {
        i = i < 0 ? 0 : n - 1;
        f = (double)i;
    }
    t = s - f;
}
template <typename FT>
__device__ __forceinline__ void ks_cell(const KsGrid<FT> &g, double lr, double th, int &i, int &j,
                                        double &tr, double &tt)
{
    ks_axis((lr - g.logr0) * g.inv_dlogr, g.nr - 1, i, tr);
    ks_axis(th * g.inv_dth, g.nth - 1, j, tt);
}

// linear-shape-function gather of D^i, B^i (Sec. 4 intro) in the record type
// (lr: log r)
template <typename FT>
__device__ __forceinline__ void ks_gather(const KsGrid<FT> &g, double lr, double th, double D[3],
                                          double B[3])
{
    int i, j;
    double tr, tt;
    ks_cell(g, lr, th, i, j, tr, tt);
    FT acc[6] = {FT(0), FT(0), FT(0), FT(0), FT(0), FT(0)};
    const FT ftr = (FT)tr, ftt = (FT)tt;
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const int oi = o & 1, oj = o >> 1;
        const FT W = (oi ? ftr : FT(1) - ftr) * (oj ? ftt : FT(1) - ftt);
        const FT *rp = g.rec + ((size_t)(j + oj) * g.nr + (i + oi)) * g.stride;
#pragma unroll
        for (int k = 0; k < 6; ++k) acc[k] = fma(__ldg(rp + k), W, acc[k]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) { D[k] = widen<false>(acc[k]); B[k] = widen<false>(acc[3 + k]); }
}

__device__ __forceinline__ void cross(const double a[3], const double b[3], double x[3])
{
    x[0] = fma(a[1], b[2], -a[2] * b[1]);
    x[1] = fma(a[2], b[0], -a[0] * b[2]);
    x[2] = fma(a[0], b[1], -a[1] * b[0]);
}

// Boris push in the local frame over proper time dtau (Sec. 2.3 step 1 / 3)
__device__ __forceinline__ void boris_local(const double E[3], const double B[3], double qm,
                                            double dtau, double u[3])
{
    const double h = 0.5 * qm * dtau;
    double um[3], t[3], x[3], up[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) um[k] = fma(h, E[k], u[k]);
    const double hg = h * rsqrt64(1.0 + dot(um, um));
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = hg * B[k];
    const double sf = 2.0 * rcp64(1.0 + dot(t, t));
    cross(um, t, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = um[k] + x[k];
    cross(up, t, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = fma(h, E[k], fma(sf, x[k], um[k]));
}

// The same kick in the global coordinate basis (the option of Sec. 2.3 and
// 2.4 that needs no tetrad): covariant u and D_i = gamma_ij D^j, contravariant
// B^k, t^k = h B^k / Gamma-, |t|^2 = gamma_ij t^i t^j and cross products
// (v x t)_i = sqrt(gamma) [ijk] v^j t^k of raised vectors; the frame form
// maps onto this one because det L = 1 / sqrt(gamma).
__device__ __forceinline__ void boris_global(double a, const Metric &m, const double D[3],
                                             const double B[3], double qm, double dtau, double u[3])
{
    const double h = 0.5 * qm * dtau;
    double Dd[3], Bd[3], um[3], v[3], t[3], x[3], w[3];
    lower(a, m, D, Dd);
    lower(a, m, B, Bd);
#pragma unroll
    for (int k = 0; k < 3; ++k) um[k] = fma(h, Dd[k], u[k]);
    raise(m, um, v);
    const double hg = h * rsqrt64(1.0 + dot(um, v));
    const double sf = 2.0 * rcp64(fma(hg * hg, dot(Bd, B), 1.0));
    const double sg = sqrt_gamma(m) * hg;
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = sg * B[k];
    cross(v, t, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = um[k] + x[k];
    raise(m, w, v);
    cross(v, t, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = fma(h, Dd[k], fma(sf, x[k], um[k]));
}

// One GREOM half kick over alpha dt / 2 at x, in the basis c.basis selects
// (t: trigonometry and log r at x; m: the metric at x, returned for reuse)
template <typename FT>
__device__ __forceinline__ void half_kick(const KsGrid<FT> &g, const StepCfg &c, double qm,
                                          const double x[3], const TrigLog &t, double u[3], Metric &m)
{
    ks_metric(c.a, x[0], t, m);
    double D[3], B[3];
    ks_gather(g, t.lr, x[1], D, B);
    if (c.basis == GCB_KS_GLOBAL) {
        boris_global(c.a, m, D, B, qm, 0.5 * c.dt * m.alpha, u);
        return;
    }
    double Dh[3], Bh[3], uh[3];
    Tri tri;
    make_tri(m, tri);
    cov_to_frame(tri, u, uh);
    con_to_frame(tri, D, Dh);
    con_to_frame(tri, B, Bh);
    boris_local(Dh, Bh, qm, 0.5 * c.dt * m.alpha, uh);
    frame_to_cov(tri, uh, u);
}

// n^i G_i for a direction (nr, nt) in (r, theta), where
// G_i = -Gamma d_i alpha + u_j d_i beta^j - alpha u_j u_k d_i gamma^{jk} / (2 Gamma)
// (G_phi = 0: axisymmetric; iGam = 1 / Gam).  With d the derivative along n:
// d alpha = -alpha^3 dz/2, d beta^r = dz/(1+z)^2 and, from u_j u_k gamma^{jk} =
// Q/rho^2 - beta^r u_r^2, Q = (r^2 + a^2) u_r^2 + 2a u_r u_phi + u_theta^2 +
// u_phi^2/sin^2.  One direction costs half of both components.
// (WR, WT: whether nr and nt are given; nt = 1 or nr = 1 alone for GREOM)
template <bool WR, bool WT>
__device__ __forceinline__ double geodesic_G(double a, const Metric &m, const double u[3], double Gam,
                                             double iGam, double nr, double nt)
{
    const double r2 = m.r + m.r;
    const double u02 = u[0] * u[0], us = u[2] * m.is2;
    const double Q = fma(us, u[2], fma(u[0], fma(m.ra2, u[0], (a + a) * u[2]), u[1] * u[1]));
    const double sc = (m.s + m.s) * m.c;               // d sin^2 / d theta
    double drho2 = 0.0, dQ = 0.0, dz = 0.0;
    if (WR) {
        const double k = WT ? r2 * nr : r2;
        drho2 = k;
        dQ = k * u02;
        dz = WT ? (nr + nr) * m.irho2 : m.irho2 + m.irho2;
    }
    if (WT) {
        const double k = WR ? sc * nt : sc;
        drho2 = WR ? fma(-a * a, k, drho2) : -a * a * k;
        dQ = WR ? fma(-k, us * us, dQ) : -k * (us * us);
    }
    const double di = -drho2 * (m.irho2 * m.irho2);    // d (1/rho^2)
    dz = WR ? fma(r2, di, dz) : r2 * di;
    const double a2 = m.alpha * m.alpha;
    const double db = dz * (a2 * a2);
    const double duu = fma(di, Q, fma(m.irho2, dQ, -db * u02));
    const double ha = 0.5 * m.alpha;
    return fma(ha * a2 * dz, Gam, fma(u[0], db, -(ha * iGam) * duu));
}

__device__ __forceinline__ bool imr_done(const StepCfg &c, int iters, double res, bool &nonconv)
{
    if (c.fixed_iters > 0) return iters >= c.fixed_iters;
    if (gt_nonneg(c.tol, res)) return true;
    if (iters >= c.max_iter) { nonconv = true; return true; }
    return false;
}
// (a NaN change never converges)
__device__ __forceinline__ void max_change(double &res, double d)
{
    const double e = fabs(d);
    res = gt_nonneg(e, res) ? e : res;
}

// GREOM: half kick, implicit midpoint for (x, u) (no field inside), half kick.
// (t0: trigonometry and log r at x^n; mfin: the metric at x^{n+1})
template <typename FT>
__device__ void greom_step(const KsGrid<FT> &g, const StepCfg &c, double qm, double x[3],
                           double u[3], const TrigLog &t0, int &iters, bool &nonconv, Metric &mfin)
{
    const double ir0 = rcp64(x[0]);
    double up[3] = {u[0], u[1], u[2]};
    half_kick(g, c, qm, x, t0, up, mfin);
    double xk[3] = {x[0], x[1], x[2]}, wk[3] = {up[0], up[1], up[2]};
    iters = 0;
    nonconv = false;
    for (;;) {
        double xb[3], ub[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) { xb[k] = 0.5 * (xk[k] + x[k]); ub[k] = 0.5 * (wk[k] + up[k]); }
        TrigLog tb;
        trig_log_near(t0, x[0], ir0, x[1], xb[0], xb[1], tb);
        Metric m;
        ks_metric(c.a, xb[0], tb, m);
        double v[3];
        raise(m, ub, v);
        const double G2 = 1.0 + dot(ub, v);
        const double iGam = rsqrt64(G2), Gam = G2 * iGam;
        const double G[2] = {geodesic_G<true, false>(c.a, m, ub, Gam, iGam, 1.0, 0.0),
                             geodesic_G<false, true>(c.a, m, ub, Gam, iGam, 0.0, 1.0)};
        const double f = m.alpha * iGam;
        const double V[3] = {fma(f, v[0], -m.beta), f * v[1], f * v[2]};
        double res = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double xn = fma(c.dt, V[k], x[k]);
            const double wn = k < 2 ? fma(c.dt, G[k < 2 ? k : 0], up[k]) : up[k];
            max_change(res, xn - xk[k]);
            if (k < 2) max_change(res, wn - wk[k]);
            xk[k] = xn;
            wk[k] = wn;
        }
        ++iters;
        if (imr_done(c, iters, res, nonconv)) break;
    }
    TrigLog t1;
    trig_log_near(t0, x[0], ir0, x[1], xk[0], xk[1], t1);
    half_kick(g, c, qm, xk, t1, wk, mfin);
#pragma unroll
    for (int k = 0; k < 3; ++k) { x[k] = xk[k]; u[k] = wk[k]; }
}

// GRGCA frame at a point (Sec. 2.4): B contravariant and covariant, ib = 1/|B|,
// v_E covariant and contravariant, om = 1 - v_E^2, kap = 1/sqrt(om),
// Dpar = D.b.
struct GFrame {
    Metric m;
    double B[3], Bd[3], ib, B2, vE[3], vu[3], om, kap, Dpar;
    bool ok;
    __device__ __forceinline__ double Bk() const { return B2 * ib * kap; }    // |B| kappa
};

// (t: trigonometry and log r at R; D2: D_i D^i, for the switch)
template <typename FT, bool SW = false>
__device__ __forceinline__ void gr_frame(const KsGrid<FT> &g, double a, const double R[3],
                                         const TrigLog &t, GFrame &F, double *D2 = nullptr)
{
    ks_metric(a, R[0], t, F.m);
    double D[3];
    ks_gather(g, t.lr, R[1], D, F.B);
    lower(a, F.m, F.B, F.Bd);
    F.B2 = dot(F.Bd, F.B);
    F.ib = rsqrt64(F.B2);
    const double sg = sqrt_gamma(F.m) * (F.ib * F.ib);
    double x[3];
    cross(D, F.B, x);
#pragma unroll
    for (int i = 0; i < 3; ++i) F.vE[i] = sg * x[i];
    raise(F.m, F.vE, F.vu);
    F.om = 1.0 - dot(F.vE, F.vu);
    F.ok = !not_pos_normal(F.B2) && !not_pos_normal(F.om);
    F.kap = rsqrt64(F.om);
    F.Dpar = dot(D, F.Bd) * F.ib;
    if constexpr (SW) {
        double Dd[3];
        lower(a, F.m, D, Dd);
        *D2 = dot(D, Dd);
    }
}

// The frame at x^n kept between the switch and the step: the values a step
// reads, one shared-memory row each (sin, cos and log r beside it, s_T; r and
// sin^2 from those).
constexpr int NFR = 27;

__device__ __forceinline__ void frame_store(double (*s)[TPB], int t, const GFrame &F)
{
    const double v[NFR] = {F.m.is2, F.m.ra2, F.m.rho2, F.m.irho2, F.m.onez, F.m.alpha, F.m.beta,
                           F.m.grr, F.m.grp, F.m.gpp, F.B[0], F.B[1], F.B[2], F.Bd[0], F.Bd[1],
                           F.Bd[2], F.ib, F.B2, F.vE[0], F.vE[1], F.vE[2], F.vu[0], F.vu[1],
                           F.vu[2], F.om, F.kap, F.Dpar};
#pragma unroll
    for (int k = 0; k < NFR; ++k) s[k][t] = v[k];
}

__device__ __forceinline__ void frame_load(const double (*s)[TPB], int t, double r, const TrigLog &tl,
                                           GFrame &F)
{
    double v[NFR];
#pragma unroll
    for (int k = 0; k < NFR; ++k) v[k] = s[k][t];
    F.m.s = tl.s; F.m.c = tl.c; F.m.r = r; F.m.s2 = tl.s * tl.s;
    F.m.is2 = v[0]; F.m.ra2 = v[1]; F.m.rho2 = v[2]; F.m.irho2 = v[3]; F.m.onez = v[4];
    F.m.alpha = v[5]; F.m.beta = v[6]; F.m.grr = v[7]; F.m.grp = v[8]; F.m.gpp = v[9];
    F.ib = v[16]; F.B2 = v[17]; F.om = v[24]; F.kap = v[25]; F.Dpar = v[26];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        F.B[k] = v[10 + k];
        F.Bd[k] = v[13 + k];
        F.vE[k] = v[18 + k];
        F.vu[k] = v[21 + k];
    }
}

// GRGCA: half kick of u_par by D_par, implicit midpoint on (R, u_par) with the
// full velocity rebuilt at the midpoint, half kick (Sec. 2.4 steps 1-3).
// ug: the gyrating momentum at x^n (covariant, its direction kept), up2 = u_g^2,
// mu2 = 2 mu/m = u_g^2/(|B| kappa), iBk = 1/(|B| kappa) there.
// (Fb: the frame at x^n on entry, which is also the first iterate's midpoint;
// the frame at R^{n+1} on return)
template <typename FT>
__device__ bool grgca_step(const KsGrid<FT> &g, const StepCfg &c, double qm, GFrame &Fb,
                           const TrigLog &t0, double R[3], double &upar, double mu2, double up2,
                           double iBk, const double ug[3], int &iters, bool &nonconv)
{
    const double ir0 = rcp64(R[0]);
    const double hq = 0.5 * c.dt * qm, hdt = 0.5 * c.dt;
    const double u1 = fma(hq * Fb.m.alpha, Fb.Dpar, upar);
    double Rk[3] = {R[0], R[1], R[2]}, wk = u1;
    iters = 0;
    nonconv = false;
    bool okall = Fb.ok;
    for (;;) {
        const double ub = 0.5 * (wk + u1);
        const double Bk = Fb.Bk();
        const double G2 = fma(ub, ub, 1.0) + (c.mu_mode ? up2 : mu2 * Bk);
        const double rg = rsqrt64(G2);
        const double Gam = Fb.kap * (G2 * rg);
        const double iGam = rg * (Fb.om * Fb.kap);
        const double sc = c.mu_mode ? 1.0 : sqrt64(Bk * iBk);   // u_g's growth
        const double ubb = ub * Fb.ib, uv = ubb * iGam;
        double uf[3], V[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            uf[i] = fma(ubb, Fb.Bd[i], fma(Fb.vE[i], Gam, sc * ug[i]));
            V[i] = Fb.m.alpha * fma(uv, Fb.B[i], Fb.vu[i]);
        }
        V[0] -= Fb.m.beta;
        const double Gb = Fb.ib * geodesic_G<true, true>(c.a, Fb.m, uf, Gam, iGam, Fb.B[0], Fb.B[1]);
        double res = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double rn = fma(c.dt, V[k], R[k]);
            max_change(res, rn - Rk[k]);
            Rk[k] = rn;
        }
        const double wn = fma(c.dt, Gb, u1);
        max_change(res, wn - wk);
        wk = wn;
        ++iters;
        if (imr_done(c, iters, res, nonconv)) break;
        // the next iterate's midpoint (Rk + R)/2 and its frame
        double Rb[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) Rb[k] = fma(hdt, V[k], R[k]);
        TrigLog tb;
        trig_log_near(t0, R[0], ir0, R[1], Rb[0], Rb[1], tb);
        gr_frame(g, c.a, Rb, tb, Fb);
        okall = okall && Fb.ok;
    }
    if (!okall) return false;
    TrigLog t1;
    trig_log_near(t0, R[0], ir0, R[1], Rk[0], Rk[1], t1);
    gr_frame(g, c.a, Rk, t1, Fb);   // also the reconstruction's frame
    if (!Fb.ok) return false;
    upar = fma(hq * Fb.m.alpha, Fb.Dpar, wk);
#pragma unroll
    for (int k = 0; k < 3; ++k) R[k] = Rk[k];
    return true;
}

struct Args {
    int64_t np;
    const double *xin[3], *uin[3];
    const uint8_t *flagsin;
    const int64_t *pidin;
    double *x[3], *u[3];
    uint8_t *flags;
    int64_t *pid;
    double qm[4];
    StepCfg c;
    unsigned long long *stats;
};

// one coupled covariant step of one particle (Sec. 3.2); returns the branch
// taken (0 GCA, 1 GREOM) and fills the flag bits
// (F: the frame at x^n, overwritten; mfin: the metric at the new position,
// before any pole reflection, which leaves it unchanged: it depends on theta
// through sin^2 and cos^2 only)
template <typename FT>
__device__ int ks_particle(const KsGrid<FT> &g, const StepCfg &c, double qm, int S, GFrame &F,
                           const TrigLog &t0, double x[3], double u[3], int &iters, bool &nonconv,
                           bool &fail, Metric &mfin)
{
    fail = false;
    if (S == 0) {
        if (F.ok) {
            // decomposition at R^n = x^n with Gamma of the full u (Sec. 3.2)
            double v[3], ug[3];
            raise(F.m, u, v);
            const double Gfull = sqrt64(1.0 + dot(u, v));
            double upar = dot(u, F.B) * F.ib;
            const double upb = upar * F.ib;
#pragma unroll
            for (int i = 0; i < 3; ++i) ug[i] = fma(-Gfull, F.vE[i], fma(-upb, F.Bd[i], u[i]));
            raise(F.m, ug, v);
            const double up2 = fmax(dot(ug, v), 0.0);
            const double iBk = F.ib * (F.om * F.kap);
            const double mu2 = up2 * iBk;
            double R[3] = {x[0], x[1], x[2]};
            if (grgca_step(g, c, qm, F, t0, R, upar, mu2, up2, iBk, ug, iters, nonconv)) {
                // reconstruction at R^{n+1} (the step's frame there), gyration
                // direction kept
                const double Bk = F.Bk();
                const double G1 = F.kap * sqrt64(fma(upar, upar, 1.0) + (c.mu_mode ? up2 : mu2 * Bk));
                const double sc = c.mu_mode ? 1.0 : sqrt64(Bk * iBk);
                const double ubb = upar * F.ib;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    u[i] = fma(ubb, F.Bd[i], fma(F.vE[i], G1, sc * ug[i]));
                    x[i] = R[i];
                }
                mfin = F.m;
                return 0;
            }
        }
        fail = true;
    }
    greom_step(g, c, qm, x, u, t0, iters, nonconv, mfin);
    return 1;
}

// Three resident blocks per SM (at most 170 registers a thread).
// STATS: with the counters (a.stats), else none are kept.
template <typename FT, bool STATS>
__global__ void __launch_bounds__(TPB, 3) k_push_ks(const KsGrid<FT> g, const Args a)
{
    __shared__ double s_x[3][TPB], s_u[3][TPB];
    __shared__ double s_F[NFR][TPB];
    __shared__ double s_T[3][TPB];   // sin theta, cos theta, log r at x^n
    __shared__ uint8_t s_fl[TPB], s_ok[TPB];
    __shared__ unsigned short s_perm[TPB];
    __shared__ int s_wc[2][NWARP];
    __shared__ unsigned long long s_acc[ST_COUNT];
    __shared__ double s_ek;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (STATS && tid < ST_COUNT) s_acc[tid] = 0ull;
    if (STATS && tid == 0) s_ek = 0.0;
    unsigned nb = 0, ng = 0, tg = 0, tb = 0, nc = 0, gf = 0, nf = 0, si = 0, mi = 0;
    unsigned ne = 0;   // frozen after leaving [r_in, r_out]
    double ek = 0.0;
    const double PI = 3.141592653589793;

    const int64_t ntiles = (a.np + TPB - 1) / TPB;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t i = tile * TPB + tid;
        const bool valid = i < a.np;
        int cls = 2;
        uint8_t fl = 0;
        double xs[3] = {0, 0, 0}, us[3] = {0, 0, 0};
        __syncthreads();  // the previous tile's slots are no longer read
        s_ok[tid] = 0;
        if (valid) {
            fl = a.flagsin[i];
            bool fin = true;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                xs[k] = a.xin[k][i];
                us[k] = a.uin[k][i];
                fin = fin && finite64(xs[k]) && finite64(us[k]);
            }
            const uint8_t fl_in = fl;
            if (!fin && !(fl & GCB_FLAG_NONFINITE)) { fl |= GCB_FLAG_NONFINITE; }
            if (fin && !(fl & (GCB_FLAG_NONFINITE | GCB_FLAG_EXITED))) {
                // switch (Sec. 3, 4.2): Gamma/(|q/m| B) against the cell size of
                // Eq. (volint), |D^|/|B^| against f_E; squared, division-free
                TrigLog t;
                trig_log(xs[0], xs[1], t);
                GFrame F;
                double D2;
                gr_frame<FT, true>(g, a.c.a, xs, t, F, &D2);
                frame_store(s_F, tid, F);   // the step starts from this frame
                s_T[0][tid] = t.s;
                s_T[1][tid] = t.c;
                s_T[2][tid] = t.lr;
                s_ok[tid] = F.ok ? 1 : 0;
                double v[3];
                raise(F.m, us, v);
                const double G2 = 1.0 + dot(us, v);
                int ci, cj;
                double tr, tt;
                ks_cell(g, t.lr, xs[1], ci, cj, tr, tt);
                const double dl = g.dl[(size_t)cj * (g.nr - 1) + ci];
                const double th = a.c.f_rho * dl * a.qm[(fl >> GCB_SPECIES_SHIFT) & 3];
                // B = 0 or v_E >= c: Boris
                int S = (F.ok && G2 < th * th * F.B2 && D2 < a.c.f_E2 * F.B2) ? 0 : 1;
                if (a.c.force == GCB_FORCE_BORIS) S = 1;
                if (a.c.force == GCB_FORCE_GCA) S = 0;
                cls = S;
            } else if ((fl_in & GCB_FLAG_EXITED) && !(fl_in & GCB_FLAG_NONFINITE)) {
                ++ne;
            } else {
                ++nf;
            }
            if (cls == 2) {
#pragma unroll
                for (int k = 0; k < 3; ++k) { a.x[k][i] = xs[k]; a.u[k][i] = us[k]; }
                a.flags[i] = fl;
            }
            if (a.pidin != a.pid) a.pid[i] = a.pidin[i];
        }
        if (valid) {
#pragma unroll
            for (int k = 0; k < 3; ++k) { s_x[k][tid] = xs[k]; s_u[k][tid] = us[k]; }
        }
        s_fl[tid] = fl;
        const unsigned bgm = __ballot_sync(0xffffffffu, cls == 0);
        const unsigned bbm = __ballot_sync(0xffffffffu, cls == 1);
        if (lane == 0) { s_wc[0][warp] = __popc(bgm); s_wc[1][warp] = __popc(bbm); }
        __syncthreads();
        int offG = 0, offB = 0, totG = 0, totB = 0;
#pragma unroll
        for (int w = 0; w < NWARP; ++w) {
            const int cg = s_wc[0][w], cb = s_wc[1][w];
            if (w < warp) { offG += cg; offB += cb; }
            totG += cg;
            totB += cb;
        }
        const unsigned lt = (1u << lane) - 1u;
        if (cls == 0) s_perm[offG + __popc(bgm & lt)] = (unsigned short)tid;
        if (cls == 1) s_perm[totG + offB + __popc(bbm & lt)] = (unsigned short)tid;
        __syncthreads();
        if (tid < totG + totB) {
            const int sl = s_perm[tid];
            const uint8_t f0 = s_fl[sl];
            const int S = tid < totG ? 0 : 1;
            const double qm = a.qm[(f0 >> GCB_SPECIES_SHIFT) & 3];
            double x[3], u[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) { x[k] = s_x[k][sl]; u[k] = s_u[k][sl]; }
            const TrigLog t0 = {s_T[0][sl], s_T[1][sl], s_T[2][sl]};
            GFrame F;
            frame_load(s_F, sl, x[0], t0, F);
            F.ok = s_ok[sl] != 0;
            int it = 0;
            bool ncv = false, fail = false;
            Metric mfin;
            const int br = ks_particle(g, a.c, qm, S, F, t0, x, u, it, ncv, fail, mfin);
            // poles: reflect theta, rotate phi by pi, flip u_theta
            if (x[1] < 0.0) { x[1] = -x[1]; x[2] += PI; u[1] = -u[1]; }
            if (x[1] > PI) { x[1] = 2.0 * PI - x[1]; x[2] += PI; u[1] = -u[1]; }
            x[2] -= 2.0 * PI * floor(x[2] * (0.5 / PI));
            if (x[2] >= 2.0 * PI) x[2] -= 2.0 * PI;
            bool fin = true;
#pragma unroll
            for (int k = 0; k < 3; ++k) fin = fin && finite64(x[k]) && finite64(u[k]);
            const int Sprev = f0 & GCB_FLAG_S;
            uint8_t nfl = (uint8_t)((f0 & 0xC0) | (Sprev ? GCB_FLAG_SPREV : 0) | (S ? GCB_FLAG_S : 0));
            const int64_t gi = tile * TPB + sl;
            if (fin) {
                if (fail) nfl |= GCB_FLAG_GCAFAIL;
                if (ncv) nfl |= GCB_FLAG_NONCONV;
                if (x[0] < a.c.r_in || x[0] > a.c.r_out) nfl |= GCB_FLAG_EXITED;
#pragma unroll
                for (int k = 0; k < 3; ++k) { a.x[k][gi] = x[k]; a.u[k][gi] = u[k]; }
                if (br == 0) ++ng; else ++nb;
                if (Sprev && !S) ++tg;
                if (!Sprev && S) ++tb;
                if (ncv) ++nc;
                if (fail) ++gf;
                si += it;
                mi = max(mi, (unsigned)it);
                if constexpr (STATS) {
                    double v[3];
                    raise(mfin, u, v);
                    const double u2 = dot(u, v);
                    ek = fma(u2, rcp64(1.0 + sqrt64(1.0 + u2)), ek);
                }
            } else {
                nfl |= GCB_FLAG_NONFINITE;
                ++nf;
#pragma unroll
                for (int k = 0; k < 3; ++k) { a.x[k][gi] = s_x[k][sl]; a.u[k][gi] = s_u[k][sl]; }
            }
            a.flags[gi] = nfl;
        }
    }
    if constexpr (!STATS) return;
    unsigned vals[9] = {nb, ng, tg, tb, nc, gf, nf, si, mi};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        unsigned v = __reduce_add_sync(0xffffffffu, vals[k]);
        if (lane == 0 && v) atomicAdd(&s_acc[k], (unsigned long long)v);
    }
    {
        const unsigned v = __reduce_add_sync(0xffffffffu, ne);
        if (lane == 0 && v) atomicAdd(&a.stats[ST_EXITED], (unsigned long long)v);
    }
    unsigned mx = __reduce_max_sync(0xffffffffu, vals[8]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ek += __shfl_xor_sync(0xffffffffu, ek, o);
    __syncthreads();
    if (lane == 0) {
        if (mx) atomicMax(&s_acc[ST_MAX_ITER], (unsigned long long)mx);
        atomicAdd(&s_ek, ek);
    }
    __syncthreads();
    if (tid < ST_MAX_ITER) {
        if (s_acc[tid]) atomicAdd(&a.stats[tid], s_acc[tid]);
    } else if (tid == ST_MAX_ITER) {
        if (s_acc[tid]) atomicMax(&a.stats[tid], s_acc[tid]);
    } else if (tid == ST_EKIN) {
        atomicAdd(reinterpret_cast<double *>(&a.stats[ST_EKIN]), s_ek);
    }
}

// Effective cell size (Sec. 3, Eq. volint): dl = (integral of
// sqrt(gamma_rr gamma_thth - gamma_rth^2) dr dtheta over the cell)^(1/2),
// 4x4 Gauss-Legendre in (r, theta); for Kerr-Schild gamma_rth = 0.
__global__ void k_cell_size(int nr, int nth, double logr0, double dlogr, double dth, double a,
                            double *dl)
{
    const double gx[4] = {-0.8611363115940526, -0.3399810435848563, 0.3399810435848563,
                          0.8611363115940526};
    const double gw[4] = {0.3478548451374538, 0.6521451548625461, 0.6521451548625461,
                          0.3478548451374538};
    const int ncell = (nr - 1) * (nth - 1);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        const int i = c % (nr - 1), j = c / (nr - 1);
        const double r0 = exp(logr0 + i * dlogr), r1 = exp(logr0 + (i + 1) * dlogr);
        const double t0 = j * dth, t1 = (j + 1) * dth;
        double area = 0.0;
        for (int p = 0; p < 4; ++p)
            for (int q = 0; q < 4; ++q) {
                const double r = 0.5 * (r0 + r1) + 0.5 * (r1 - r0) * gx[p];
                const double th = 0.5 * (t0 + t1) + 0.5 * (t1 - t0) * gx[q];
                const double c2 = cos(th) * cos(th);
                const double rho2 = r * r + a * a * c2;
                area += gw[p] * gw[q] * sqrt((1.0 + 2.0 * r / rho2) * rho2);
            }
        dl[c] = sqrt(area * 0.25 * (r1 - r0) * (t1 - t0));
    }
}

template <typename FT, bool STATS>
static gcb_status launch(const KsGrid<FT> &g, const Args &a, cudaStream_t st)
{
    static int grid_cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        set_error("cudaGetDevice failed");
        return GCB_ECUDA;
    }
    if (grid_cache[dev] == 0) {
        int nsm = 0, occ = 0;
        if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_push_ks<FT, STATS>, TPB, 0) != cudaSuccess) {
            set_error("occupancy query failed");
            return GCB_ECUDA;
        }
        grid_cache[dev] = nsm * (occ > 0 ? occ : 1);
    }
    const int64_t ntiles = (a.np + TPB - 1) / TPB;
    if (ntiles == 0) return GCB_OK;
    const int nb = (int)(ntiles < grid_cache[dev] ? ntiles : grid_cache[dev]);
    k_push_ks<FT, STATS><<<nb, TPB, 0, st>>>(g, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("k_push_ks launch: %s", cudaGetErrorString(e));
        return GCB_ECUDA;
    }
    return GCB_OK;
}

template <typename FT>
static gcb_status push_step(const gcb_particles *p, const gcb_particles *in, const gcb_grid_ks *gk,
                            const gcb_ks_params *kp, const gcb_params *prm, cudaStream_t st,
                            unsigned long long *stats)
{
    KsGrid<FT> g;
    g.rec = static_cast<const FT *>(gk->g.rec);
    g.stride = gk->g.stride;
    g.nr = (int)gk->g.n[0];
    g.nth = (int)gk->g.n[1];
    g.logr0 = gk->logr0;
    g.inv_dlogr = 1.0 / gk->g.dx[0];
    g.inv_dth = 1.0 / gk->g.dx[1];
    g.dl = gk->dl;
    Args a;
    a.np = p->n;
    for (int k = 0; k < 3; ++k) {
        a.xin[k] = static_cast<const double *>(in->x[k]);
        a.uin[k] = static_cast<const double *>(in->u[k]);
        a.x[k] = static_cast<double *>(p->x[k]);
        a.u[k] = static_cast<double *>(p->u[k]);
    }
    a.flagsin = in->flags;
    a.flags = p->flags;
    a.pid = p->pid;
    a.pidin = p->pid ? in->pid : nullptr;
    for (int k = 0; k < 4; ++k) a.qm[k] = prm->qm[k];
    a.c.a = kp->a;
    a.c.dt = prm->dt;
    a.c.f_rho = prm->f_rho;
    a.c.f_E2 = prm->f_E * prm->f_E;
    a.c.r_in = kp->r_in;
    a.c.r_out = kp->r_out;
    a.c.tol = prm->gca_tol;
    a.c.max_iter = prm->gca_max_iter;
    a.c.fixed_iters = prm->gca_fixed_iters;
    a.c.force = prm->force;
    a.c.mu_mode = prm->mu_mode;
    a.c.basis = kp->kick_basis;
    a.stats = stats;
    return stats ? launch<FT, true>(g, a, st) : launch<FT, false>(g, a, st);
}

}  // namespace ks

gcb_status push_step_ks(const gcb_particles *p, const gcb_particles *in, const gcb_grid_ks *g,
                        const gcb_ks_params *kp, const gcb_params *prm, cudaStream_t st,
                        unsigned long long *stats)
{
    return g->g.dtype == GCB_F32 ? ks::push_step<float>(p, in, g, kp, prm, st, stats)
                                 : ks::push_step<double>(p, in, g, kp, prm, st, stats);
}

gcb_status ks_cell_size(const gcb_grid_ks *g, const gcb_ks_params *kp, double *dl, cudaStream_t st)
{
    const int nr = (int)g->g.n[0], nth = (int)g->g.n[1];
    const int ncell = (nr - 1) * (nth - 1);
    const int nb = (ncell + 255) / 256 < 4096 ? (ncell + 255) / 256 : 4096;
    ks::k_cell_size<<<nb, 256, 0, st>>>(nr, nth, g->logr0, g->g.dx[0], g->g.dx[1], kp->a, dl);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("k_cell_size launch: %s", cudaGetErrorString(e));
        return GCB_ECUDA;
    }
    return GCB_OK;
}

}  // namespace gcb
