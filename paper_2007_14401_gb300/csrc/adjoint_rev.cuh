// adjoint_rev.cuh -- transposed derivative (reverse mode) of one flat-space
// particle-step, 2D with gradient records.  Every function *_bwd takes the
// forward inputs and the adjoint of the outputs and ADDS the adjoint of the
// inputs into its accumulators, recomputing the forward intermediates it
// needs.  The step's structure (Sec. 3.1 with Sec. 2.2.2 and Sec. 2.1):
//   F0 = field at x^n;  conversion at R^{n-1/2} = x^n - dxp/2 -> (u_par, mu,
//   u_perp, gyrophase direction);  u_par update at x^n (quadratic in Gamma);
//   K fixed-point iterates d^k = dt/2 (V^n + V^{k-1}) with V^{k-1} the
//   guiding-center velocity at x^n + d^{k-1};  reconstruction of u at
//   R^{n+1/2} = x^n + d^K/2;  outputs x^{n+1} = x^n + d^K, dxp = d^K, u.
#pragma once

#include "gcb_device.cuh"

namespace gcb {
namespace rev {

// Reciprocals and reciprocal roots: the approximate instructions in FP32, one
// Householder step from them in FP64 (real64.cuh).
__device__ __forceinline__ float rsq_r(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq_r(double x) { return rsqrt64(x); }
__device__ __forceinline__ float rcp_r(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp_r(double x) { return rcp64(x); }

// The frame as the transposes need it: with 1/|B|, its square, E x B, 1 -
// v_E^2/c^2, 1/kappa and the unscaled directional derivatives w = (b.grad)B, y =
// (v_E.grad)B kept.  bgb = w/|B| and vgb = y/|B| are left unprojected: every
// use is b x (.) or v_E . (.), which annihilates their component along b for
// any fields, so that the step's derivative does not depend on it.  1 -
// v_E^2/c^2 from v_E, as the forward step's frame has it: |E x B|^2 is a fourth
// power of the field, which FP32 holds for 1e-9 < |B| < 4e9 only.
template <typename T, int ND>
struct RFrame {
    T Bmag, ib, ib2, b[3], x[3], vE[3], om, kappa, ikap, Epar, w[3], y[3], bgb[3], vgb[3];

    __device__ __forceinline__ void make(const FieldPt<T, ND> &F, T c, T inv_c2)
    {
        const T B2 = dot3(F.B, F.B);
        ib = rsq_r(B2);
        Bmag = B2 * ib;
        ib2 = ib * ib;
        cross3(F.E, F.B, x);
        const T cv = c * ib2;
#pragma unroll
        for (int k = 0; k < 3; ++k) { b[k] = F.B[k] * ib; vE[k] = cv * x[k]; }
        om = one_minus_beta2<T>(F.E, F.B, B2, c, dot3(vE, vE) * inv_c2);
        kappa = rsq_r(om);
        ikap = om * kappa;
        Epar = dot3(F.E, b);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T sw = b[0] * F.dB[0][j], sy = vE[0] * F.dB[0][j];
#pragma unroll
            for (int i = 1; i < ND; ++i) {
                sw = fma(b[i], F.dB[i][j], sw);
                sy = fma(vE[i], F.dB[i][j], sy);
            }
            w[j] = sw;
            y[j] = sy;
            bgb[j] = sw * ib;
            vgb[j] = sy * ib;
        }
    }
};

template <typename T>
struct FrameAdj {
    T Bmag, b[3], vE[3], kappa, Epar, bgb[3], vgb[3];
    __device__ __forceinline__ void zero()
    {
        Bmag = kappa = Epar = T(0);
#pragma unroll
        for (int k = 0; k < 3; ++k) b[k] = vE[k] = bgb[k] = vgb[k] = T(0);
    }
};

// Adjoint of RFrame::make: aF = (d frame / dF)^T af.
template <typename T, int ND>
__device__ __forceinline__ void frame_bwd(const FieldPt<T, ND> &F, const RFrame<T, ND> &f, T c,
                                          T inv_c2, const FrameAdj<T> &af, FieldPt<T, ND> &aF)
{
    T ab[3], avE[3], aw[3], ay[3];
    // bgb = w ib,  vgb = y ib
    T aib = dot3(af.bgb, f.w) + dot3(af.vgb, f.y);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        aw[j] = af.bgb[j] * f.ib;
        ay[j] = af.vgb[j] * f.ib;
        ab[j] = af.b[j];
        avE[j] = af.vE[j];
    }
    // w_j = sum_i b_i dB_ij,  y_j = sum_i vE_i dB_ij
#pragma unroll
    for (int i = 0; i < ND; ++i) {
        ab[i] += dot3(aw, F.dB[i]);
        avE[i] += dot3(ay, F.dB[i]);
#pragma unroll
        for (int j = 0; j < 3; ++j) aF.dB[i][j] = fma(aw[j], f.b[i], ay[j] * f.vE[i]);
    }
    // Epar = E.b
#pragma unroll
    for (int k = 0; k < 3; ++k) ab[k] = fma(af.Epar, F.E[k], ab[k]);
    // kappa = (1 - beta2)^(-1/2):  d kappa / d beta2 = kappa^3 / 2
    const T k2 = af.kappa * f.kappa * f.kappa * f.kappa * inv_c2;
#pragma unroll
    for (int k = 0; k < 3; ++k) avE[k] = fma(k2, f.vE[k], avE[k]);
    // vE = c x ib2,  x = E x B
    const T cv = c * f.ib2;
    T ax[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ax[k] = cv * avE[k];
    const T aib2 = c * dot3(avE, f.x);
    T tE[3], tB[3];
    cross3(F.B, ax, tE);
    cross3(ax, F.E, tB);
    // b = B ib,  ib2 = ib^2,  ib = 1/|B|,  |B| = sqrt(B.B)
    aib += dot3(ab, F.B) + T(2) * f.ib * aib2;
    const T aBmag = af.Bmag - aib * f.ib2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        aF.E[k] = fma(af.Epar, f.b[k], tE[k]);
        aF.B[k] = fma(ab[k], f.ib, fma(aBmag, f.b[k], tB[k]));
    }
}

template <typename T, typename F>
__device__ __forceinline__ T perp2_r(const F &f, const StepPar<T> &s, T mu, T uperp)
{
    return s.mu_mode ? uperp * uperp : T(2) * mu * f.Bmag * f.kappa;
}
template <typename T, typename F>
__device__ __forceinline__ void perp2_bwd(const F &f, const StepPar<T> &s, T mu, T uperp, T aP,
                                          FrameAdj<T> &af, T &amu, T &auperp)
{
    if (s.mu_mode) {
        auperp = fma(T(2) * uperp, aP, auperp);
    } else {
        const T a2 = T(2) * aP;
        amu = fma(f.Bmag * f.kappa, a2, amu);
        af.Bmag = fma(mu * f.kappa, a2, af.Bmag);
        af.kappa = fma(mu * f.Bmag, a2, af.kappa);
    }
}

// Gamma = kappa S, S = sqrt(1 + (u_par^2 + P)/c^2), with its reciprocals
template <typename T>
struct Gam { T S, iS, G, iG; };

template <typename T, typename F>
__device__ __forceinline__ Gam<T> gamma_r(const F &f, const StepPar<T> &s, T upar, T mu, T uperp)
{
    Gam<T> g;
    const T S2 = fma(fma(upar, upar, perp2_r(f, s, mu, uperp)), s.inv_c2, T(1));
    g.iS = rsq_r(S2);
    g.S = S2 * g.iS;
    g.G = f.kappa * g.S;
    g.iG = f.ikap * g.iS;
    return g;
}
template <typename T, typename F>
__device__ __forceinline__ void gamma_bwd(const F &f, const StepPar<T> &s, const Gam<T> &g, T upar,
                                          T mu, T uperp, T aG, FrameAdj<T> &af, T &aupar, T &amu,
                                          T &auperp)
{
    af.kappa = fma(aG, g.S, af.kappa);
    const T ain = T(0.5) * aG * f.kappa * s.inv_c2 * g.iS;
    aupar = fma(T(2) * upar, ain, aupar);
    perp2_bwd(f, s, mu, uperp, ain, af, amu, auperp);
}

// v_c = pref b x (k2 bgb + u_par vgb),  k2 = u_par^2/G,  pref = c kappa^2/(q/m |B|)
template <typename T, typename F>
__device__ __forceinline__ void vcurv_r(const F &f, const StepPar<T> &s, T upar, T iG, T vc[3])
{
    if (!s.curvature) { vc[0] = vc[1] = vc[2] = T(0); return; }
    T a[3], x[3];
    const T k2 = upar * upar * iG;
#pragma unroll
    for (int k = 0; k < 3; ++k) a[k] = fma(k2, f.bgb[k], upar * f.vgb[k]);
    cross3(f.b, a, x);
    const T pref = s.cq * f.kappa * f.kappa * f.ib;
#pragma unroll
    for (int k = 0; k < 3; ++k) vc[k] = pref * x[k];
}
template <typename T, typename F>
__device__ __forceinline__ void vcurv_bwd(const F &f, const StepPar<T> &s, T upar, T iG,
                                          const T avc[3], FrameAdj<T> &af, T &aupar, T &aG)
{
    if (!s.curvature) return;
    const T ig = upar * iG, k2 = upar * ig;
    T a[3], x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) a[k] = fma(k2, f.bgb[k], upar * f.vgb[k]);
    cross3(f.b, a, x);
    const T pref = s.cq * f.kappa * f.kappa * f.ib;
    const T apref = pref * dot3(avc, x);
    T ax[3], t[3], aa[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ax[k] = pref * avc[k];
    cross3(a, ax, t);
    cross3(ax, f.b, aa);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        af.b[k] += t[k];
        af.bgb[k] = fma(k2, aa[k], af.bgb[k]);
        af.vgb[k] = fma(upar, aa[k], af.vgb[k]);
    }
    const T ak2 = dot3(aa, f.bgb);
    aupar += fma(T(2) * ig, ak2, dot3(aa, f.vgb));
    aG = fma(-ig * ig, ak2, aG);
    af.kappa = fma(T(2) * f.ikap, apref, af.kappa);
    af.Bmag = fma(-f.ib, apref, af.Bmag);
}

// V = (u_par/G) b + vE + v_c,  G = Gamma(u_par, mu)
template <typename T, typename F>
__device__ __forceinline__ void gc_vel_bwd(const F &f, const StepPar<T> &s, T upar, T mu, T uperp,
                                           const T aV[3], FrameAdj<T> &af, T &aupar, T &amu,
                                           T &auperp)
{
    const Gam<T> g = gamma_r(f, s, upar, mu, uperp);
    const T ig = upar * g.iG;
    const T aig = dot3(aV, f.b) * g.iG;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        af.b[k] = fma(ig, aV[k], af.b[k]);
        af.vE[k] += aV[k];
    }
    aupar += aig;
    T aG = -ig * aig;
    vcurv_bwd(f, s, upar, g.iG, aV, af, aupar, aG);
    gamma_bwd(f, s, g, upar, mu, uperp, aG, af, aupar, amu, auperp);
}

// u_par update at x^n (Sec. 2.2.1 without curvature; Sec. 2.2.2 with it: the
// Lorentz factor G1 is the larger root of k1 G^2 + k2 G + k3 = 0, whose
// derivative follows from the quadratic itself: dG1 = -(G1^2 dk1 + G1 dk2 +
// dk3) / (2 k1 G1 + k2)).
template <typename T>
struct Quad { T A, gg, D, iD, upr, P0, k1, k2, G1, upn; Gam<T> g0; };

// (of k1 G^2 + k2 G + k3 = 0 with k1 < 0 < k3 the one positive root, as in the
// forward step)
template <typename T, typename F>
__device__ __forceinline__ void quad_r(const F &f0, const StepPar<T> &s, T upar, T mu, T uperp, Quad<T> &q)
{
    q.A = dot3(f0.vE, f0.bgb);
    q.gg = dot3(f0.vE, f0.vgb);
    q.D = fma(-s.half_dt, q.A, T(1));
    q.iD = rcp_r(q.D);
    q.g0 = gamma_r(f0, s, upar, mu, uperp);
    q.upr = fma(upar, fma(s.half_dt, q.A, T(1)),
                fma(s.qm * s.dt, f0.Epar, s.half_dt * q.g0.G * q.gg));
    const T c2 = s.c * s.c, D2 = q.D * q.D;
    q.P0 = perp2_r(f0, s, mu, uperp);
    q.k1 = T(0.25) * s.dt * s.dt * q.gg * q.gg - c2 * D2 * f0.om;
    q.k2 = q.upr * s.dt * q.gg;
    const T k3 = fma(q.upr, q.upr, (c2 + q.P0) * D2);
    const T disc = fma(q.k2, q.k2, T(-4) * q.k1 * k3);
    const T sq = disc * rsq_r(disc);
    const T h = T(-0.5) * (q.k2 + (q.k2 >= T(0) ? sq : -sq));
    q.G1 = q.k2 >= T(0) ? h * rcp_r(q.k1) : k3 * rcp_r(h);
    q.upn = fma(s.half_dt * q.G1, q.gg, q.upr) * q.iD;
}

// u_par^{n+1/2} from the frame at x^n
template <typename T, typename F>
__device__ __forceinline__ T upar_new(const F &f0, const StepPar<T> &s, T upar, T mu, T uperp)
{
    if (!s.curvature) return fma(s.qm * s.dt, f0.Epar, upar);
    Quad<T> q;
    quad_r(f0, s, upar, mu, uperp, q);
    return q.upn;
}

template <typename T, typename F>
__device__ __forceinline__ void upar_bwd(const F &f0, const StepPar<T> &s, T upar, T mu, T uperp,
                                         T aupn, FrameAdj<T> &af, T &aupar, T &amu, T &auperp)
{
    if (!s.curvature) {
        aupar += aupn;
        af.Epar = fma(s.qm * s.dt, aupn, af.Epar);
        return;
    }
    Quad<T> q;
    quad_r(f0, s, upar, mu, uperp, q);
    const T c2 = s.c * s.c;
    const T av = aupn * q.iD;
    const T aG1 = av * s.half_dt * q.gg;
    T agg = av * s.half_dt * q.G1;
    T aupr = av;
    T aD = -av * q.upn;
    const T ak3 = -aG1 * rcp_r(fma(T(2) * q.k1, q.G1, q.k2));
    const T ak2 = q.G1 * ak3;
    const T ak1 = q.G1 * ak2;
    // k3 = upr^2 + (c^2 + P0) D^2
    aupr = fma(T(2) * q.upr, ak3, aupr);
    const T aP0 = q.D * q.D * ak3;
    aD = fma(T(2) * (c2 + q.P0) * q.D, ak3, aD);
    // k2 = upr dt gg
    aupr = fma(s.dt * q.gg, ak2, aupr);
    agg = fma(q.upr * s.dt, ak2, agg);
    // k1 = dt^2 gg^2 / 4 - c^2 D^2 / kappa^2
    agg = fma(T(0.5) * s.dt * s.dt * q.gg, ak1, agg);
    aD = fma(T(-2) * c2 * q.D * f0.om, ak1, aD);
    af.kappa = fma(T(2) * c2 * q.D * q.D * f0.om * f0.ikap, ak1, af.kappa);
    // upr = u_par (1 + dt/2 A) + (q/m) dt Epar + dt/2 G0 gg
    aupar = fma(fma(s.half_dt, q.A, T(1)), aupr, aupar);
    // D = 1 - dt/2 A
    const T aA = s.half_dt * fma(upar, aupr, -aD);
    af.Epar = fma(s.qm * s.dt, aupr, af.Epar);
    const T aG0 = s.half_dt * q.gg * aupr;
    agg = fma(s.half_dt * q.g0.G, aupr, agg);
    gamma_bwd(f0, s, q.g0, upar, mu, uperp, aG0, af, aupar, amu, auperp);
    perp2_bwd(f0, s, mu, uperp, aP0, af, amu, auperp);
    // gg = vE.vgb,  A = vE.bgb
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        af.vE[k] += fma(agg, f0.vgb[k], aA * f0.bgb[k]);
        af.vgb[k] = fma(agg, f0.vE[k], af.vgb[k]);
        af.bgb[k] = fma(aA, f0.vE[k], af.bgb[k]);
    }
}

// Conversion at R^{n-1/2}:  G = Gamma(u), u_par = u.b,
// u_g = u - u_par b - (vE + v_c(u_par, G)) G,  u_perp = |u_g|, bpg = u_g/u_perp,
// mu = u_perp^2 / (2 |B| kappa).
template <typename T>
struct Conv { T G, iG, upar, vc[3], uperp, iu, mu, bpg[3]; };

template <typename T, typename F>
__device__ __forceinline__ void conv_fwd(const F &fm, const StepPar<T> &s, const T u[3], Conv<T> &q)
{
    const T G2 = fma(dot3(u, u), s.inv_c2, T(1));
    q.iG = rsq_r(G2);
    q.G = G2 * q.iG;
    q.upar = dot3(u, fm.b);
    vcurv_r(fm, s, q.upar, q.iG, q.vc);
    T ug[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ug[k] = fma(-q.G, fm.vE[k] + q.vc[k], fma(-q.upar, fm.b[k], u[k]));
    const T up2 = dot3(ug, ug);
    q.iu = rsq_r(up2);
    q.uperp = up2 * q.iu;
    if (!(q.uperp >= Eps<T>::tiny)) {
        q.uperp = q.iu = q.mu = T(0);
        q.bpg[0] = q.bpg[1] = q.bpg[2] = T(0);
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) q.bpg[k] = ug[k] * q.iu;
        q.mu = T(0.5) * up2 * fm.ib * fm.ikap;
    }
}

template <typename T, typename F>
__device__ __forceinline__ void conv_bwd(const F &fm, const StepPar<T> &s, const T u[3],
                                         const Conv<T> &q, T aupar, T amu, T auperp, const T abpg[3],
                                         FrameAdj<T> &af, T au[3])
{
    T aug[3] = {T(0), T(0), T(0)};
    if (q.uperp > T(0)) {
        auperp = fma(amu * q.uperp, fm.ib * fm.ikap, auperp);
        af.Bmag = fma(-amu * q.mu, fm.ib, af.Bmag);
        af.kappa = fma(-amu * q.mu, fm.ikap, af.kappa);
        const T abb = dot3(abpg, q.bpg);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            aug[k] = fma(fma(-abb, q.bpg[k], abpg[k]), q.iu, auperp * q.bpg[k]);
    }
    T avc[3];
    T aGf = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        au[k] += aug[k];
        af.b[k] = fma(-q.upar, aug[k], af.b[k]);
        af.vE[k] = fma(-q.G, aug[k], af.vE[k]);
        avc[k] = -q.G * aug[k];
        aGf = fma(-aug[k], fm.vE[k] + q.vc[k], aGf);
    }
    aupar -= dot3(aug, fm.b);
    vcurv_bwd(fm, s, q.upar, q.iG, avc, af, aupar, aGf);
    const T ag = aGf * s.inv_c2 * q.iG;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        au[k] += fma(aupar, fm.b[k], ag * u[k]);
        af.b[k] = fma(aupar, u[k], af.b[k]);
    }
}

// Reconstruction at R^{n+1/2}:  u = u_par b + (vE + v_c) G + u_n bpg,
// u_n = u_perp (mu_mode) or sqrt(2 mu |B| kappa).
template <typename T, typename F>
__device__ __forceinline__ void recon_bwd(const F &fp, const StepPar<T> &s, T upn, T mu, T uperp,
                                          const T bpg[3], const T lamu[3], FrameAdj<T> &af, T &aupn,
                                          T &amu, T &auperp, T abpg[3])
{
    const Gam<T> g = gamma_r(fp, s, upn, mu, uperp);
    T vc[3];
    vcurv_r(fp, s, upn, g.iG, vc);
    const T Bk = fp.Bmag * fp.kappa;
    const T un2 = T(2) * mu * Bk;
    const T iun = un2 > T(0) ? rsq_r(un2) : T(0);
    const T un = s.mu_mode ? uperp : un2 * iun;
    aupn += dot3(lamu, fp.b);
    T avc[3];
    T aGp = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        af.b[k] = fma(upn, lamu[k], af.b[k]);
        af.vE[k] = fma(g.G, lamu[k], af.vE[k]);
        abpg[k] = fma(un, lamu[k], abpg[k]);
        avc[k] = g.G * lamu[k];
        aGp = fma(lamu[k], fp.vE[k] + vc[k], aGp);
    }
    const T aun = dot3(lamu, bpg);
    if (s.mu_mode) {
        auperp += aun;
    } else {
        const T t = aun * iun;
        amu = fma(t, Bk, amu);
        af.Bmag = fma(t * mu, fp.kappa, af.Bmag);
        af.kappa = fma(t * mu, fp.Bmag, af.kappa);
    }
    vcurv_bwd(fp, s, upn, g.iG, avc, af, aupn, aGp);
    gamma_bwd(fp, s, g, upn, mu, uperp, aGp, af, aupn, amu, auperp);
}

// Relativistic Boris push (Sec. 2.1) and disp = dt u/gamma: adjoints of u, E, B.
template <typename T, int ND>
__device__ __forceinline__ void boris_bwd(const T E[3], const T B[3], const StepPar<T> &s,
                                          const T u[3], const T lamu[3], const T ldisp[ND],
                                          T au[3], T aE[3], T aB[3])
{
    const T h = s.qm * s.half_dt;
    T um[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) um[k] = fma(h, E[k], u[k]);
    const T gm = sqrt(T(1) + dot3(um, um) * s.inv_c2);
    const T ht = h / (s.c * gm);
    T t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = ht * B[k];
    const T sf = T(2) / (T(1) + dot3(t, t));
    T x1[3], up[3], x2[3], un[3];
    cross3(um, t, x1);
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = um[k] + x1[k];
    cross3(up, t, x2);
#pragma unroll
    for (int k = 0; k < 3; ++k) un[k] = fma(h, E[k], fma(sf, x2[k], um[k]));
    const T g = sqrt(T(1) + dot3(un, un) * s.inv_c2);
    const T f = s.dt / g;

    // disp_d = f un_d (d < ND)
    T aun[3] = {lamu[0], lamu[1], lamu[2]};
    T af = T(0);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        af += ldisp[d] * un[d];
        aun[d] += f * ldisp[d];
    }
    const T ag = -af * s.dt / (g * g);
#pragma unroll
    for (int k = 0; k < 3; ++k) aun[k] += ag * un[k] * s.inv_c2 / g;
    // un = um + sf x2 + h E
    T aum[3], ax2[3], aup[3], ax1[3], at[3], tmp[3];
    const T asf = dot3(aun, x2);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        aum[k] = aun[k];
        ax2[k] = sf * aun[k];
        aE[k] = h * aun[k];
    }
    // x2 = up x t
    cross3(t, ax2, aup);
    cross3(ax2, up, at);
    // up = um + x1
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        aum[k] += aup[k];
        ax1[k] = aup[k];
    }
    // x1 = um x t
    cross3(t, ax1, tmp);
#pragma unroll
    for (int k = 0; k < 3; ++k) aum[k] += tmp[k];
    cross3(ax1, um, tmp);
    // sf = 2/(1 + t.t)
#pragma unroll
    for (int k = 0; k < 3; ++k) at[k] += tmp[k] - sf * sf * asf * t[k];
    // t = ht B,  ht = h/(c gm)
    const T aht = dot3(at, B);
    const T agm = -aht * ht / gm;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        aB[k] = ht * at[k];
        aum[k] += agm * um[k] * s.inv_c2 / gm;
        au[k] = aum[k];
        aE[k] += h * aum[k];
    }
}

}  // namespace rev
}  // namespace gcb
