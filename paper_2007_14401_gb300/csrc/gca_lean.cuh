// gca_lean.cuh -- the guiding-center step of gcb_device.cuh arranged for the
// fewest operations, for the simplified drift frame in FP64 (2D and 3D) and
// FP32 2D.  Same equations, gathers and iterations; what differs:
//   - b is never formed: B and 1/|B| are, and (b.grad)b and (v_E.grad)b meet
//     in one contraction.  With g = u_par b/Gamma + v_E (the velocity without
//     the curvature drift) v_c = (c kappa^2 u_par/(q B^2)) b x (g.grad)B,
//     6 ND products fewer per velocity than the two directional derivatives;
//   - Gamma enters as 1/Gamma = rsqrt(1 + (u_par^2 + 2 mu B kappa)/c^2) / kappa
//     with 1/kappa = (1 - v_E^2/c^2) kappa: one reciprocal root per velocity;
//   - the gyrating momentum is kept as the vector u_g with 2 mu =
//     u_g^2/(B kappa): the reconstruction scales it by
//     sqrt(B kappa at R^{n+1/2} / B kappa at R^{n-1/2}), no direction is
//     normalised;
//   - of the quadratic's two roots only the positive one is formed.
// Measured on GB300 (before -> after, gca_step_c's arrangement first): FP64,
// bound by its pipe, 1343 -> 1019 pipe slots a particle-step of the 2D
// reconnection push (2^20 particles 2.61 -> 1.95 ms a step; the 3D sheet,
// 300007 particles, with gather_dw64 1.16 -> 0.79 ms); FP32 2D, bound by
// issue, 1603 -> 1401 instructions (2^24 particles, 8 steps and a sort 9.83 ->
// 9.42 ms).  FP32 3D keeps gca_step_c and its record cache.
#pragma once

#include "gcb_device.cuh"

namespace gcb {

__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt64(x); }
__device__ __forceinline__ float rcp(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp(double x) { return rcp64(x); }
__device__ __forceinline__ bool pos_finite(float x) { return x > 0.0f; }
__device__ __forceinline__ bool pos_finite(double x) { return !not_pos_normal(x); }

// Local frame at a point: v_E, and through B2 = |B|^2, ib = 1/|B|, om = 1 -
// v_E^2/c^2 and kap = 1/sqrt(om) the factors of the drift terms.
// The unit of the fields is the caller's.  FP64's exponents hold |E x B|^2 and
// |B|^-3 for |B| of 1e-77 to 1e77, so that the factors 1/|B| are gathered into
// one; FP32's hold |E x B|^2 for 1e-9 to 4e9 only.  There (F32) |v_E|^2 is taken
// from v_E and every product of two fields meets its 1/|B| before the next
// (lean_drift, the u_par update), which keeps all of them within |B|^2, good for
// 1e-19 to 1e19 (from 1e-19 sqrt(c) up, c/|B|^2 being one of them).  It costs
// (GB300, 2D, against one factor |B|^-3) 7 of 1358 instructions a particle-step:
// 2^24 particles, 8 steps and their sort 8.18 -> 8.21 ms; 8 steps of 3000017
// particles in one launch 1.45 -> 1.48 ms.  The order of lean_drift's prefactor
// matters: with kappa^2 apart 8 B more are spilled, 8.37 ms.
template <typename R>
struct LeanFrame {
    static constexpr bool F32 = sizeof(R) == 4;
    R B2, ib, ib2, om, kap, vE[3];
    bool ok;
    __device__ __forceinline__ R Bk() const { return B2 * ib * kap; }      // |B| kappa
    // 1/(|B| kappa); FP32: the reciprocal of Bk(), so that the error of the
    // approximate roots cancels in the ratio of Bk at two neighbouring points
    __device__ __forceinline__ R iBk() const
    {
        if constexpr (sizeof(R) == 8) return ib * (om * kap);
        else return rcp(Bk());
    }
};

template <typename R, int ND>
__device__ __forceinline__ void lean_frame(const FieldPt<R, ND> &F, const StepPar<R> &s,
                                           LeanFrame<R> &f)
{
    f.B2 = dot3(F.B, F.B);
    f.ib = rsq(f.B2);
    f.ib2 = f.ib * f.ib;
    R x[3];
    cross3(F.E, F.B, x);
    const R cv = s.c * f.ib2;
#pragma unroll
    for (int k = 0; k < 3; ++k) f.vE[k] = cv * x[k];
    if constexpr (LeanFrame<R>::F32) {
        f.om = one_minus_beta2<R>(F.E, F.B, f.B2, s.c, dot3(f.vE, f.vE) * s.inv_c2);
    } else {
        const R v2 = dot3(x, x) * f.ib2;   // |E x B|^2/B^2 = B^2 v_E^2/c^2
        f.om = fma(-v2, f.ib2, R(1));
    }
    f.ok = pos_finite(f.B2) && pos_finite(f.om);
    f.kap = rsq(f.om);
}

// Drift velocity v_E + v_c (+ grad-B drift) for upar and iG = 1/Gamma, and
// ig = upar iG/|B| (the parallel velocity is ig B).  The gradients' index
// runs over the ND grid axes; gs scales them (gradients of the shape functions
// come per cell, not per length, from the FP64 gather).
template <typename R, int ND, bool RAW, bool MIR>
__device__ __forceinline__ void lean_drift(const FieldPt<R, ND> &F, const LeanFrame<R> &f,
                                           const StepPar<R> &s, const R gs[ND], R upar, R iG, R mu2,
                                           R &ig, R v[3])
{
    constexpr bool F32 = LeanFrame<R>::F32;
    ig = upar * (iG * f.ib);
    if (s.curvature) {
        R a[3], x[3];
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            R gi = fma(ig, F.B[i], f.vE[i]);
            if (RAW) gi *= gs[i];
            if (F32) gi *= f.ib;
#pragma unroll
            for (int j = 0; j < 3; ++j) a[j] = i == 0 ? gi * F.dB[i][j] : fma(gi, F.dB[i][j], a[j]);
        }
        cross3(F.B, a, x);
        R pf = s.cq * upar;               // c kappa^2 u_par/(q |B|^3); F32: |B|^2
        if constexpr (F32) pf = pf * (f.ib * f.kap) * (f.ib * f.kap);
        else pf = pf * (f.ib * f.ib2) * (f.kap * f.kap);
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = fma(pf, x[k], f.vE[k]);
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = f.vE[k];
    }
    if constexpr (MIR) {
        R h[3] = {R(0), R(0), R(0)}, x[3];
#pragma unroll
        for (int i = 0; i < ND; ++i) {    // |B| grad|B|; F32: grad|B|
            h[i] = dot3(F.B, F.dB[i]);
            if (RAW) h[i] *= gs[i];
            if (F32) h[i] *= f.ib;
        }
        cross3(F.B, h, x);
        R pg = R(0.5) * s.cq * f.kap * mu2 * iG * f.ib2;
        if (!F32) pg *= f.ib;
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = fma(pg, x[k], v[k]);
    }
}

// sin and cos of the gyro-phase -num/den, taken in FP64 (the angle reaches
// Omega_C dt ~ 1e5 rad in strongly magnetized runs): the angle in half turns,
// wrapped into [-1, 1] (exact for the multiples of 2 removed), then sin and cos
// of pi times it.  Out of line: an option's code.
__device__ __forceinline__ double half_turns(double num, double den)
{
    const double t = -num / den * 0.31830988618379067;   // 1/pi
    return fma(-2.0, rint(0.5 * t), t);
}
static __device__ __noinline__ void gyro_sincos(double num, double den, float &sn, float &cs)
{
    sincospif((float)half_turns(num, den), &sn, &cs);
}
static __device__ __noinline__ void gyro_sincos(double num, double den, double &sn, double &cs)
{
    sincospi(half_turns(num, den), &sn, &cs);
}

// The step: arguments and result as gca_step_c.
template <typename R, int ND, int GM, typename Gth, bool MIR = false>
__device__ __forceinline__ bool gca_step_lean(const Gth &gth, const StepPar<R> &s, const int ib[ND],
                                              const R ln[ND], const R dxp[ND],
                                              const FieldPt<R, ND> &F0, R u[3], R disp[ND],
                                              int &iters, bool &nonconv,
                                              R *vz = nullptr)
{
    constexpr bool RAW = RawGrad<R, GM>::value, F32 = LeanFrame<R>::F32;
    R gs[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) gs[d] = gth.g.inv_dx[d];
    FieldPt<R, ND> F;
    LeanFrame<R> f0, f;
    lean_frame<R, ND>(F0, s, f0);

    // conversion at R^{n-1/2} = x^n - dxp/2 (Sec. 3.1): u = u_par b + (v_E +
    // v_c) Gamma + u_g
    R pt[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) pt[d] = fma(R(-0.5), dxp[d], ln[d]);
    gth(ib, pt, F);
    lean_frame<R, ND>(F, s, f);
    if (!(f0.ok && f.ok)) return false;
    R v[3], ig;
    R G = fma(dot3(u, u), s.inv_c2, R(1));
    const R iGf = rsq(G);
    G = G * iGf;
    const R upar = dot3(u, F.B) * f.ib;
    lean_drift<R, ND, RAW, false>(F, f, s, gs, upar, iGf, R(0), ig, v);
    const R upb = upar * f.ib;
    R ug[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ug[k] = fma(-G, v[k], fma(-upb, F.B[k], u[k]));
    const R up2 = dot3(ug, ug);
    const R iBk = f.iBk();
    const R mu2 = up2 * iBk;              // 2 mu / m
    // 2 mu B kappa/m, or u_g^2 when that is held in mu's place

    // u_par update at R^n (Sec. 2.2.1 / Eqs. dupardtcase2discsol, duparprimedtcase2discsol)
    const R Epar = dot3(F0.E, F0.B) * f0.ib;
    R fm = R(0);                          // dt times the mirror force (MIR)
    R upn;
    const R P0 = s.mu_mode ? up2 : mu2 * f0.Bk();
    if constexpr (MIR) {
        R bg = R(0);                      // B . grad|B| |B|; F32: B . grad|B|
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const R h = F0.B[i] * (F32 ? f0.ib * dot3(F0.B, F0.dB[i]) : dot3(F0.B, F0.dB[i]));
            bg += RAW ? h * gs[i] : h;
        }
        const R iG0 = rsq(fma(fma(upar, upar, P0), s.inv_c2, R(1))) * (f0.om * f0.kap);
        fm = R(-0.5) * s.dt * mu2 * bg * (F32 ? f0.ib : f0.ib2) * iG0 * (f0.om * f0.kap);
    }
    if (!s.curvature) {
        upn = fma(s.qm * s.dt, Epar, upar) + fm;
    } else {
        R a = R(0), gg = R(0);            // v_E.(b.grad)b and v_E.(v_E.grad)b
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            R z = dot3(f0.vE, F0.dB[i]);
            if (RAW) z *= gs[i];
            if (F32) z *= f0.ib;
            a = i == 0 ? F0.B[i] * z : fma(F0.B[i], z, a);
            gg = i == 0 ? f0.vE[i] * z : fma(f0.vE[i], z, gg);
        }
        a *= F32 ? f0.ib : f0.ib2;
        if (!F32) gg *= f0.ib;
        const R ha = s.half_dt * a;
        const R hg = s.half_dt * gg;
        const R D = R(1) - ha;
        R G0 = fma(fma(upar, upar, P0), s.inv_c2, R(1));
        G0 = f0.kap * (G0 * rsq(G0));
        R upr = fma(upar, R(1) + ha, fma(s.qm * s.dt, Epar, G0 * hg));
        if constexpr (MIR) upr += fm;
        const R c2 = s.c * s.c;
        const R D2 = D * D;
        const R k1 = fma(hg, hg, -c2 * D2 * f0.om);
        const R k2 = R(2) * upr * hg;
        const R k3 = fma(upr, upr, (c2 + P0) * D2);
        // k1 < 0 < k3: one root is positive; the other has the opposite sign
        R disc = fma(k2, k2, R(-4) * k1 * k3);
        if (!(k1 < R(0)) || !(disc >= R(0)) || D == R(0)) return false;
        const R sq = disc * rsq(disc);
        const bool kp = k2 >= R(0);
        const R q = R(-0.5) * (k2 + (kp ? sq : -sq));
        const R num = kp ? q : k3, den = kp ? k1 : q;
        if constexpr (sizeof(R) == 8) {
            const R inv = rcp(den * D);
            const R G1 = num * (D * inv);
            if (!(G1 >= R(1))) return false;
            upn = fma(G1, hg, upr) * (den * inv);
        } else {
            const R G1 = num / den;
            if (!(G1 >= R(1))) return false;
            upn = fma(G1, hg, upr) / D;
        }
    }

    // guiding-center velocity, Eq. (dRdt)
    const R U1 = fma(upn * upn, s.inv_c2, R(1));
    const R Pc = (s.mu_mode ? up2 : mu2) * s.inv_c2;
    auto gam2 = [&](const LeanFrame<R> &q) {   // (Gamma/kappa)^2
        return s.mu_mode ? U1 + Pc : fma(Pc, q.Bk(), U1);
    };
    auto velocity = [&](const FieldPt<R, ND> &Fp, const LeanFrame<R> &q, R V[3]) {
        const R iG = rsq(gam2(q)) * (q.om * q.kap);
        R w, dv[3];
        lean_drift<R, ND, RAW, MIR>(Fp, q, s, gs, upn, iG, mu2, w, dv);
#pragma unroll
        for (int k = 0; k < 3; ++k) V[k] = fma(w, Fp.B[k], dv[k]);
    };

    // fixed point on Eq. (dRdtcase2disc): R^{k+1} = R^n + dt/2 (V^n + V^k),
    // iterated on the displacement R^{k+1} - R^n from R^0 = R^n.
    R Vn[3];
    velocity(F0, f0, Vn);
    R dk[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) dk[d] = R(0);
    R V[3] = {Vn[0], Vn[1], Vn[2]};
    iters = 0;
    nonconv = false;
    bool okall = true;
    for (;;) {
        R res = R(0), big = R(0);
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const R nd = s.half_dt * (Vn[d] + V[d]);
            const R e = fabs(nd - dk[d]);
            const R m = fabs(nd);
            if constexpr (sizeof(R) == 8) {
                res = gt_nonneg(e, res) ? e : res;
                big = gt_nonneg(m, big) ? m : big;
            } else {
                res = fmax(res, e);
                big = fmax(big, m);
            }
            dk[d] = nd;
        }
        ++iters;
        if (s.fixed_iters > 0) {
            if (iters >= s.fixed_iters) break;
        } else {
            // floor of the arithmetic: the change within 8 ulp of the displacement
            if constexpr (sizeof(R) == 8) {
                if (gt_nonneg(s.tol, res) || !gt_nonneg(res, R(8) * Eps<R>::value * big)) break;
            } else {
                if (res < s.tol || res <= R(8) * Eps<R>::value * big) break;
            }
            if (iters >= s.max_iter) { nonconv = true; break; }
        }
#pragma unroll
        for (int d = 0; d < ND; ++d) pt[d] = ln[d] + dk[d];
        gth(ib, pt, F);
        lean_frame<R, ND>(F, s, f);
        okall = okall && f.ok;   // a bad frame fails the step after the loop
        velocity(F, f, V);
    }
    if (!okall) return false;

    // reconstruction at R^{n+1/2} = (R^{n+1} + R^n)/2 (Sec. 3.1)
#pragma unroll
    for (int d = 0; d < ND; ++d) pt[d] = fma(R(0.5), dk[d], ln[d]);
    gth(ib, pt, F);
    lean_frame<R, ND>(F, s, f);
    if (!f.ok) return false;
    R Gp = gam2(f);
    const R rg = rsq(Gp);
    Gp = f.kap * (Gp * rg);
    lean_drift<R, ND, RAW, false>(F, f, s, gs, upn, rg * (f.om * f.kap), R(0), ig, v);
    R sc = R(1);                          // u_g's growth
    if (!s.mu_mode) {
        // near 1, where the approximate root's error does not average out over
        // the steps: one Newton correction in FP32
        const R r = f.Bk() * iBk, y = rsq(r);
        sc = r * y;
        if constexpr (sizeof(R) == 4) sc = fma(fma(-sc, sc, r), R(0.5) * y, sc);
    }
    if (s.phase) {
        // evolved gyration phase: u_g turns about b by the step's gyro-phase
        // phi = -(q/m) B dt/(c kappa Gamma) (the lab-time rate of the gyration
        // in the frame drifting with v_E)
        R sn, cs;
        gyro_sincos((double)s.qm * (double)(f.B2 * f.ib) * (double)s.dt,
                    (double)s.c * (double)f.kap * (double)Gp, sn, cs);
        R bxd[3];
        cross3(F.B, ug, bxd);
#pragma unroll
        for (int k = 0; k < 3; ++k) ug[k] = fma(cs, ug[k], sn * f.ib * bxd[k]);
    }
    const R upnb = upn * f.ib;
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = fma(upnb, F.B[k], fma(v[k], Gp, sc * ug[k]));
#pragma unroll
    for (int d = 0; d < ND; ++d) disp[d] = dk[d];
    // out-of-plane component of the step's guiding-center velocity (V^n + V^K)/2
    // (2D current deposition); the in-plane ones are disp/dt
    if (vz) *vz = R(0.5) * (Vn[2] + V[2]);
    return true;
}

// Boris push as boris() with reciprocal roots in place of roots and quotients.
template <int ND>
__device__ __forceinline__ void boris_lean(const double E[3], const double B[3],
                                           const StepPar<double> &s, double u[3], double disp[ND])
{
    const double h = s.qm * s.half_dt;
    double um[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) um[k] = fma(h, E[k], u[k]);
    const double ht = (h * s.c * s.inv_c2) * rsqrt64(fma(dot3(um, um), s.inv_c2, 1.0));
    double t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = ht * B[k];
    const double sf = 2.0 * rcp64(fma(t[0], t[0], fma(t[1], t[1], fma(t[2], t[2], 1.0))));
    double x[3], up[3];
    cross3(um, t, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = um[k] + x[k];
    cross3(up, t, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = fma(h, E[k], fma(sf, x[k], um[k]));
    const double f = s.dt * rsqrt64(fma(dot3(u, u), s.inv_c2, 1.0));
#pragma unroll
    for (int d = 0; d < ND; ++d) disp[d] = f * u[d];
}

}  // namespace gcb
