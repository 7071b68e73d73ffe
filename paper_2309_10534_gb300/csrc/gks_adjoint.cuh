// gks_adjoint.cuh -- reverse-mode (vector-Jacobian) counterparts of the
// per-point arithmetic in gks_device.cuh, written out by hand.
//
// Scope: the collision-free interface flux (tau = 0, the setting of the
// paper's smooth-flow tests, Sec. 5.1 and 5.5) in 2-D: the kinetic merge of
// the two reconstructed sides into the equilibrium state and its slopes
// (Eqs. 2.6, 3.25, 3.26), the Euler flux of that state and its time
// derivative from the compatibility condition (Sec. 2.2).  TENO-D is taken
// with the stencil selection of the forward pass held fixed: once the
// selection (large stencil, or which small stencils with weights 1/3) is
// fixed, every reconstructed value and slope is a linear function of the
// five cell averages, and its transpose is below.
//
// Convention: a function named *_vjp adds, to the g* outputs, the product of
// the transposed Jacobian of the forward function with the given cotangents
// of the forward outputs; it recomputes what it needs of the forward values.
#pragma once

#include "gks_device.cuh"

namespace gks {

// ------------------------------------------------------------------ TENO-D, frozen selection
// Both transposes go through the first differences the reconstruction is
// formed from (TenoSel): cotangents of A, B, C, D (or of the sub-stencils'
// coefficients) -> of e_1 .. e_4 -> of the five cells; gq is set.
template <typename T>
GKS_HD void teno_e_T(T ge1, T ge2, T ge3, T ge4, T gc, T* gq)
{
    gq[0] = -ge1;
    gq[1] = ge1 - ge2;
    gq[2] = gc + (ge2 - ge3);
    gq[3] = ge3 - ge4;
    gq[4] = ge4;
}
// kept sub-stencils: cotangents of 2 sum w b and 2 sum w c (teno_small)
template <typename T>
GKS_HD void teno_small_T(const TenoSel<T>& S, T gb, T gc, T g2, T* gq)
{
    const T b0 = S.w[0] * gb, b1 = S.w[1] * gb, b2 = S.w[2] * gb;
    const T c0 = S.w[0] * gc, c1 = S.w[1] * gc, c2 = S.w[2] * gc;
    // B0 = 3 e2 - e1, A = e2 + e3, B2 = 3 e3 - e4; C0 = e2 - e1, C = e3 - e2, C2 = e4 - e3
    teno_e_T(-b0 - c0, T(3) * b0 + b1 + (c0 - c1), T(3) * b2 + b1 + (c1 - c2), c2 - b2, g2, gq);
}
// large stencil: cotangents of A, B, C, D
template <typename T>
GKS_HD void teno_large_T(T gA, T gB, T gC, T gD, T g2, T* gq)
{
    teno_e_T(gB - gD, gA - gC, gA + gC, gB + gD, g2, gq);
}

// transpose of teno_faces: cotangents of (vp, dp, vm, dm) -> gq[0..4]
template <typename T>
GKS_HD void teno_faces_T(const TenoSel<T>& S, T gvp, T gdp, T gvm, T gdm, T* gq)
{
    const T ge = gvp + gvm, go = gvp - gvm, gde = gdp + gdm, gdo = gdp - gdm;
    if (S.large) {
        // even = q2 + (13 C - D)/120, odd = (7 A - B)/24, deven = (13 A - B)/24, dodd = (15 C - D)/24
        const T e = T(1.0 / 120.0) * ge, o = T(1.0 / 24.0) * go, d = T(1.0 / 24.0) * gde, p = T(1.0 / 24.0) * gdo;
        teno_large_T(T(7) * o + T(13) * d, -(o + d), T(13) * e + T(15) * p, -(e + p), ge, gq);
    } else {
        // even = q2 + sc/12, odd = sb/4, deven = sb/2, dodd = sc/2
        teno_small_T(S, T(0.25) * go + T(0.5) * gde, T(1.0 / 12.0) * ge + T(0.5) * gdo, ge, gq);
    }
}

// transpose of teno_gauss_pm: cotangents of the values and derivatives at
// xi = -g (gvm, gdm) and +g (gvp, gdp) -> gq[0..4]
template <typename T>
GKS_HD void teno_gauss_pm_T(const TenoSel<T>& S, T g, T gvm, T gdm, T gvp, T gdp, T* gq)
{
    const T gE = gvp + gvm, gO = g * (gvp - gvm), gEd = gdp + gdm, gOd = g * (gdp - gdm);
    if (S.large) {
        // E = q2 - R/4320, O = (43 A - 7 B)/72, Ed = P/12, Od = (12 C - D)/9, P = 7 A - B, R = D - 3 C
        const T r = T(-1.0 / 4320.0) * gE, o = T(1.0 / 72.0) * gO, p = T(1.0 / 12.0) * gEd, d = T(1.0 / 9.0) * gOd;
        teno_large_T(T(43) * o + T(7) * p, -(T(7) * o + p), T(12) * d - T(3) * r, r - d, gE, gq);
    } else {
        // E = q2, O = Ed = sb/2, Od = sc
        teno_small_T(S, T(0.5) * (gO + gEd), gOd, gE, gq);
    }
}

// ------------------------------------------------------------------ kinetic layer (2-D)
// The flux is formed from the slopes of (rho, U, V, p) and the moments
// u_0 .. u_2 (gks_device.cuh); its reverse walks the same few products back,
// about 160 operations per side and 130 for the equilibrium part, where the
// reverse of the micro slopes and moment matrices took three times as many.

// cotangents of a state's primitive variables and of th = p/rho
template <typename T> struct PrimCot {
    T U, V, q, p, th, r;
};

// prim_slope: cotangents g of (rho', rho U', rho V', p', rho th') -> adds to
// the slope's gd and to the state's c
template <typename T>
GKS_HD void prim_slope_vjp(const Grad<T>& s, T U, T V, T q, T th, T gm1, Grad<T> g, T* gd, PrimCot<T>& c)
{
    g.p += g.mT;  // rho th' = p' - th rho'
    c.th = fma(-s.r, g.mT, c.th);
    g.r = fma(-th, g.mT, g.r);
    const T x = gm1 * g.p;  // p' = gm1 (E' - U rho U' - V rho V' - q rho')
    c.U = fma(-s.mU, x, c.U);
    c.V = fma(-s.mV, x, c.V);
    c.q = fma(-s.r, x, c.q);
    g.mU = fma(-U, x, g.mU);
    g.mV = fma(-V, x, g.mV);
    g.r = fma(-q, x, g.r);
    c.U = fma(-s.r, g.mU, c.U);  // rho U' = (rho U)' - U rho'
    c.V = fma(-s.r, g.mV, c.V);
    gd[0] += fma(-U, g.mU, fma(-V, g.mV, g.r));
    gd[1] += g.mU;
    gd[2] += g.mV;
    gd[3] += x;
}

// the state itself: th = p/rho, p = gm1 (E - rho q), q = (U^2 + V^2)/2,
// (U, V) = (rho U, rho V)/rho -> adds to gW
template <typename T>
GKS_HD void prim_vjp(T r, T ir, T U, T V, T q, T th, T gm1, PrimCot<T> c, T* gW)
{
    const T ith = ir * c.th;
    const T x = gm1 * (c.p + ith);
    c.q = fma(-r, x, c.q);
    c.U = fma(U, c.q, c.U);
    c.V = fma(V, c.q, c.V);
    const T iU = ir * c.U, iV = ir * c.V;
    gW[0] += c.r - fma(q, x, fma(U, iU, fma(V, iV, th * ith)));
    gW[1] += iU;
    gW[2] += iV;
    gW[3] += x;
}

// Reverse of side_terms (NONEQ = false, 2-D): cotangents of the side's
// contributions to W0, W0_n, W0_t -> cotangents of the side's W, Wn, Wt.
template <typename T>
GKS_HD void side_vjp(const Side<T>& S, const Prim<T>& s, T sg, const FluxParams<T>& P, const T* gW0, const T* gW0n,
                     const T* gW0t, Side<T>& gS)
{
    // ---- forward values
    const T r = s.r, ir = s.ir, U = s.U, V = s.V, q = s.q;
    const T th = s.p * ir, sl = M<T>::rsqrt_(T(2) * th), hit = sl * sl;
    T u0, gz;
    half_space_start<T>(sl * U, sg, u0, gz);
    const T w = (sg * T(0.56418958354775628)) * (sl * gz), wt = th * w;
    const T u1 = fma(U, u0, wt), u2 = fma(U, u1, th * u0);
    const T e = fma(P.hkv, th, s.hv2), Uh = U * hit;

    // ---- W0 += (r u0, r u1, V r u0, r u2/2 + e r u0)
    PrimCot<T> c;
    const T A0 = fma(V, gW0[2], fma(e, gW0[3], gW0[0]));
    const T hr3 = T(0.5) * gW0[3], ru0 = r * u0;
    c.r = fma(u0, A0, fma(u1, gW0[1], u2 * hr3));
    c.V = ru0 * gW0[2];
    c.U = c.q = c.p = T(0);
    T ge = ru0 * gW0[3], gu0 = r * A0, gu1 = r * gW0[1], gu2 = r * hr3;
    T gw = T(0), gwt = T(0), ghit = T(0);
    c.th = T(0);
    // ---- W0_d += (n0, n1, V n0 + mV u0, n2/2 + e n0 + kn u0) per direction
    auto dir = [&](const T* d, const T* x, T* gd) {
        Grad<T> n;
        prim_slope<T, 2>(d, U, V, q, th, P.gm1, n);
        const T cn = hit * n.mT, kn = kappa<2>(V, n, P.hkv);
        const T m0 = fma(-U, cn, n.mU);
        const T n0 = fma(n.r, u0, w * m0);
        const T g0 = fma(V, x[2], fma(e, x[3], x[0])), g1 = x[1], g2 = T(0.5) * x[3];
        c.V = fma(n0, x[2], c.V);
        ge = fma(n0, x[3], ge);
        gu0 += fma(n.mV, x[2], fma(kn, x[3], fma(n.mT, g2, fma(n.mU, g1, n.r * g0))));
        const T gk = u0 * x[3];
        c.V = fma(n.mV, gk, c.V);
        Grad<T> g;
        g.p = T(0);
        g.r = fma(u2, g2, fma(u1, g1, u0 * g0));
        g.mV = fma(u0, x[2], V * gk);
        gu2 = fma(n.r, g2, gu2);
        gu1 = fma(T(2) * n.mU, g2, fma(n.r, g1, gu1));
        gwt = fma(cn, g1, gwt);
        gw = fma(m0, g0, gw);
        const T wg = w * g0;
        g.mU = fma(T(2) * u1, g2, fma(u0, g1, wg));
        c.U = fma(-cn, wg, c.U);
        const T gc = fma(wt, g1, -U * wg);
        ghit = fma(n.mT, gc, ghit);
        g.mT = fma(u0, g2, fma(P.hkv, gk, hit * gc));
        prim_slope_vjp(n, U, V, q, th, P.gm1, g, gd, c);
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) gS.W[i] = gS.Wn[i] = gS.Wt[i] = T(0);
    dir(S.Wn, gW0n, gS.Wn);
    dir(S.Wt, gW0t, gS.Wt);
    // ---- moments: u2 = U u1 + th u0, u1 = U u0 + wt, wt = th w,
    // du0/dU = w, du0/dth = -U hit w, dw/dU = -2 U hit w, dw/dth = hit w (2 U^2 hit - 1)
    c.U = fma(u1, gu2, c.U);
    gu1 = fma(U, gu2, gu1);
    c.th = fma(u0, gu2, c.th);
    gu0 = fma(th, gu2, gu0);
    c.U = fma(u0, gu1, c.U);
    gu0 = fma(U, gu1, gu0);
    gwt += gu1;
    c.th = fma(w, gwt, c.th);
    gw = fma(th, gwt, gw);
    c.U = fma(w, fma(T(-2) * Uh, gw, gu0), c.U);
    c.th = fma(w, fma(-Uh, gu0, hit * fma(T(2) * U, Uh, T(-1)) * gw), c.th);
    c.th = fma(T(-2) * hit * hit, ghit, c.th);
    c.V = fma(V, ge, c.V);
    c.th = fma(P.hkv, ge, c.th);
    prim_vjp(r, ir, U, V, q, th, P.gm1, c, gS.W);
}

// Reverse of the equilibrium part of point_flux for tau = 0 (2-D): F = F0,
// dF = F2 of equilibrium().
template <typename T>
GKS_HD void equilibrium_vjp(const T* W0, const T* W0n, const T* W0t, const FluxParams<T>& P, const T* gF, const T* y,
                            T* gW0, T* gW0n, T* gW0t)
{
    const T gm1 = P.gm1;
    Prim<T> s;
    prim_state<T, 2>(W0, gm1, s);
    const T U = s.U, V = s.V, th = s.p * s.ir, Ep = W0[3] + s.p, H = Ep * s.ir;
    Grad<T> n, t, g;
    prim_slope<T, 2>(W0n, U, V, s.q, th, gm1, n);
    prim_slope<T, 2>(W0t, U, V, s.q, th, gm1, t);
    time_slope<T, 2>(n, t, U, V, th, gm1, g);
    // F2 = (mt, U (mt + rho U_t) + p_t, V mt + U rho V_t, H mt + U rho H_t)
    const T mt = fma(U, g.r, g.mU);
    const T rdH = fma(V, g.mV, fma(U, g.mU, P.cp * g.mT));
    PrimCot<T> c;
    const T gmt = fma(U, y[1], fma(V, y[2], fma(H, y[3], y[0])));
    const T gdH = U * y[3];
    c.U = fma(mt + g.mU, y[1], fma(g.mV, y[2], fma(rdH, y[3], fma(g.r, gmt, g.mU * gdH))));
    c.V = fma(mt, y[2], g.mV * gdH);
    c.th = g.r * y[1];
    Grad<T> x;  // cotangents of the time slopes
    x.r = fma(U, gmt, th * y[1]);
    x.mU = fma(U, y[1], fma(U, gdH, gmt));
    x.mV = fma(U, y[2], V * gdH);
    x.mT = fma(P.cp, gdH, y[1]);
    const T gH = mt * y[3];
    // time slopes -> both directions' slopes
    const T div = n.mU + t.mV, gt = (gm1 * th) * x.mT;
    c.U -= fma(n.r, x.r, fma(n.mU, x.mU, fma(n.mV, x.mV, n.mT * x.mT)));
    c.V -= fma(t.r, x.r, fma(t.mU, x.mU, fma(t.mV, x.mV, t.mT * x.mT)));
    c.th = fma(-gm1 * div, x.mT, c.th);
    c.q = T(0);
    Grad<T> gn, gx;
    gn.r = -U * x.r;
    gn.mU = -fma(U, x.mU, x.r + gt);
    gn.mV = -U * x.mV;
    gn.p = -x.mU;
    gn.mT = -U * x.mT;
    gx.r = -V * x.r;
    gx.mU = -V * x.mU;
    gx.mV = -fma(V, x.mV, x.r + gt);
    gx.p = -x.mV;
    gx.mT = -V * x.mT;
    prim_slope_vjp(n, U, V, s.q, th, gm1, gn, gW0n, c);
    prim_slope_vjp(t, U, V, s.q, th, gm1, gx, gW0t, c);
    // F0 = (W1, W1 U + p, W1 V, U (W3 + p)), H = (W3 + p)/rho
    const T iH = s.ir * gH, u3 = fma(U, gF[3], iH);
    c.U = fma(W0[1], gF[1], fma(Ep, gF[3], c.U));
    c.V = fma(W0[1], gF[2], c.V);
    c.p = gF[1] + u3;
    c.r = -H * iH;
    gW0[1] += fma(U, gF[1], fma(V, gF[2], gF[0]));
    gW0[3] += u3;
    prim_vjp(s.r, s.ir, U, V, s.q, th, gm1, c, gW0);
}

// Reverse of point_flux<T, 2, false, false> (tau = 0): cotangents of F and
// dF/dt at one Gauss point -> cotangents of both sides.
template <typename T>
GKS_HD void point_flux_vjp(const Side<T>& L, const Side<T>& R, T sg, const FluxParams<T>& P, const T* gF, const T* gdF,
                           Side<T>& gL, Side<T>& gR)
{
    T W0[4], W0n[4], W0t[4];
    Prim<T> pl, pr;
    prim_state<T, 2>(L.W, P.gm1, pl);
    prim_state<T, 2>(R.W, P.gm1, pr);
    side_terms<false, T, 2, false, false>(L, pl, sg, P, W0, W0n, W0t, nullptr, nullptr, nullptr, nullptr, nullptr);
    side_terms<true, T, 2, false, false>(R, pr, -sg, P, W0, W0n, W0t, nullptr, nullptr, nullptr, nullptr, nullptr);
    T gW0[4] = {T(0), T(0), T(0), T(0)}, gW0n[4] = {T(0), T(0), T(0), T(0)}, gW0t[4] = {T(0), T(0), T(0), T(0)};
    equilibrium_vjp(W0, W0n, W0t, P, gF, gdF, gW0, gW0n, gW0t);
    side_vjp(L, pl, sg, P, gW0, gW0n, gW0t, gL);
    side_vjp(R, pr, -sg, P, gW0, gW0n, gW0t, gR);
}

}  // namespace gks
