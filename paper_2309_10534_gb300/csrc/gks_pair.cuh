// gks_pair.cuh -- packed float32 pairs for the reconstructions of the
// float32 kernels.
//
// GB300's FP32 units execute two-lane packed instructions (FFMA2, FADD2,
// FMUL2: one issue slot, two IEEE round-to-nearest results).  Where the same
// TENO-D arithmetic runs on two independent streams, the float32 kernels run
// them as one packed stream: in the 2-D sweep the normal reconstruction of
// variables (0, 1) and (2, 3) and the tangential reconstruction of a face
// side's value and normal-slope line averages; in the 1-D kernels the
// normal reconstruction of (rho, rho u).  (The flux's two sides were
// measured packed the same way and kept scalar: no gain.)  `f2` is a drop-in
// arithmetic type for the templated kernel arithmetic: a product stays
// unevaluated (`Prod`) until it is added, so `a * b + c` becomes one fused
// multiply-add, as the compiler's contraction does for scalar code.
// Divisions and comparisons run per lane.
#pragma once

#include "gks_device.cuh"

namespace gks {

struct __align__(8) f2 {
    float2 v;
    f2() = default;
    GKS_HD f2(float s) : v(make_float2(s, s)) {}
    GKS_HD f2(double s) : v(make_float2((float)s, (float)s)) {}
    GKS_HD f2(int s) : v(make_float2((float)s, (float)s)) {}
    GKS_HD f2(float a, float b) : v(make_float2(a, b)) {}
    GKS_HD explicit f2(float2 p) : v(p) {}
    GKS_HD float x() const { return v.x; }
    GKS_HD float y() const { return v.y; }
};

GKS_HD f2 pmul(f2 a, f2 b)
{
#ifdef __CUDA_ARCH__
    return f2(__fmul2_rn(a.v, b.v));
#else
    return f2(a.v.x * b.v.x, a.v.y * b.v.y);
#endif
}
GKS_HD f2 padd(f2 a, f2 b)
{
#ifdef __CUDA_ARCH__
    return f2(__fadd2_rn(a.v, b.v));
#else
    return f2(a.v.x + b.v.x, a.v.y + b.v.y);
#endif
}
GKS_HD f2 pfma(f2 a, f2 b, f2 c)
{
#ifdef __CUDA_ARCH__
    return f2(__ffma2_rn(a.v, b.v, c.v));
#else
    return f2(fmaf(a.v.x, b.v.x, c.v.x), fmaf(a.v.y, b.v.y, c.v.y));
#endif
}
GKS_HD f2 pneg(f2 a) { return f2(-a.v.x, -a.v.y); }

// an unevaluated product a * b
struct Prod {
    f2 a, b;
    GKS_HD operator f2() const { return pmul(a, b); }
};

GKS_HD Prod operator*(f2 a, f2 b) { return Prod{a, b}; }
GKS_HD Prod operator*(Prod p, f2 b) { return Prod{f2(p), b}; }
GKS_HD Prod operator*(f2 a, Prod p) { return Prod{a, f2(p)}; }
GKS_HD Prod operator*(Prod p, Prod q) { return Prod{f2(p), f2(q)}; }

GKS_HD f2 operator+(f2 a, f2 b) { return padd(a, b); }
GKS_HD f2 operator+(Prod p, f2 c) { return pfma(p.a, p.b, c); }
GKS_HD f2 operator+(f2 c, Prod p) { return pfma(p.a, p.b, c); }
GKS_HD f2 operator+(Prod p, Prod q) { return pfma(p.a, p.b, f2(q)); }

GKS_HD f2 operator-(f2 a) { return pneg(a); }
GKS_HD Prod operator-(Prod p) { return Prod{pneg(p.a), p.b}; }
GKS_HD f2 operator-(f2 a, f2 b) { return padd(a, pneg(b)); }
GKS_HD f2 operator-(Prod p, f2 c) { return pfma(p.a, p.b, pneg(c)); }
GKS_HD f2 operator-(f2 c, Prod p) { return pfma(pneg(p.a), p.b, c); }
GKS_HD f2 operator-(Prod p, Prod q) { return pfma(p.a, p.b, pneg(f2(q))); }

// per-lane division (the build's float division, as in scalar code)
GKS_HD f2 operator/(f2 a, f2 b) { return f2(a.v.x / b.v.x, a.v.y / b.v.y); }
GKS_HD f2 operator/(Prod p, f2 b) { return f2(p) / b; }

GKS_HD f2& operator+=(f2& a, f2 b) { return a = a + b; }
GKS_HD f2& operator+=(f2& a, Prod p) { return a = p + a; }
GKS_HD f2& operator-=(f2& a, f2 b) { return a = a - b; }
GKS_HD f2& operator*=(f2& a, f2 b) { return a = pmul(a, b); }

// TENO-D selection (Sec. 4.2, Eqs. 4.5-4.7 and 4.11-4.12) of two 5-cell
// stencils at once, one per lane, with the selection folded into the
// coefficients: a lane that keeps the large stencil has zero sub-stencil
// weights, a lane that keeps sub-stencils has zero quartic coefficients, so
// one formula evaluates either choice.  Same powers-of-ratios form as
// teno_select (no division by beta, nothing overflows).
struct TenoSel2 {
    f2 q2, A, B, C, D, B0, B2, C0, C2, P, R;  // as TenoSel
    f2 l, w[3];                               // 1 where the large stencil is kept, else the sub-stencils' weights
};

GKS_HD float lane_min4(float a, float b, float c, float d) { return fminf(fminf(a, b), fminf(c, d)); }

// r^q of both lanes
GKS_HD f2 pair_pow(f2 r, int q)
{
    if (q == 7) {
        const f2 r2 = r * r, r3 = r2 * r;
        return r3 * r3 * r;
    }
    return f2(ipow(r.x(), q), ipow(r.y(), q));
}

// Returns true where both lanes keep the large stencil whatever the other
// powers are (their sum with p_3 lies below 4, so p_3 >= 4 C_T1 settles Eq.
// 4.7): in smooth regions three of the four powers and reciprocals, the
// second selection and the sub-stencils' half of the evaluation (S.w is zero)
// are then never formed, half of a pair's work.  Measured: one step of a
// 1024^2 plane 0.763 -> 0.678 ms, 2048x1024 viscous 1.82 -> 1.66 ms, gradient
// of a 512^2 flow 10.9 -> 9.95 ms.  The 1-D kernels, whose flux outweighs
// their one selection per cell, lost 2 % to the branch and pass QUICK = false.
template <bool QUICK = true>
GKS_HD bool teno_select_x2(const f2 q[5], const TenoT<float>& P, TenoSel2& S)
{
    TenoSel<f2> C;
    teno_differences(q, C);
    f2 t[4];
    teno_indicators(C, f2(4.0f * P.eps), t);
    S.q2 = C.q2;
    S.A = C.A;
    S.B = C.B;
    S.C = C.C;
    S.D = C.D;
    S.B0 = C.B0;
    S.B2 = C.B2;
    S.C0 = C.C0;
    S.C2 = C.C2;
    S.P = C.P;
    S.R = C.R;
    const f2 m(lane_min4(t[0].x(), t[1].x(), t[2].x(), t[3].x()), lane_min4(t[0].y(), t[1].y(), t[2].y(), t[3].y()));
    f2 p[4];
    p[3] = pair_pow(m * f2(1.0f / t[3].x(), 1.0f / t[3].y()), P.q);
    const float sure = 4.001f * P.ct1;
    if (QUICK && p[3].x() >= sure && p[3].y() >= sure) {
        S.l = f2(1.0f);
        S.w[0] = S.w[1] = S.w[2] = f2(0.0f);
        return true;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) p[j] = m * f2(1.0f / t[j].x(), 1.0f / t[j].y());
    if (P.q == 7) {
#pragma unroll
        for (int j = 0; j < 3; ++j) p[j] = pair_pow(p[j], 7);
    } else {
#pragma unroll
        for (int j = 0; j < 3; ++j) p[j] = pair_pow(p[j], P.q);
    }
    const f2 s012 = p[0] + p[1] + p[2];
    const f2 lim = f2(P.ct1) * (s012 + p[3]);
    const float lx = (p[3].x() >= lim.x()) ? 1.0f : 0.0f, ly = (p[3].y() >= lim.y()) ? 1.0f : 0.0f;
    const f2 thr = f2(P.ct2) * s012;
    f2 d[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        d[k] = f2(p[k].x() >= thr.x() ? 1.0f : 0.0f, p[k].y() >= thr.y() ? 1.0f : 0.0f);
    // at least one sub-stencil passes the second cut (its ratio is the
    // largest, >= s012 / 3 > C_T2 s012), so dsum >= 1
    const f2 dsum = d[0] + d[1] + d[2];
    const f2 inv = f2((1.0f - lx) / dsum.x(), (1.0f - ly) / dsum.y());  // 0 on large-stencil lanes
    S.l = f2(lx, ly);
#pragma unroll
    for (int k = 0; k < 3; ++k) S.w[k] = d[k] * inv;
    return false;
}

// the selection of lane x (y) as 4 bits (bit 0: large stencil; bits 1-3:
// the kept sub-stencils): a lane that keeps sub-stencils has a positive weight
GKS_HD unsigned sel_code_x(const TenoSel2& S)
{
    const unsigned c = (S.w[0].x() > 0.0f ? 2u : 0u) | (S.w[1].x() > 0.0f ? 4u : 0u) | (S.w[2].x() > 0.0f ? 8u : 0u);
    return c ? c : 1u;
}
GKS_HD unsigned sel_code_y(const TenoSel2& S)
{
    const unsigned c = (S.w[0].y() > 0.0f ? 2u : 0u) | (S.w[1].y() > 0.0f ? 4u : 0u) | (S.w[2].y() > 0.0f ? 8u : 0u);
    return c ? c : 1u;
}

// 2 sum w_k b_k and 2 sum w_k c_k of the kept sub-stencils
GKS_HD void teno_small_x2(const TenoSel2& S, f2& sb, f2& sc)
{
    sb = S.w[0] * S.B0;
    sb += S.w[1] * S.A;
    sb += S.w[2] * S.B2;
    sc = S.w[0] * S.C0;
    sc += S.w[1] * S.C;
    sc += S.w[2] * S.C2;
}

// values and xi-derivatives at the faces xi = +-1/2 of both lanes' selection:
// teno_faces with both choices evaluated, the other one's terms zeroed;
// large: both lanes keep the large stencil (the same bits without the
// sub-stencils)
GKS_HD void teno_faces_x2(const TenoSel2& S, bool large, f2& vp, f2& dp, f2& vm, f2& dm)
{
    if (large) {
        const f2 k(1.0f / 24.0f);
        const f2 even = f2(1.0f / 120.0f) * f2(f2(13.0f) * S.C - S.D) + S.q2;
        const f2 odd = k * S.P;
        const f2 de = k * f2(f2(13.0f) * S.A - S.B);
        const f2 dod = k * f2(f2(15.0f) * S.C - S.D);
        vp = even + odd;
        vm = even - odd;
        dp = de + dod;
        dm = de - dod;
        return;
    }
    f2 sb, sc;
    teno_small_x2(S, sb, sc);
    const f2 l24 = S.l * f2(1.0f / 24.0f), l120 = S.l * f2(1.0f / 120.0f);
    const f2 even = l120 * f2(f2(13.0f) * S.C - S.D) + f2(f2(1.0f / 12.0f) * sc + S.q2);
    const f2 odd = l24 * S.P + f2(f2(0.25f) * sb);
    const f2 de = l24 * f2(f2(13.0f) * S.A - S.B) + f2(f2(0.5f) * sb);
    const f2 dod = l24 * f2(f2(15.0f) * S.C - S.D) + f2(f2(0.5f) * sc);
    vp = even + odd;
    vm = even - odd;
    dp = de + dod;
    dm = de - dod;
}

// Normal reconstruction of one 1-D cell's three variables (rho, rho u, E):
// float32 TENO-D runs (rho, rho u) as one packed pair and E alone; otherwise
// variable by variable with the scheme's reconstruction.  Face values and
// xi-slopes at +1/2 (vp, dp) and -1/2 (vm, dm).
template <int REC, typename T>
GKS_HD void recon_cell3(const T q[3][5], const TenoT<T>& P, T* vp, T* dp, T* vm, T* dm)
{
    if constexpr (sizeof(T) == 4 && REC == 0) {
        f2 qq[5];
#pragma unroll
        for (int s = 0; s < 5; ++s) qq[s] = f2(q[0][s], q[1][s]);
        TenoSel2 S2;
        f2 a, b, c, d;
        teno_select_x2<false>(qq, P, S2);
        teno_faces_x2(S2, false, a, b, c, d);
        vp[0] = a.x(); vp[1] = a.y();
        dp[0] = b.x(); dp[1] = b.y();
        vm[0] = c.x(); vm[1] = c.y();
        dm[0] = d.x(); dm[1] = d.y();
        TenoSel<T> S;
        teno_select<false>(q[2], P, S);
        teno_faces(q[2], S, vp[2], dp[2], vm[2], dm[2]);
    } else {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            TenoSel<T> S;
            rec_select<REC, false>(q[v], P, S);
            rec_faces<REC>(q[v], S, vp[v], dp[v], vm[v], dm[v]);
        }
    }
}

// values and xi-derivatives at the two Gauss points xi = -g and xi = +g
// (g = 1/(2 sqrt 3)) of both lanes' selection: teno_gauss_pm with both
// choices evaluated, the other one's terms zeroed; large as in teno_faces_x2
GKS_HD void teno_gauss_pm_x2(const TenoSel2& S, bool large, float g, f2& vm, f2& dm, f2& vp, f2& dp)
{
    if (large) {
        const f2 E = S.q2 - f2(1.0f / 4320.0f) * S.R;
        const f2 O = f2(43.0f / 72.0f) * S.A - f2(7.0f / 72.0f) * S.B;
        const f2 Ed = f2(1.0f / 12.0f) * S.P;
        const f2 Od = f2(12.0f / 9.0f) * S.C - f2(1.0f / 9.0f) * S.D;
        const f2 G(g);
        vm = E - G * O;
        vp = E + G * O;
        dm = Ed - G * Od;
        dp = Ed + G * Od;
        return;
    }
    f2 sb, sc;
    teno_small_x2(S, sb, sc);
    const f2 hb = f2(0.5f) * sb;
    const f2 E = S.q2 - f2(S.l * f2(1.0f / 4320.0f)) * S.R;
    const f2 O = S.l * f2(f2(43.0f / 72.0f) * S.A - f2(7.0f / 72.0f) * S.B) + hb;
    const f2 Ed = f2(S.l * f2(1.0f / 12.0f)) * S.P + hb;
    const f2 Od = S.l * f2(f2(12.0f / 9.0f) * S.C - f2(1.0f / 9.0f) * S.D) + sc;
    const f2 G(g);
    vm = E - G * O;
    vp = E + G * O;
    dm = Ed - G * Od;
    dp = Ed + G * Od;
}

GKS_HD f2 fabs(f2 a) { return f2(fabsf(a.v.x), fabsf(a.v.y)); }

// the reconstruction parameters broadcast to both lanes (WENO5-AO)
GKS_HD TenoT<f2> pair_teno(const TenoT<float>& P)
{
    TenoT<f2> Q;
    Q.eps = f2(P.eps);
    Q.ct1 = f2(P.ct1);
    Q.ct2 = f2(P.ct2);
    Q.q = P.q;
#pragma unroll
    for (int k = 0; k < 4; ++k) Q.g[k] = f2(P.g[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) Q.gr[k] = f2(P.gr[k]);
    Q.ig3 = f2(P.ig3);
    Q.eps_ao = f2(P.eps_ao);
    return Q;
}

// The scheme's reconstruction of two stencils at once: face values and
// xi-slopes (normal direction), or values and xi-derivatives at the two
// Gauss points (tangential).  REC 0: TENO-D with the folded selection above;
// REC 1: WENO5-AO through its templated arithmetic, whose weights have no
// branches.
template <int REC, bool QUICK = true>
GKS_HD void packed_faces(const f2 q[5], const TenoT<float>& P, f2& vp, f2& dp, f2& vm, f2& dm)
{
    if constexpr (REC == 0) {
        TenoSel2 S;
        if (teno_select_x2<QUICK>(q, P, S)) teno_faces_x2(S, true, vp, dp, vm, dm);
        else teno_faces_x2(S, false, vp, dp, vm, dm);
    } else {
        TenoSel<f2> S;
        ao_select(q, pair_teno(P), S);
        ao_faces(q, S, vp, dp, vm, dm);
    }
}
template <int REC>
GKS_HD void packed_gauss(const f2 q[5], const TenoT<float>& P, float gA, float gB, f2& va, f2& da, f2& vb, f2& db)
{
    if constexpr (REC == 0) {
        // the Gauss points are symmetric: gA = -gB
        TenoSel2 S;
        if (teno_select_x2(q, P, S)) teno_gauss_pm_x2(S, true, gB, va, da, vb, db);
        else teno_gauss_pm_x2(S, false, gB, va, da, vb, db);
    } else {
        TenoSel<f2> S;
        ao_select(q, pair_teno(P), S);
        ao_gauss(S, f2(gA), va, da);
        ao_gauss(S, f2(gB), vb, db);
    }
}

}  // namespace gks
