// gks_device.cuh -- device arithmetic of the TENO-D gas-kinetic scheme.
//
// Everything here runs per cell or per interface point in registers:
//   * TENO-D reconstruction of one 5-cell stencil (paper Sec. 4.2), written
//     with the Legendre-type coefficients of the quartic and the (b, c)
//     coefficients of the three quadratics, evaluated at the cell faces
//     (xi = +-1/2) or at the Gauss points xi = +-1/(2 sqrt 3);
//   * Maxwellian moments, the closed-form micro-slope solve, kinetic merge
//     and the time-dependent BGK flux at one point (Sec. 2.1, Eqs. 2.5-2.9),
//     with the two time integrals of Sec. 2.2 folded into F and dF/dt.
// Templated on the arithmetic type T (float or double) and the dimension.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <type_traits>

#define GKS_HD __host__ __device__ __forceinline__

namespace gks {

// ------------------------------------------------------------------ math
template <typename T> struct M;
template <> struct M<float> {
    static GKS_HD float erfc_(float x) { return erfcf(x); }
    static GKS_HD float exp_(float x) { return expf(x); }
    static GKS_HD float sqrt_(float x) { return sqrtf(x); }
#ifdef __CUDA_ARCH__
    static GKS_HD float rsqrt_(float x) { return rsqrtf(x); }
#else
    static GKS_HD float rsqrt_(float x) { return 1.0f / sqrtf(x); }
#endif
    static constexpr float tiny = 1.17549435e-38f;  // FLT_MIN: smallest eps kept normal
    static constexpr int nseries = 16;               // terms of the time-coefficient series
    static constexpr float s_series = 2.0f;          // series below, closed form above
    static constexpr float s_noexp = 48.0f;          // above: exp(-s/2) < 4e-11, below float32 resolution
};
template <> struct M<double> {
    static GKS_HD double erfc_(double x) { return erfc(x); }
    static GKS_HD double exp_(double x) { return exp(x); }
    static GKS_HD double sqrt_(double x) { return sqrt(x); }
#ifdef __CUDA_ARCH__
    static GKS_HD double rsqrt_(double x) { return rsqrt(x); }
#else
    static GKS_HD double rsqrt_(double x) { return 1.0 / sqrt(x); }
#endif
    static constexpr double tiny = 0.0;
    static constexpr int nseries = 22;
    static constexpr double s_series = 1.0;
    static constexpr double s_noexp = 90.0;           // above: exp(-s/2) < 3e-20, below float64 resolution
};

// bits of a float64 and float32 (device: register moves)
GKS_HD int hi_word(double x)
{
#ifdef __CUDA_ARCH__
    return __double2hiint(x);
#else
    int64_t b;
    memcpy(&b, &x, 8);
    return (int)(b >> 32);
#endif
}
GKS_HD unsigned lo_word(double x)
{
#ifdef __CUDA_ARCH__
    return (unsigned)__double2loint(x);
#else
    int64_t b;
    memcpy(&b, &x, 8);
    return (unsigned)b;
#endif
}
GKS_HD float as_float(unsigned u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}
GKS_HD float quick_div(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}
GKS_HD int imax(int a, int b) { return a > b ? a : b; }

// float32 <-> float64 on the integer pipe.  A conversion instruction occupies
// GB300's float64 pipe for 64 cycles a warp, which made the float32 kernels'
// one float64 update per value (a subtraction between two conversions) wait
// on that pipe; these take about ten integer operations and the same bits:
// widening is exact, narrowing rounds to nearest even, and float32 denormals
// are zero, as everywhere in those kernels.
GKS_HD unsigned float_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned u;
    memcpy(&u, &x, 4);
    return u;
#endif
}
GKS_HD double make_double(unsigned hi, unsigned lo)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = ((uint64_t)hi << 32) | lo;
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
GKS_HD double widen(float x)
{
    const unsigned u = float_bits(x), e = u & 0x7f800000u;
    unsigned hi = ((u & 0x7fffffffu) >> 3) + (896u << 20);  // exponent bias 127 -> 1023
    hi = e == 0u ? 0u : (e == 0x7f800000u ? (hi | 0x7ff00000u) : hi);
    return make_double(hi | (u & 0x80000000u), e == 0u ? 0u : u << 29);
}
GKS_HD float narrow(double x)
{
    const unsigned hi = (unsigned)hi_word(x), lo = lo_word(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    unsigned v = ((unsigned)(e - 896) << 23) + m;
    v += ((lo & 0x1fffffffu) + 0x0fffffffu + (v & 1u)) >> 29;  // a carry runs into the exponent, up to infinity
    if (e <= 896) v = 0u;
    if (e >= 1151) v = (e == 0x7ff && (m | lo) != 0u) ? 0x7fffffffu : 0x7f800000u;
    return as_float(v | (hi & 0x80000000u));
}
// a float64 value in the kernel's arithmetic type, and back
template <typename T> GKS_HD T from_f64(double x) { return x; }
template <> GKS_HD float from_f64<float>(double x) { return narrow(x); }
GKS_HD double to_f64(double x) { return x; }
GKS_HD double to_f64(float x) { return widen(x); }

// integer power by squaring (q of Eq. 4.5 is a small positive integer)
template <typename T>
GKS_HD T ipow(T x, int q)
{
    T r = T(1);
    while (q) {
        if (q & 1) r *= x;
        x *= x;
        q >>= 1;
    }
    return r;
}

// ------------------------------------------------------------------ reconstruction parameters
// recon 0: TENO-D (Sec. 4.2); 1: WENO5-AO (Sec. 3.2), the reconstruction the
// paper compares against; 2: WENO5-Z and 3: TENO5, the conventional path
// (Sec. 3.1, 4.1; 1-D grids).
struct TenoParams {
    double eps;
    int q;
    double ct1, ct2;  // thresholds of the first / second selection
    int recon = 0;
    double d_hi = 0.85, d_lo = 0.85, eps_ao = 1e-8;  // WENO5-AO
};

// the same parameters in the arithmetic type of the kernel (no conversions
// from double inside the hot loop); eps is clamped to the smallest normal
// float in float32.  WENO5-AO: linear weights g[0..3] of the three
// sub-stencils and the large stencil, gr[k] = g[k]/g[3], and 1/g[3].
template <typename T> struct TenoT {
    T eps, ct1, ct2;
    int q;
    T g[4], gr[3], ig3, eps_ao;
    // float64 kernels' float32 selection (teno_code_f32): 4 eps as
    // eps4_m 2^eps4_e, the cut-offs, and the relative distance from a cut-off
    // that float32 decides
    float eps4_m, fct1, fct2, margin;
    int eps4_e;
};

template <typename T>
inline TenoT<T> teno_t(const TenoParams& P)
{
    TenoT<T> t;
    t.eps = (T)P.eps;
    if (t.eps < (T)M<T>::tiny) t.eps = (T)M<T>::tiny;
    t.ct1 = (T)P.ct1;
    t.ct2 = (T)P.ct2;
    t.q = P.q;
    const double g3 = P.d_hi, g1 = (1.0 - P.d_hi) * P.d_lo, g0 = 0.5 * (1.0 - P.d_hi) * (1.0 - P.d_lo);
    t.g[0] = (T)g0;
    t.g[1] = (T)g1;
    t.g[2] = (T)g0;
    t.g[3] = (T)g3;
    t.gr[0] = (T)(g0 / g3);
    t.gr[1] = (T)(g1 / g3);
    t.gr[2] = (T)(g0 / g3);
    t.ig3 = (T)(1.0 / g3);
    t.eps_ao = (T)P.eps_ao;
    t.eps4_m = (float)frexp(4.0 * P.eps, &t.eps4_e);
    t.fct1 = (float)P.ct1;
    t.fct2 = (float)P.ct2;
    t.margin = 2e-4f * (float)(P.q + 1);
    return t;
}

// Result of a reconstruction's selection on one 5-cell stencil.  TENO-D:
// either the large stencil, or the equal-weight (d_k = 1/3) average of the
// kept sub-stencils, on the first differences of the cells.  WENO5-AO,
// WENO5-Z, TENO5: the candidates' coefficients and weights.
template <typename T> struct TenoSel {
    T q2;               // centre cell average
    // TENO-D: with e_i = q_i - q_(i-1), A = e2 + e3, B = e1 + e4, C = e3 - e2,
    // D = e4 - e1: twice the quadratics' coefficients (2 b_k = B0, A, B2;
    // 2 c_k = C0, C, C2) and the quartic's combinations P = 7 A - B, R = D - 3 C
    T A, B, C, D, B0, B2, C0, C2, P, R;
    T b[3], c[3];       // others: quadratic k: p = q2 - c/12 + b xi + c xi^2
    T u1, u2, u3, u4;   // others: quartic in the Legendre-type basis
    T w[3];             // sub-stencil weights (0 when the large stencil is used)
    T w3;               // WENO5-AO: weight of the quartic (TENO-D: unused)
    bool large;
};

// the sub-stencil quadratics and the large-stencil quartic (Sec. 3.1),
// formed from the sums and differences of the cells at equal distance from
// the centre (the quartic's odd coefficients only see the differences, its
// even ones only the sums): every coefficient is one to three fused
// multiply-adds
template <typename T>
GKS_HD void stencil_coeffs(const T q[5], TenoSel<T>& S)
{
    const T q0 = q[0], q1 = q[1], q2 = q[2], q3 = q[3], q4 = q[4];
    const T s1 = q1 + q3, d1 = q3 - q1, s0 = q0 + q4, d0 = q4 - q0;
    S.q2 = q2;
    S.b[0] = T(1.5) * q2 + (T(0.5) * q0 - T(2) * q1);  // (q0 - 4 q1 + 3 q2) / 2
    S.c[0] = T(0.5) * (q0 + q2) - q1;                   // (q0 - 2 q1 + q2) / 2
    S.b[1] = T(0.5) * d1;                               // (q3 - q1) / 2
    S.c[1] = T(0.5) * s1 - q2;                          // (q1 - 2 q2 + q3) / 2
    S.b[2] = T(2) * q3 - (T(1.5) * q2 + T(0.5) * q4);   // (-3 q2 + 4 q3 - q4) / 2
    S.c[2] = T(0.5) * (q2 + q4) - q3;                   // (q2 - 2 q3 + q4) / 2
    S.u1 = T(82.0 / 120.0) * d1 - T(11.0 / 120.0) * d0;                       // (11 q0 - 82 q1 + 82 q3 - 11 q4) / 120
    S.u2 = T(40.0 / 56.0) * s1 - (T(3.0 / 56.0) * s0 + T(74.0 / 56.0) * q2);  // (-3 q0 + 40 q1 - 74 q2 + 40 q3 - 3 q4) / 56
    S.u3 = T(1.0 / 12.0) * d0 - T(1.0 / 6.0) * d1;                            // (-q0 + 2 q1 - 2 q3 + q4) / 12
    S.u4 = T(1.0 / 24.0) * s0 + (T(0.25) * q2 - T(1.0 / 6.0) * s1);          // (q0 - 4 q1 + 6 q2 - 4 q3 + q4) / 24
}

// TENO-D works on first differences e_i: every sub-stencil coefficient is a
// combination of two of them and the quartic's of A, B (odd) or C, D (even),
// and every reconstructed value is q2 plus such combinations.  Against the
// coefficients formed from the cell averages this takes 14 instead of 26
// operations and no large common part cancels; the indicators, faces and
// Gauss points share P and R.  Measured: one step of a 1024^2 float32 plane
// 0.844 -> 0.810 ms, of a 400^2 float64 plane 5.77 -> 5.12 ms.
template <typename T>
GKS_HD void teno_differences(const T q[5], TenoSel<T>& S)
{
    const T e1 = q[1] - q[0], e2 = q[2] - q[1], e3 = q[3] - q[2], e4 = q[4] - q[3];
    S.q2 = q[2];
    S.A = e2 + e3;
    S.B = e1 + e4;
    S.C = e3 - e2;
    S.D = e4 - e1;
    S.B0 = T(3) * e2 - e1;  // q0 - 4 q1 + 3 q2
    S.C0 = e2 - e1;         // q0 - 2 q1 + q2
    S.B2 = T(3) * e3 - e4;  // -3 q2 + 4 q3 - q4
    S.C2 = e4 - e3;         // q2 - 2 q3 + q4
    S.P = T(7) * S.A - S.B;
    S.R = S.D - T(3) * S.C;
}

// smoothness indicators t_k = 4 (beta_k + eps) of Eq. (3.7): quadratics
// b^2 + 13/3 c^2; the quartic in Balsara's Legendre form, whose four squares
// are u1 + u3/10 = P/12, u2 + 123/455 u4 = (163 C - 11 D)/260,
// u3 = (B - A)/12 and u4 = R/24.  eps4 = 4 eps.
template <typename T>
GKS_HD void teno_indicators(const TenoSel<T>& S, T eps4, T* t)
{
    const T k = T(13.0 / 3.0);
    t[0] = S.B0 * S.B0 + (k * S.C0 * S.C0 + eps4);
    t[1] = S.A * S.A + (k * S.C * S.C + eps4);
    t[2] = S.B2 * S.B2 + (k * S.C2 * S.C2 + eps4);
    const T u3 = S.B - S.A, bq = S.C - T(11.0 / 163.0) * S.D;
    t[3] = T(1.0 / 36.0) * S.P * S.P
         + (T(13.0 / 3.0 * (163.0 / 130.0) * (163.0 / 130.0)) * bq * bq
            + (T(781.0 / 720.0) * u3 * u3 + (T(1421461.0 / 327600.0) * S.R * S.R + eps4)));
}

// WENO5-AO (Sec. 3.2): beta by Eq. (3.7), global indicator
// tau = mean |beta_3 - beta_k|, weights gamma_k (1 + (tau/(beta_k + eps))^2)
// normalised over the four stencils, and the AO(5,3) polynomial
//   P = wbar_3/gamma_3 p_3 + sum_k (wbar_k - wbar_3 gamma_k/gamma_3) p_k,
// stored as the evaluation weights w3 (quartic) and w[k] (quadratics).
template <typename T>
GKS_HD void ao_select(const T q[5], const TenoT<T>& P, TenoSel<T>& S)
{
    stencil_coeffs(q, S);
    T beta[4];
#pragma unroll
    for (int k = 0; k < 3; ++k) beta[k] = S.b[k] * S.b[k] + T(13.0 / 3.0) * S.c[k] * S.c[k];
    {
        const T a = S.u1 + T(0.1) * S.u3, bq = S.u2 + T(123.0 / 455.0) * S.u4;
        beta[3] = a * a + T(13.0 / 3.0) * bq * bq + T(781.0 / 20.0) * S.u3 * S.u3
                + T(1421461.0 / 2275.0) * S.u4 * S.u4;
    }
    const T tau = (fabs(beta[3] - beta[0]) + fabs(beta[3] - beta[1]) + fabs(beta[3] - beta[2])) * T(1.0 / 3.0);
    T om[4], sum = T(0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const T r = tau / (beta[k] + P.eps_ao);
        om[k] = P.g[k] * (T(1) + r * r);
        sum += om[k];
    }
    const T is = T(1) / sum;
    const T w3 = om[3] * is;
    S.w3 = w3 * P.ig3;
#pragma unroll
    for (int k = 0; k < 3; ++k) S.w[k] = om[k] * is - w3 * P.gr[k];
    S.large = false;
}

// Selection of Eqs. (4.5)-(4.7) and (4.11)-(4.12) as 4 bits: bit 0 the large
// stencil, bits 1-3 the kept sub-stencils.
// chi_k = t_k^-q / sum_j t_j^-q.  With m = min_j t_j and r_j = m / t_j in
// (0, 1], chi_k = r_k^q / sum_j r_j^q: nothing overflows, and an r^q that
// underflows belongs to a chi far below any cut-off.  The same powers serve
// both selections (the second normalises over k = 0..2 only, where d_k = 1/3
// cancels).
template <typename T>
GKS_HD T teno_pow(T r, int q)
{
    if (q == 7) {
        const T r2 = r * r, r3 = r2 * r;
        return r3 * r3 * r;
    }
    return ipow(r, q);
}
// QUICK: leave at once where the large stencil is settled by its own power
template <bool QUICK, typename T>
GKS_HD unsigned teno_code(const T t[4], T ct1, T ct2, int q)
{
    T m = t[0] < t[1] ? t[0] : t[1];
    m = m < t[2] ? m : t[2];
    m = m < t[3] ? m : t[3];
    T p[4];
    p[3] = teno_pow(m * (T(1) / t[3]), q);
    if (QUICK && p[3] >= T(4.001) * ct1) return 1u;  // s012 + p[3] < 4: the first selection is settled
#pragma unroll
    for (int j = 0; j < 3; ++j) p[j] = teno_pow(m * (T(1) / t[j]), q);
    const T s012 = p[0] + p[1] + p[2];
    // first selection (Eqs. 4.6, 4.7): keep the large stencil when chi_{3,1} >= C_T1
    if (p[3] >= ct1 * (s012 + p[3])) return 1u;
    // second selection among the small stencils (Eqs. 4.11, 4.12)
    const T thr = ct2 * s012;
    return (p[0] >= thr ? 2u : 0u) | (p[1] >= thr ? 4u : 0u) | (p[2] >= thr ? 8u : 0u);
}

// The float64 selection decided in float32, or 0 where float32 cannot decide.
//
// GB300's float64 pipe takes a warp instruction every 64 cycles, and the
// selection is a comparison: of ~150 float64 operations per stencil, the
// indicators, four reciprocals, powers and cut-offs took two thirds.  The
// four first differences, scaled by a common power of two (their exponents
// are read from the high words on the integer pipe, so not even a
// conversion runs on the float64 pipe), give every indicator in float32 to
// 6e-5: a truncated difference is off by 2^-23 and the quadratic forms
// amplify that at most 88 times (the largest eigenvalue of |Q| over the
// smallest of Q, over the four forms), 2 * 88 * 2^-23 = 2.1e-5, plus the
// rounding of their evaluation; a ratio of two is then off by less than 1e-4
// and its q-th power by q 1e-4.  A cut-off further away than twice that is
// decided; the rest (about one selection in 1e4, and the stencils beside an
// exactly constant run, whose smallest indicator is lost in the scaling)
// takes teno_code in float64.  Measured: one step of a 400^2 float64 plane
// 5.12 -> 3.27 ms, the same states to round-off.
GKS_HD float scaled_float(double x, int base)
{
    // x scaled by a power of two and truncated to float32, by bits: float32's
    // exponent field is x's minus base (modulo 2^8, the field's width, once
    // it is known to lie in 1..127); zero, denormal and smaller x give 0
    const int hi = hi_word(x), ex = (hi >> 20) & 0x7ff;
    const unsigned v = ((((unsigned)hi << 3) | (lo_word(x) >> 29)) - ((unsigned)base << 23)) & 0x7fffffffu;
    return as_float((ex == 0 || ex - base < 1) ? 0u : (v | ((unsigned)hi & 0x80000000u)));
}

template <bool QUICK>
GKS_HD unsigned teno_code_f32(const double q[5], const TenoT<double>& P)
{
    const double d1 = q[1] - q[0], d2 = q[2] - q[1], d3 = q[3] - q[2], d4 = q[4] - q[3];
    const int h = imax(imax(hi_word(d1) & 0x7fffffff, hi_word(d2) & 0x7fffffff),
                       imax(hi_word(d3) & 0x7fffffff, hi_word(d4) & 0x7fffffff)) >> 20;
    // exponent field of the largest difference (0: all zero or denormal;
    // 2047: infinite or NaN, left to float64)
    const int base = h - 127;
    const float e1 = scaled_float(d1, base), e2 = scaled_float(d2, base), e3 = scaled_float(d3, base),
                e4 = scaled_float(d4, base);
    // 4 eps in the same scale, 2^(2 (1023 - h)) eps4; at most 2^60
    const int ee = -imax(-(P.eps4_e + 2 * (1023 - h)), -60);
    const float eps4 = ee < -126 ? 0.0f : P.eps4_m * as_float((unsigned)(ee + 127) << 23);
    const float A = e2 + e3, B = e1 + e4, C = e3 - e2, D = e4 - e1;
    const float B0 = 3.0f * e2 - e1, C0 = e2 - e1, B2 = 3.0f * e3 - e4, C2 = e4 - e3;
    const float Pp = 7.0f * A - B, R = D - 3.0f * C, u3 = B - A, bq = C - (float)(11.0 / 163.0) * D;
    const float k = (float)(13.0 / 3.0);
    const float t0 = B0 * B0 + (k * C0 * C0 + eps4), t1 = A * A + (k * C * C + eps4);
    const float t2 = B2 * B2 + (k * C2 * C2 + eps4);
    const float t3 = (float)(1.0 / 36.0) * Pp * Pp
                   + ((float)(13.0 / 3.0 * (163.0 / 130.0) * (163.0 / 130.0)) * bq * bq
                      + ((float)(781.0 / 720.0) * u3 * u3 + ((float)(1421461.0 / 327600.0) * R * R + eps4)));
    const float m = fminf(fminf(t0, t1), fminf(t2, t3));
    // m: not lost in the scaling, finite; no square over- or underflows in
    // float64 either
    if (!(m > 1e-30f && m < 1e30f && h < 1423 && (h > 623 || P.eps4_m > 0.0f))) return 0u;
    const float up = 1.0f + P.margin, dn = 1.0f - P.margin;
    float p[4];
    p[3] = teno_pow(quick_div(m, t3), P.q);
    if (QUICK && p[3] > 4.0f * up * P.fct1 && P.fct1 > 1e-25f) return 1u;  // s012 + p[3] < 4
    p[0] = teno_pow(quick_div(m, t0), P.q);
    p[1] = teno_pow(quick_div(m, t1), P.q);
    p[2] = teno_pow(quick_div(m, t2), P.q);
    const float s012 = p[0] + p[1] + p[2];
    const float lim = P.fct1 * (s012 + p[3]), thr = P.fct2 * s012;
    const bool large = p[3] > lim * up, small = p[3] < lim * dn;
    const bool clear = (p[0] > thr * up || p[0] < thr * dn) && (p[1] > thr * up || p[1] < thr * dn) &&
                       (p[2] > thr * up || p[2] < thr * dn);
    if (!(lim > 1e-25f && thr > 1e-25f)) return 0u;  // the cut-offs well inside float32's range
    if (large) return 1u;
    if (!(small && clear)) return 0u;
    return (p[0] > thr ? 2u : 0u) | (p[1] > thr ? 4u : 0u) | (p[2] > thr ? 8u : 0u);
}

// TENO-D (Sec. 4.2) of one stencil: differences, selection, weights
template <bool QUICK = true, typename T>
GKS_HD void teno_select(const T q[5], const TenoT<T>& P, TenoSel<T>& S)
{
    teno_differences(q, S);
    unsigned code = 0;
#ifdef __CUDA_ARCH__
    if constexpr (std::is_same<T, double>::value) code = teno_code_f32<QUICK>(q, P);
#endif
    if (code == 0) {
        T t[4];
        teno_indicators(S, T(4) * P.eps, t);
        code = teno_code<QUICK>(t, P.ct1, P.ct2, P.q);
    }
    S.large = (code & 1u) != 0;
    const int n = ((code >> 1) & 1u) + ((code >> 2) & 1u) + ((code >> 3) & 1u);
    const T inv = n == 1 ? T(1) : (n == 2 ? T(0.5) : T(1.0 / 3.0));
#pragma unroll
    for (int k = 0; k < 3; ++k) S.w[k] = (code & (2u << k)) ? inv : T(0);
}

// 2 sum w_k b_k and 2 sum w_k c_k of the kept sub-stencils
template <typename T>
GKS_HD void teno_small(const TenoSel<T>& S, T& sb, T& sc)
{
    sb = S.w[0] * S.B0 + S.w[1] * S.A + S.w[2] * S.B2;
    sc = S.w[0] * S.C0 + S.w[1] * S.C + S.w[2] * S.C2;
}

// values and xi-derivatives at the faces xi = +1/2 (vp, dp) and -1/2 (vm, dm):
// each value even +- odd.  Large stencil: Eqs. (4.8), (4.9) and their mirror;
// sub-stencils: Eqs. (4.13), (4.14), p_k(+-1/2) = q2 +- b/2 + c/6,
// p_k'(+-1/2) = b +- c
template <typename T>
GKS_HD void teno_faces(const T q[5], const TenoSel<T>& S, T& vp, T& dp, T& vm, T& dm)
{
    T even, odd, de, dod;
    if (S.large) {
        even = S.q2 + T(1.0 / 120.0) * (T(13) * S.C - S.D);
        odd = T(1.0 / 24.0) * S.P;
        de = T(1.0 / 24.0) * (T(13) * S.A - S.B);
        dod = T(1.0 / 24.0) * (T(15) * S.C - S.D);
    } else {
        T sb, sc;
        teno_small(S, sb, sc);
        even = S.q2 + T(1.0 / 12.0) * sc;
        odd = T(0.25) * sb;
        de = T(0.5) * sb;
        dod = T(0.5) * sc;
    }
    vp = even + odd;
    vm = even - odd;
    dp = de + dod;
    dm = de - dod;
    (void)q;
}

// one face of teno_faces: value and xi-derivative at xi = +1/2 (PLUS) or -1/2
template <bool PLUS, typename T>
GKS_HD void teno_face(const T q[5], const TenoSel<T>& S, T& v, T& d)
{
    T vp, dp, vm, dm;
    teno_faces(q, S, vp, dp, vm, dm);
    v = PLUS ? vp : vm;
    d = PLUS ? dp : dm;
}

// WENO5-AO values and xi-derivatives at the faces: the quartic's (Eqs. 4.8,
// 4.9 and mirror) and the quadratics' (Eqs. 4.13, 4.14) blended by S.w3, S.w
template <typename T>
GKS_HD void ao_faces(const T q[5], const TenoSel<T>& S, T& vp, T& dp, T& vm, T& dm)
{
    const T lvp = (T(2) * q[0] - T(13) * q[1] + T(47) * q[2] + T(27) * q[3] - T(3) * q[4]) * T(1.0 / 60.0);
    const T ldp = (q[1] - T(15) * q[2] + T(15) * q[3] - q[4]) * T(1.0 / 12.0);
    const T lvm = (T(-3) * q[0] + T(27) * q[1] + T(47) * q[2] - T(13) * q[3] + T(2) * q[4]) * T(1.0 / 60.0);
    const T ldm = (q[0] - T(15) * q[1] + T(15) * q[2] - q[3]) * T(1.0 / 12.0);
    T svp = T(0), sdp = T(0), svm = T(0), sdm = T(0), ws = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const T w = S.w[k], bh = T(0.5) * S.b[k], c6 = S.c[k] * T(1.0 / 6.0);
        svp += w * (bh + c6);
        svm += w * (c6 - bh);
        sdp += w * (S.b[k] + S.c[k]);
        sdm += w * (S.b[k] - S.c[k]);
        ws += w;
    }
    vp = S.w3 * lvp + ws * S.q2 + svp;
    vm = S.w3 * lvm + ws * S.q2 + svm;
    dp = S.w3 * ldp + sdp;
    dm = S.w3 * ldm + sdm;
}

// WENO5-AO value and xi-derivative at the Gauss point xi = g (xi^2 = 1/12)
template <typename T>
GKS_HD void ao_gauss(const TenoSel<T>& S, T g, T& v, T& d)
{
    T sv = T(0), sd = T(0), ws = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        sv += S.w[k] * S.b[k] * g;
        sd += S.w[k] * (S.b[k] + T(2) * S.c[k] * g);
        ws += S.w[k];
    }
    const T lv = S.q2 + S.u1 * g - S.u3 * g * T(1.0 / 15.0) - S.u4 * T(1.0 / 180.0);
    const T ld = S.u1 + T(2) * S.u2 * g + T(0.1) * S.u3 - T(2.0 / 21.0) * S.u4 * g;
    v = S.w3 * lv + ws * S.q2 + sv;
    d = S.w3 * ld + sd;
}

// values and xi-derivatives at the Gauss points xi = -g (vm, dm) and xi = +g
// (vp, dp), g = 1/(2 sqrt 3), where P2 = 0, P3 = -xi/15, P4 = -1/180,
// P3' = 1/10, P4' = -2 xi/21: each value is E + xi O and each derivative
// Ed + xi Od, with E = q2 - u4/180, O = u1 - u3/15, Ed = u1 + u3/10,
// Od = 2 u2 - 2/21 u4 of the quartic, or q2, sum w b, sum w b, 2 sum w c
template <typename T>
GKS_HD void teno_gauss_pm(const TenoSel<T>& S, T g, T& vm, T& dm, T& vp, T& dp)
{
    T E, O, Ed, Od;
    if (S.large) {
        E = S.q2 - T(1.0 / 4320.0) * S.R;
        O = T(43.0 / 72.0) * S.A - T(7.0 / 72.0) * S.B;
        Ed = T(1.0 / 12.0) * S.P;
        Od = T(12.0 / 9.0) * S.C - T(1.0 / 9.0) * S.D;
    } else {
        T sb;
        teno_small(S, sb, Od);
        E = S.q2;
        O = Ed = T(0.5) * sb;
    }
    vm = E - g * O;
    vp = E + g * O;
    dm = Ed - g * Od;
    dp = Ed + g * Od;
}

// The conventional path (Sec. 3.1, 4.1): WENO5-Z (REC 2) or TENO5 (REC 3)
// face values from the three quadratics, slopes from the quadratic through
// the cell average and the two face values (Eq. 3.11).  The selection keeps,
// per sub-stencil, the part of the weight that does not depend on the point:
// WENO-Z 1 + tau/(beta_k + eps) (Eq. 3.5, tau = |beta_0 - beta_2|), TENO5 the
// cut-off delta_k of Eq. (4.3).  TENO5's chi_k = gamma_k / sum gamma with
// gamma_k = (1 + tau/t_k)^q, t_k = beta_k + eps (Eqs. 4.1, 4.2), is formed
// from gamma_k / gamma_max = ((t_m / t_k) (t_k + tau)/(t_m + tau))^q, t_m the
// smallest t (the largest gamma), so nothing overflows in float32.
template <int REC, typename T>
GKS_HD void weno3_select(const T q[5], const TenoT<T>& P, TenoSel<T>& S)
{
    stencil_coeffs(q, S);
    T beta[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) beta[k] = S.b[k] * S.b[k] + T(13.0 / 3.0) * S.c[k] * S.c[k];
    const T tau = fabs(beta[0] - beta[2]);
    if constexpr (REC == 2) {
#pragma unroll
        for (int k = 0; k < 3; ++k) S.w[k] = T(1) + tau / (beta[k] + P.eps_ao);
    } else {
        T t[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) t[k] = beta[k] + P.eps;
        T m = t[0] < t[1] ? t[0] : t[1];
        m = m < t[2] ? m : t[2];
        const T imt = T(1) / (m + tau);
        T p[3], sum = T(0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const T r = (m / t[k]) * ((t[k] + tau) * imt);
            if (P.q == 6) {
                const T r3 = r * r * r;
                p[k] = r3 * r3;
            } else {
                p[k] = ipow(r, P.q);
            }
            sum += p[k];
        }
        const T thr = P.ct1 * sum;
#pragma unroll
        for (int k = 0; k < 3; ++k) S.w[k] = (p[k] >= thr) ? T(1) : T(0);
    }
    S.w3 = T(0);
    S.large = false;
}

// values at xi = +-1/2 with the linear weights of each face (d = 0.1, 0.6,
// 0.3 at +1/2, mirrored at -1/2), omega_k = d_k w_k / sum d_j w_j, and the
// xi-slopes of Eq. (3.11)
template <typename T>
GKS_HD void weno3_faces(const T q[5], const TenoSel<T>& S, T& vp, T& dp, T& vm, T& dm)
{
    const T dP[3] = {T(0.1), T(0.6), T(0.3)};
    T np = T(0), nm = T(0), sp = T(0), sm = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const T bh = T(0.5) * S.b[k], c6 = S.c[k] * T(1.0 / 6.0);
        const T ap = dP[k] * S.w[k], am = dP[2 - k] * S.w[k];
        np += ap * (bh + c6);  // p_k(+1/2) - q2
        nm += am * (c6 - bh);  // p_k(-1/2) - q2
        sp += ap;
        sm += am;
    }
    const T ep = np / sp, em = nm / sm;
    vp = S.q2 + ep;
    vm = S.q2 + em;
    dp = T(2) * (em + T(2) * ep);
    dm = T(-2) * (T(2) * em + ep);
    (void)q;
}

// WENO5-Z / TENO5 value and xi-derivative at the Gauss point xi = g
// (g^2 = 1/12): the quadratics blended with the point's linear weights (from
// their definition, sum d_k p_k(g) = p_3(g): (210 + sqrt 3)/1080, 11/18,
// (210 - sqrt 3)/1080 at g = -1/(2 sqrt 3), mirrored at +), and the same
// blend's derivative (the tangential derivative of Step 3)
template <typename T>
GKS_HD void weno3_gauss(const TenoSel<T>& S, T g, T& v, T& d)
{
    const T r = T(1.7320508075688772 / 1080.0);
    const T sgn = (g < T(0)) ? T(1) : T(-1);
    const T dk[3] = {T(7.0 / 36.0) + sgn * r, T(11.0 / 18.0), T(7.0 / 36.0) - sgn * r};
    T num = T(0), dnum = T(0), den = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const T a = dk[k] * S.w[k];
        num += a * (S.b[k] * g);                 // p_k(g) - q2 = b g + c (g^2 - 1/12)
        dnum += a * (S.b[k] + T(2) * S.c[k] * g);
        den += a;
    }
    const T iden = T(1) / den;
    v = S.q2 + num * iden;
    d = dnum * iden;
}

// the large-stencil quartic through five averages, value and xi-derivative
// at the Gauss point xi = g (the conventional path's linear reconstruction
// of the equilibrium line averages, Step 4)
template <typename T>
GKS_HD void quartic_gauss(const T q[5], T g, T& v, T& d)
{
    TenoSel<T> S;
    stencil_coeffs(q, S);
    v = S.q2 + S.u1 * g - S.u3 * g * T(1.0 / 15.0) - S.u4 * T(1.0 / 180.0);
    d = S.u1 + T(2) * S.u2 * g + T(0.1) * S.u3 - T(2.0 / 21.0) * S.u4 * g;
}

// the scheme's reconstruction: REC 0 = TENO-D, 1 = WENO5-AO, 2 = WENO5-Z and
// 3 = TENO5 (the conventional path)
template <int REC, bool QUICK = true, typename T>
GKS_HD void rec_select(const T q[5], const TenoT<T>& P, TenoSel<T>& S)
{
    if constexpr (REC == 0) teno_select<QUICK>(q, P, S);
    else if constexpr (REC == 1) ao_select(q, P, S);
    else weno3_select<REC>(q, P, S);
}
template <int REC, typename T>
GKS_HD void rec_faces(const T q[5], const TenoSel<T>& S, T& vp, T& dp, T& vm, T& dm)
{
    if constexpr (REC == 0) teno_faces(q, S, vp, dp, vm, dm);
    else if constexpr (REC == 1) ao_faces(q, S, vp, dp, vm, dm);
    else weno3_faces(q, S, vp, dp, vm, dm);
}
template <int REC, typename T>
GKS_HD void rec_gauss(const TenoSel<T>& S, T g, T& v, T& d)
{
    static_assert(REC != 0, "TENO-D: teno_gauss_pm");
    if constexpr (REC == 1) ao_gauss(S, g, v, d);
    else weno3_gauss(S, g, v, d);
}

// the same at both Gauss points xi = -g (vm, dm) and xi = +g (vp, dp)
template <int REC, typename T>
GKS_HD void rec_gauss_pm(const TenoSel<T>& S, T g, T& vm, T& dm, T& vp, T& dp)
{
    if constexpr (REC == 0) {
        teno_gauss_pm(S, g, vm, dm, vp, dp);
    } else {
        rec_gauss<REC>(S, -g, vm, dm);
        rec_gauss<REC>(S, g, vp, dp);
    }
}

// ------------------------------------------------------------------ characteristic variables
// Sec. 3.1: for Euler systems the reconstructed quantities may be the
// characteristic variables.  Reconstruction code REC_TENO_CHAR is TENO-D on
// C = L W per face: L = R^-1, R the right eigenvectors of the Jacobian of the
// normal Euler flux in the face's local frame (normal velocity first),
// evaluated at the arithmetic mean of the two cells adjacent to the face;
// the reconstructed values and slopes are mapped back by R.  The tangential
// (Gauss-point) reconstruction of the 2-D sweep stays component-wise TENO-D.
constexpr int REC_TENO_CHAR = 4;
// the per-quantity reconstruction a kernel with code REC runs
__host__ __device__ constexpr int rec_base(int REC) { return REC == REC_TENO_CHAR ? 0 : REC; }
// WENO5-Z and TENO5: the conventional path (equilibrium state and slopes
// from their own linear reconstructions)
__host__ __device__ constexpr bool rec_conventional(int REC) { return REC == 2 || REC == 3; }

// Eigen-system of dF/dW at a state with velocity (U, V), sound speed c and
// total enthalpy H: eigenvalues U - c, U (entropy), U (shear; 2-D), U + c in
// slots 0..3 (1-D: slot 2 unused).  b1 = (gamma - 1)/c^2, k = |U|^2/2.
template <typename T> struct CharBasis {
    T U, V, c, ic, H, k, b1;
    bool ok;  // false: the mean state is not physical; projection = identity
};

// basis at the arithmetic mean of the conserved states wa, wb (4 slots,
// energy in slot 3)
template <typename T, int DIM>
GKS_HD void char_basis(const T* wa, const T* wb, T gm1, CharBasis<T>& B)
{
    const T r = T(0.5) * (wa[0] + wb[0]);
    const T ir = T(1) / r;
    B.U = T(0.5) * (wa[1] + wb[1]) * ir;
    B.V = (DIM == 2) ? T(0.5) * (wa[2] + wb[2]) * ir : T(0);
    const T E = T(0.5) * (wa[3] + wb[3]);
    B.k = T(0.5) * (B.U * B.U + B.V * B.V);
    const T p = gm1 * (E - r * B.k);
    B.ok = r > T(0) && p > T(0) && isfinite(p);
    const T c2 = (gm1 + T(1)) * p * ir;
    B.c = B.ok ? M<T>::sqrt_(c2) : T(1);
    B.ic = T(1) / B.c;
    B.H = (E + p) * ir;
    B.b1 = gm1 / c2;
}

// C = L q: with pt = b1 (q3 - U q1 - V q2 + k q0) and t = (q1 - U q0)/c,
// C = ((pt - t)/2, q0 - pt, q2 - V q0, (pt + t)/2)
template <typename T, int DIM>
GKS_HD void char_project(const CharBasis<T>& B, const T* q, T* C)
{
    if (!B.ok) {
#pragma unroll
        for (int i = 0; i < 4; ++i) C[i] = q[i];
        return;
    }
    const T q2 = (DIM == 2) ? q[2] : T(0);
    const T pt = B.b1 * (q[3] - B.U * q[1] - B.V * q2 + B.k * q[0]);
    const T t = B.ic * (q[1] - B.U * q[0]);
    C[0] = T(0.5) * (pt - t);
    C[1] = q[0] - pt;
    C[2] = (DIM == 2) ? q2 - B.V * q[0] : T(0);
    C[3] = T(0.5) * (pt + t);
}

// q = R C: the columns (1, U - c, V, H - U c), (1, U, V, k), (0, 0, 1, V),
// (1, U + c, V, H + U c)
template <typename T, int DIM>
GKS_HD void char_back(const CharBasis<T>& B, const T* C, T* q)
{
    if (!B.ok) {
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = C[i];
        return;
    }
    const T s = C[0] + C[3], d = C[3] - C[0];
    const T c2 = (DIM == 2) ? C[2] : T(0);
    q[0] = s + C[1];
    q[1] = B.U * q[0] + B.c * d;
    q[2] = (DIM == 2) ? B.V * q[0] + c2 : T(0);
    q[3] = B.H * s + B.U * B.c * d + B.k * C[1] + B.V * c2;
}

// Both sides of one face in characteristic variables: w[0..5] are the six
// cells i-2 .. i+3 around the face between cells i and i+1 (4 slots each;
// 1-D slot 2 = 0).  Left side: TENO-D of cells i-2 .. i+2 at xi = +1/2;
// right side: of cells i-1 .. i+3 at xi = -1/2; values and xi-derivatives
// back in conserved variables.
template <typename T, int DIM>
GKS_HD void char_face(const T (*w)[4], const TenoT<T>& P, T gm1, T* vl, T* dl, T* vr, T* dr)
{
    CharBasis<T> B;
    char_basis<T, DIM>(w[2], w[3], gm1, B);
    T C[6][4];
#pragma unroll
    for (int s = 0; s < 6; ++s) char_project<T, DIM>(B, w[s], C[s]);
    T cvl[4], cdl[4], cvr[4], cdr[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (DIM == 1 && k == 2) {
            cvl[k] = cdl[k] = cvr[k] = cdr[k] = T(0);
            continue;
        }
        T q[5];
        TenoSel<T> S;
#pragma unroll
        for (int s = 0; s < 5; ++s) q[s] = C[s][k];
        teno_select(q, P, S);
        teno_face<true>(q, S, cvl[k], cdl[k]);
#pragma unroll
        for (int s = 0; s < 5; ++s) q[s] = C[s + 1][k];
        teno_select(q, P, S);
        teno_face<false>(q, S, cvr[k], cdr[k]);
    }
    char_back<T, DIM>(B, cvl, vl);
    char_back<T, DIM>(B, cdl, dl);
    char_back<T, DIM>(B, cvr, vr);
    char_back<T, DIM>(B, cdr, dr);
}

// ------------------------------------------------------------------ kinetic layer
// The moments of a micro slope need no micro slope.  With <a.psi> the slope
// of a Maxwellian g, rho (a.psi) g is the derivative of rho g, so
//   rho <u^k v^m (a.psi) psi> = d (rho <u^k v^m psi>),
// and the half-space moments u_k = int u^k g du of a normal distribution of
// mean U and variance th = 1/(2 lambda) = p/rho have the derivatives
//   du_k/dU = k u_(k-1),  du_k/dth = k (k-1)/2 u_(k-2)   (k >= 2),
// with a term at u = 0 more for k = 0, 1.  Everything Eqs. (2.5), (2.6),
// (3.25) and (3.26) ask for is then a few products of the moments u_0 .. u_4
// with the slopes of (rho, U, V, th): per point about 520 operations (Euler
// collision time; 205 for tau = 0), against 1120 with the slopes a solved
// from <psi psi> a = b and multiplied into moment matrices up to u_6, which
// also scaled their rounding by lambda^2.  Measured (float32 / float64): one
// step of a 1024^2 plane 0.986 -> 0.844 ms, a 400^2 float64 plane 6.88 ->
// 5.77 ms, a 2^22-cell tube 0.481 -> 0.455 ms; errors against a float64
// evaluation unchanged (5.6e-8, 2.1e-16).

// slopes of one direction (or time): d rho, rho dU, rho dV, dp, rho dth
template <typename T> struct Grad {
    T r, mU, mV, p, mT;
};

// from the slopes d of the conserved variables (gamma - 1 = 2 / (K + D))
template <typename T, int DIM>
GKS_HD void prim_slope(const T* d, T U, T V, T q, T th, T gm1, Grad<T>& s)
{
    s.r = d[0];
    s.mU = fma(-U, d[0], d[1]);
    if constexpr (DIM == 2) {
        s.mV = fma(-V, d[0], d[2]);
        s.p = gm1 * fma(-U, s.mU, fma(-V, s.mV, fma(-q, d[0], d[3])));
    } else {
        s.mV = T(0);
        s.p = gm1 * fma(-U, s.mU, fma(-q, d[0], d[3]));
    }
    s.mT = fma(-th, d[0], s.p);
}

// the time slopes that the compatibility condition <a_n u + a_t v + A> = 0
// gives: the Euler equations in (rho, U, V, th)
template <typename T, int DIM>
GKS_HD void time_slope(const Grad<T>& n, const Grad<T>& t, T U, T V, T th, T gm1, Grad<T>& g)
{
    if constexpr (DIM == 2) {
        const T div = n.mU + t.mV;
        g.r = fma(-U, n.r, fma(-V, t.r, -div));
        g.mU = fma(-U, n.mU, fma(-V, t.mU, -n.p));
        g.mV = fma(-U, n.mV, fma(-V, t.mV, -t.p));
        g.mT = fma(-U, n.mT, fma(-V, t.mT, -(gm1 * th) * div));
    } else {
        g.r = fma(-U, n.r, -n.mU);
        g.mU = fma(-U, n.mU, -n.p);
        g.mV = T(0);
        g.mT = fma(-U, n.mT, -(gm1 * th) * n.mU);
    }
    g.p = fma(th, g.r, g.mT);
}

// a Maxwellian's u-moments (half or full space) with the multiples their
// derivatives take
template <typename T> struct UMom {
    T u0, u1, u2, u3, u4;
    T u1x2, u1x3, u2x3, u2x6, u3x4;
};
template <typename T>
GKS_HD void u_moments(UMom<T>& m, T U, T th, bool fourth)
{
    m.u2 = fma(U, m.u1, th * m.u0);
    m.u1x2 = T(2) * m.u1;
    m.u3 = fma(U, m.u2, th * m.u1x2);
    if (fourth) {
        m.u1x3 = T(3) * m.u1;
        m.u2x3 = T(3) * m.u2;
        m.u4 = fma(U, m.u3, th * m.u2x3);
        m.u2x6 = T(2) * m.u2x3;
        m.u3x4 = T(4) * m.u3;
    }
}

// d(rho u_k), k = 2, 3, 4
template <typename T> GKS_HD T d_u2(const UMom<T>& m, const Grad<T>& g) { return fma(g.mT, m.u0, fma(g.mU, m.u1x2, g.r * m.u2)); }
template <typename T> GKS_HD T d_u3(const UMom<T>& m, const Grad<T>& g) { return fma(g.mT, m.u1x3, fma(g.mU, m.u2x3, g.r * m.u3)); }
template <typename T> GKS_HD T d_u4(const UMom<T>& m, const Grad<T>& g) { return fma(g.mT, m.u2x6, fma(g.mU, m.u3x4, g.r * m.u4)); }

// rho d((V^2 + (K + D - 1) th)/2)
template <int DIM, typename T> GKS_HD T kappa(T V, const Grad<T>& g, T hkv)
{
    return (DIM == 2) ? fma(V, g.mV, hkv * g.mT) : hkv * g.mT;
}

// o (+)= d(rho <u^k psi>) from Dk = d(rho u_k), Dk+1, Dk+2: with
// e = (V^2 + (K + D - 1) th)/2, <u^k psi> = (u_k, u_(k+1), V u_k,
// u_(k+2)/2 + e u_k); kap = rho de
template <bool ADD, typename T, int DIM>
GKS_HD void d_mom(T* o, T Dk, T Dk1, T Dk2, T uk, T V, T e, T mV, T kap)
{
    if constexpr (ADD) {
        o[0] += Dk;
        o[1] += Dk1;
        if constexpr (DIM == 2) o[2] = fma(V, Dk, fma(mV, uk, o[2]));
        o[3] = fma(kap, uk, fma(e, Dk, fma(T(0.5), Dk2, o[3])));
    } else {
        o[0] = Dk;
        o[1] = Dk1;
        o[2] = (DIM == 2) ? fma(V, Dk, mV * uk) : T(0);
        o[3] = fma(kap, uk, fma(e, Dk, T(0.5) * Dk2));
    }
}

// o += d(rho <u^k v psi>), <u^k v psi> = V <u^k psi> + (0, 0, u_k th, u_k th V)
template <typename T>
GKS_HD void d_cross(T* o, T Dk, T Dk1, T Dk2, T uk, T uk1, T uk2, T V, T th, T e, T mV, T mT, T kap)
{
    const T mu = mV * uk, c0 = fma(V, Dk, mu), X = fma(th, Dk, uk * mT);
    o[0] += c0;
    o[1] = fma(V, Dk1, fma(mV, uk1, o[1]));
    o[2] = fma(V, c0 + mu, o[2] + X);
    o[3] = fma(V, fma(T(0.5), Dk2, fma(e, Dk, fma(kap, uk, X))),
               fma(mu, e + th, fma(T(0.5) * mV, uk2, o[3])));
}

// o (+)= rho <u^k psi>
template <bool ADD, typename T, int DIM>
GKS_HD void mom(T* o, T r, T uk, T uk1, T uk2, T V, T e)
{
    const T ru = r * uk, hr = T(0.5) * r;
    if constexpr (ADD) {
        o[0] += ru;
        o[1] = fma(r, uk1, o[1]);
        if constexpr (DIM == 2) o[2] = fma(V, ru, o[2]);
        o[3] = fma(e, ru, fma(hr, uk2, o[3]));
    } else {
        o[0] = ru;
        o[1] = r * uk1;
        o[2] = (DIM == 2) ? V * ru : T(0);
        o[3] = fma(e, ru, hr * uk2);
    }
}

// Start of the half-space moments: h0 = 1/2 erfc(-sg z) (the mass fraction
// on the side sg of u = 0, z = sqrt(lambda) U) and g = exp(-z^2).
// float64: erfc(|z|) = erfcx(|z|) g, so one exponential serves both (erfc
// itself holds a second one).  The rounding of z^2 alone would put a relative
// error of z^2 2^-53 into g and the vanishing half (514 units of 2^-53 at |z| =
// 20 .. 26, 66 at 4 .. 10, where erfc itself is within 4.1); g (1 - lo), lo
// what z^2 lost, takes it out (2.0 and 4.1 at any |z|; z^2 is at most ~1e17
// in a state whose p is resolved) for two operations of the point's ~520.
// float32: erfc by Abramowitz & Stegun 7.1.26
// (Hastings' rational approximation, |error| <= 1.5e-7 on x >= 0), which
// reuses g the same way; its argument is an approximate reciprocal (largest
// absolute error of the half 5.2 units of 2^-24, 4.0 with one rounded to
// nearest, which moves no step's error against a 64-bit evaluation).
template <typename T>
GKS_HD void half_space_start(T z, T sg, T& h0, T& g)
{
    g = M<T>::exp_(-z * z);
    h0 = T(0.5) * M<T>::erfc_(-sg * z);
}
template <>
GKS_HD void half_space_start<double>(double z, double sg, double& h0, double& g)
{
#ifdef __CUDA_ARCH__
    const double zz = z * z;
    g = exp(-zz);
    g = fma(-fma(z, z, -zz), g, g);
    const double h = 0.5 * (g * erfcx(fabs(z)));
    h0 = ((hi_word(z) < 0) == (sg < 0.0)) ? 1.0 - h : h;
#else
    g = exp(-z * z);
    h0 = 0.5 * erfc(-sg * z);
#endif
}
template <>
GKS_HD void half_space_start<float>(float z, float sg, float& h0, float& g)
{
    const float x = fabsf(z);
#ifdef __CUDA_ARCH__
    g = __expf(-x * x);
    const float t = __fdividef(1.0f, fmaf(0.3275911f, x, 1.0f));
#else
    g = expf(-x * x);
    const float t = 1.0f / (1.0f + 0.3275911f * x);
#endif
    const float poly = t * (0.254829592f + t * (-0.284496736f + t * (1.421413741f + t * (-1.453152027f
                     + t * 1.061405429f))));
    const float h = 0.5f * poly * g;  // 1/2 erfc(|z|)
    h0 = (sg * z >= 0.0f) ? 1.0f - h : h;
}

// ------------------------------------------------------------------ time coefficients
// With s = dt/tau, the time integrals of Eq. (2.5) over [0, delta] are
// q_k = tau^{p_k} phi_k(delta/tau), p = (1,2,2,1,2,2).  The flux and its time
// derivative (Sec. 2.2) need F = (4 F(dt/2) - F(dt))/dt and
// dF = 4 (F(dt) - 2 F(dt/2))/dt^2, i.e. per coefficient
//   cF_k = (4 phi_k(s/2) - phi_k(s)) / s^{p_k}
//   cD_k = (phi_k(s) - 2 phi_k(s/2)) / s^{p_k}
// and then  qF_k = cF_k * dt^{p_k-1},  qD_k = 4 cD_k * dt^{p_k-2}.
// Small s: power series (coefficients generated at compile time from the
// Taylor series of exp, plus the 1/s terms of cF_4, cF_5); large s: closed
// forms in y = exp(-s/2) with the polynomial parts cancelled analytically.
template <typename E> struct SeriesTable {
    E c[12][24];
};

constexpr double cx_fact(int n) { return n <= 1 ? 1.0 : n * cx_fact(n - 1); }
constexpr double cx_pow2neg(int n) { return n == 0 ? 1.0 : 0.5 * cx_pow2neg(n - 1); }
// Taylor coefficient a_n of phi_k(x) = sum a_n x^n
constexpr double cx_phi(int k, int n)
{
    const double e = ((n % 2) ? -1.0 : 1.0) / cx_fact(n);  // (-1)^n / n!
    switch (k) {
    case 0: return n >= 2 ? e : 0.0;                   // x - 1 + e^-x
    case 1: return n >= 3 ? (n - 2) * e : 0.0;         // 2 - x - (x+2) e^-x
    case 2: return n >= 3 ? -e : 0.0;                  // x^2/2 - x + 1 - e^-x
    case 3: return n >= 1 ? -e : 0.0;                  // 1 - e^-x
    case 4: return n >= 1 ? (2 - n) * e : 0.0;         // -2 + (x+2) e^-x
    default: return n >= 1 ? e : 0.0;                  // -(1 - e^-x)
    }
}
constexpr int cx_p(int k) { return (k == 0 || k == 3) ? 1 : 2; }
template <typename E>
constexpr SeriesTable<E> make_series_table()
{
    SeriesTable<E> t{};
    for (int k = 0; k < 6; ++k)
        for (int m = 0; m < 24; ++m) {
            const int n = m + cx_p(k);  // coefficient of s^m after dividing by s^p
            const double w2 = cx_pow2neg(n);
            t.c[k][m] = (E)(cx_phi(k, n) * (4.0 * w2 - 1.0));       // cF_k
            t.c[6 + k][m] = (E)(cx_phi(k, n) * (1.0 - 2.0 * w2));   // cD_k
        }
    return t;
}
__constant__ SeriesTable<double> kSeriesD = make_series_table<double>();
__constant__ SeriesTable<float> kSeriesF = make_series_table<float>();
// host copies (operation counting, host replicas)
constexpr SeriesTable<double> kSeriesHostD = make_series_table<double>();
constexpr SeriesTable<float> kSeriesHostF = make_series_table<float>();

template <typename T> struct SeriesOf {
    static GKS_HD T c(int k, int m)
    {
#ifdef __CUDA_ARCH__
        return (T)kSeriesD.c[k][m];
#else
        return (T)kSeriesHostD.c[k][m];
#endif
    }
};
template <> struct SeriesOf<float> {
    static GKS_HD float c(int k, int m)
    {
#ifdef __CUDA_ARCH__
        return kSeriesF.c[k][m];
#else
        return kSeriesHostF.c[k][m];
#endif
    }
};

template <typename T>
GKS_HD void time_coeffs(T s, T is, T* cF, T* cD)  // is = 1 / s
{
    if (s < M<T>::s_series) {
        const int n = (s < T(0.25)) ? (M<T>::nseries / 2) : M<T>::nseries;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            T acc = T(0);
            for (int m = n - 1; m >= 0; --m) acc = acc * s + SeriesOf<T>::c(k, m);
            if (k < 6) cF[k] = acc; else cD[k - 6] = acc;
        }
        // phi_4 and phi_5 start at -x: their x^1 terms leave -1/s in cF_4, cF_5
        // (they cancel in cD); the table holds the powers s^0 and up.
        cF[4] -= is;
        cF[5] -= is;
        return;
    }
    const T is2 = is * is;
    if (s > M<T>::s_noexp) {
        // y = exp(-s/2) is below the working precision next to every other
        // term: the closed forms below with y = 0
        cF[0] = (s - T(3)) * is;
        cD[0] = is;
        cF[1] = (T(6) - s) * is2;
        cD[1] = T(-2) * is2;
        cF[2] = (T(3) - s) * is2;
        cD[2] = (T(0.25) * s * s - T(1)) * is2;
        cF[3] = T(3) * is;
        cD[3] = -is;
        cF[4] = T(-6) * is2;
        cD[4] = T(2) * is2;
        cF[5] = T(-3) * is2;
        cD[5] = is2;
        return;
    }
    const T y = M<T>::exp_(T(-0.5) * s), y2 = y * y;
    const T omy = T(1) - y;
    cF[0] = (s - T(3) + T(4) * y - y2) * is;
    cD[0] = omy * omy * is;
    cF[1] = (T(6) - s - (T(2) * s + T(8)) * y + (s + T(2)) * y2) * is2;
    cD[1] = (T(-2) + (s + T(4)) * y - (s + T(2)) * y2) * is2;
    cF[2] = (T(3) - s - T(4) * y + y2) * is2;
    cD[2] = (T(0.25) * s * s - T(1) + T(2) * y - y2) * is2;
    cF[3] = omy * (T(3) - y) * is;
    cD[3] = -omy * omy * is;
    cF[4] = (T(-6) + (T(2) * s + T(8)) * y - (s + T(2)) * y2) * is2;
    cD[4] = (T(2) - (s + T(4)) * y + (s + T(2)) * y2) * is2;
    cF[5] = -omy * (T(3) - y) * is2;
    cD[5] = omy * omy * is2;
}

// ------------------------------------------------------------------ flux at a point
template <typename T> struct FluxParams {
    T gm1;        // gamma - 1
    T K;          // internal degrees of freedom of this dimension
    T dt;
    T c1, c2, mu; // collision time (Sec. 5)
    T prfac;      // 1/Pr - 1
    T hkv;        // (K + DIM - 1) / 2
    T cp;         // gamma / (gamma - 1) = (K + DIM + 2) / 2
    int tau_mode; // 0 zero, 1 Euler, 2 NS
    int merge = 0; // 0 kinetic weighting (Eqs. 3.25, 3.26), 1 arithmetic average of the sides
};

template <typename T> struct Side {  // one reconstructed side (local frame, 4 slots; 1-D slot 2 = 0)
    T W[4], Wn[4], Wt[4];
};

// Smallest internal-energy fraction (rho e / E) a float32 state may have.
// Below it the float32 pressure has no reliable digits: a reconstructed
// value carries an absolute rounding of ~1e-7 of its stencil's largest
// cell value, which is then a large part of E - rho |U|^2 / 2, and the micro
// slopes scale that error by lambda^2 = (rho / 2p)^2.  (Such points are
// reconstruction artefacts at strong shocks, e.g. a point with p = 7e-6
// beside a cell at p = 21 in the Mach 10 double Mach reflection, where the
// float32 flux came out -522 against 0.2 in float64.)  States of flows
// colder than that need the float64 path.
constexpr double kMinInternalFractionF32 = 1e-4;

// Primitive variables of a conserved state: 1/rho, velocities, V^2/2,
// |U|^2/2, pressure
template <typename T> struct Prim {
    T r, ir, U, V, hv2, q, p;
};

// x > 0 and finite (float64: by its bits, a comparison would run on the
// float64 pipe)
GKS_HD bool pos_finite(double x)
{
    const unsigned hi = (unsigned)hi_word(x);
    return hi < 0x7ff00000u && (hi | lo_word(x)) != 0u;
}
template <typename T>
GKS_HD bool pos_finite(T x)
{
    return x > T(0) && isfinite(x);
}

// Fills s and tests the state: rho > 0 and p > 0 (finite); float32 states
// also need an internal energy of at least kMinInternalFractionF32 of E
template <typename T, int DIM>
GKS_HD bool prim_state(const T* W, T gm1, Prim<T>& s)
{
    s.r = W[0];
    s.ir = T(1) / s.r;
    s.U = W[1] * s.ir;
    s.V = (DIM == 2) ? W[2] * s.ir : T(0);
    s.hv2 = (DIM == 2) ? T(0.5) * s.V * s.V : T(0);
    s.q = fma(T(0.5) * s.U, s.U, s.hv2);
    const T e = fma(-s.r, s.q, W[3]);  // internal energy per volume
    s.p = gm1 * e;
    bool ok = s.r > T(0) && pos_finite(s.p);
    if constexpr (std::is_same<T, double>::value) ok = pos_finite(s.r) && pos_finite(s.p);
    if constexpr (sizeof(T) == 4) ok = ok && e >= T(kMinInternalFractionF32) * W[3];
    return ok;
}
template <typename T, int DIM>
GKS_HD bool physical(const T* W, T gm1)
{
    Prim<T> s;
    return prim_state<T, DIM>(W, gm1, s);
}

// Kinetic merge of two states (values only; Eq. 3.25 with reading R2): the
// conventional path's line-averaged equilibrium state (Step 2).  Both sides
// must be physical.
template <typename T, int DIM>
GKS_HD void merge_values(const T* Wl, const T* Wr, const FluxParams<T>& P, T* W0)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) W0[i] = T(0);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const T* W = side ? Wr : Wl;
        const T sg = side ? T(-1) : T(1);
        const T r = W[0], ir = T(1) / r;
        const T U = W[1] * ir;
        const T V = (DIM == 2) ? W[2] * ir : T(0);
        const T p = P.gm1 * (W[3] - T(0.5) * r * (U * U + V * V));
        const T inv2l = p * ir;
        const T lam = T(0.5) / inv2l;
        const T sl = M<T>::sqrt_(lam);
        T u0, gexp;
        half_space_start<T>(sl * U, sg, u0, gexp);
        const T u1 = U * u0 + sg * T(0.28209479177387814) * gexp / sl;
        const T u2 = U * u1 + inv2l * u0;
        const T v2 = (DIM == 2) ? V * V + inv2l : T(0);
        W0[0] += r * u0;
        W0[1] += r * u1;
        if (DIM == 2) W0[2] += r * u0 * V;
        W0[3] += r * T(0.5) * (u2 + u0 * v2 + u0 * P.K * inv2l);
    }
}

// One side's contributions to the equilibrium state (kinetic merge,
// Eqs. 2.6, 3.25, 3.26) and to the non-equilibrium terms of Eq. (2.5): the
// left side (sg = 1, u > 0) or the right one (sg = -1, u < 0); ADD to the
// sums, or set them.
template <bool ADD, typename T, int DIM, bool NONEQ, bool PRFIX>
GKS_HD void side_terms(const Side<T>& S, const Prim<T>& pr, T sg, const FluxParams<T>& P, T* W0, T* W0n, T* W0t, T* S3, T* S4, T* S5, T* N4,
                       T* N5)
{
    const T r = pr.r, U = pr.U, V = pr.V, q = pr.q, hv2 = pr.hv2;
    const T th = pr.p * pr.ir;               // 1/(2 lambda)
    const T sl = M<T>::rsqrt_(T(2) * th);    // sqrt(lambda)

    // half-space u-moments: u > 0 (left state) or u < 0 (right state);
    // w = +- g(u = 0), the boundary value in the derivatives of u_0, u_1
    UMom<T> m;
    T gz;
    half_space_start<T>(sl * U, sg, m.u0, gz);
    const T w = (sg * T(0.56418958354775628)) * (sl * gz);  // 1/sqrt(pi)
    const T wt = th * w;
    m.u1 = fma(U, m.u0, wt);
    u_moments(m, U, th, NONEQ);
    const T e = fma(P.hkv, th, hv2);

    Grad<T> n, t;
    prim_slope<T, DIM>(S.Wn, U, V, q, th, P.gm1, n);
    const T hit = sl * sl;                   // 1/(2 th)
    const T kn = kappa<DIM>(V, n, P.hkv);
    mom<ADD, T, DIM>(W0, r, m.u0, m.u1, m.u2, V, e);
    const T cn = hit * n.mT;
    const T n0 = fma(n.r, m.u0, w * fma(-U, cn, n.mU));
    const T n1 = fma(n.r, m.u1, fma(n.mU, m.u0, cn * wt));
    const T n2 = d_u2(m, n);
    d_mom<ADD, T, DIM>(W0n, n0, n1, n2, m.u0, V, e, n.mV, kn);
    T t0 = T(0), t1 = T(0), t2 = T(0), kt = T(0);
    if constexpr (DIM == 2) {
        prim_slope<T, DIM>(S.Wt, U, V, q, th, P.gm1, t);
        kt = kappa<DIM>(V, t, P.hkv);
        const T ct = hit * t.mT;
        t0 = fma(t.r, m.u0, w * fma(-U, ct, t.mU));
        t1 = fma(t.r, m.u1, fma(t.mU, m.u0, ct * wt));
        t2 = d_u2(m, t);
        d_mom<ADD, T, DIM>(W0t, t0, t1, t2, m.u0, V, e, t.mV, kt);
    } else if constexpr (!ADD) {
#pragma unroll
        for (int i = 0; i < 4; ++i) W0t[i] = T(0);
    }

    if constexpr (NONEQ) {
        Grad<T> g;  // time derivative of the side's Maxwellian
        time_slope<T, DIM>(n, t, U, V, th, P.gm1, g);
        const T kg = kappa<DIM>(V, g, P.hkv);
        const T cg = hit * g.mT;
        const T g1 = fma(g.r, m.u1, fma(g.mU, m.u0, cg * wt));
        const T g2 = d_u2(m, g);
        if constexpr (PRFIX) {  // density moments of the A and slope terms (heat flux)
            const T g0 = fma(g.r, m.u0, w * fma(-U, cg, g.mU));
            d_mom<ADD, T, DIM>(N5, g0, g1, g2, m.u0, V, e, g.mV, kg);
        }
        // flux moments of the side terms of Eq. (2.5) over the half space
        mom<ADD, T, DIM>(S3, r, m.u1, m.u2, m.u3, V, e);
        d_mom<ADD, T, DIM>(S5, g1, g2, d_u3(m, g), m.u1, V, e, g.mV, kg);
        const T n3 = d_u3(m, n);
        if constexpr (PRFIX) {
            d_mom<ADD, T, DIM>(N4, n1, n2, n3, m.u1, V, e, n.mV, kn);
            if constexpr (DIM == 2) d_cross<T>(N4, t0, t1, t2, m.u0, m.u1, m.u2, V, th, e, t.mV, t.mT, kt);
        }
        d_mom<ADD, T, DIM>(S4, n2, n3, d_u4(m, n), m.u2, V, e, n.mV, kn);
        if constexpr (DIM == 2) d_cross<T>(S4, t1, t2, d_u3(m, t), m.u1, m.u2, m.u3, V, th, e, t.mV, t.mT, kt);
    }
}

// The equilibrium state g0: rho0 <u psi>_0 (F0) is the Euler flux of W0,
// rho0 <u A0 psi>_0 (F2) its time derivative, and rho0 <u (a0n u + a0t v)
// psi>_0 (F1) is d_n rho0 <u^2 psi>_0 + d_t rho0 <u v psi>_0
template <typename T> struct Equilibrium {
    T U, V, q, p;   // velocities, |U|^2/2, pressure
    Grad<T> g;      // time slopes
    T F0[4], F1[4], F2[4];
};
template <typename T, int DIM, bool NONEQ>
GKS_HD void equilibrium(const T* W0, const T* W0n, const T* W0t, const FluxParams<T>& P, Equilibrium<T>& E)
{
    const T r0 = W0[0], ir0 = T(1) / r0;
    const T U0 = W0[1] * ir0;
    const T V0 = (DIM == 2) ? W0[2] * ir0 : T(0);
    const T hv2 = (DIM == 2) ? T(0.5) * V0 * V0 : T(0);
    const T q0 = fma(T(0.5) * U0, U0, hv2);
    const T p0 = P.gm1 * fma(-r0, q0, W0[3]);
    const T Ep = W0[3] + p0, th0 = p0 * ir0;
    E.U = U0;
    E.V = V0;
    E.q = q0;
    E.p = p0;
    Grad<T> n, t;
    Grad<T>& g = E.g;
    prim_slope<T, DIM>(W0n, U0, V0, q0, th0, P.gm1, n);
    if constexpr (DIM == 2) prim_slope<T, DIM>(W0t, U0, V0, q0, th0, P.gm1, t);
    time_slope<T, DIM>(n, t, U0, V0, th0, P.gm1, g);
    E.F0[0] = W0[1];
    E.F0[1] = fma(W0[1], U0, p0);
    E.F0[2] = (DIM == 2) ? W0[1] * V0 : T(0);
    E.F0[3] = U0 * Ep;
    const T mt = fma(U0, g.r, g.mU);  // d(rho U)
    E.F2[0] = mt;
    E.F2[1] = fma(U0, mt + g.mU, g.p);
    E.F2[2] = (DIM == 2) ? fma(V0, mt, U0 * g.mV) : T(0);
    // rho U H: H d(rho U) + U rho dH, rho dH = U rho dU + V rho dV + cp rho dth
    T rdH = fma(U0, g.mU, P.cp * g.mT);
    if constexpr (DIM == 2) rdH = fma(V0, g.mV, rdH);
    E.F2[3] = fma(Ep * ir0, mt, U0 * rdH);
    if constexpr (NONEQ) {
        UMom<T> m;
        m.u0 = T(1);
        m.u1 = U0;
        u_moments(m, U0, th0, true);
        const T e = fma(P.hkv, th0, hv2);
        const T kn = kappa<DIM>(V0, n, P.hkv);
        d_mom<false, T, DIM>(E.F1, d_u2(m, n), d_u3(m, n), d_u4(m, n), m.u2, V0, e, n.mV, kn);
        if constexpr (DIM == 2)
            d_cross<T>(E.F1, fma(t.r, U0, t.mU), d_u2(m, t), d_u3(m, t), U0, m.u2, m.u3, V0, th0, e, t.mV, t.mT,
                       kappa<DIM>(V0, t, P.hkv));
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) E.F1[i] = T(0);
    }
}

// collision time over dt (Sec. 5), from the sides' pressures and p0
template <typename T>
GKS_HD T tau_over_dt(const FluxParams<T>& P, T pl, T pr, T p0, T idt)
{
    const T jump = fabs(pl - pr) / (pl + pr);
    return (P.tau_mode == 1) ? P.c1 + P.c2 * jump : P.mu * idt / p0 + P.c2 * jump;
}

// F and dF/dt (per unit time; Sec. 2.2) at one interface point in the local
// frame, from the left and right sides (sg = 1; the other way round with
// sg = -1).  state(0, L, p) and state(1, R, p) form a side's primitive variables
// (prim_state) and apply the caller's fallback where it is not physical.
// need_F = false: only dF is formed (the second stage uses nothing else).
// W0n_lin, W0_lin, W0t_lin: the conventional path's equilibrium normal
// slope (Eq. 3.12, in 2-D reconstructed to the point), state and tangential
// slope (2-D: linear reconstructions of line-averaged merges, Step 4),
// replacing the kinetic merge at the point; nullptr otherwise
template <typename T, int DIM, bool NONEQ, bool PRFIX, typename State>
GKS_HD void point_flux(Side<T>& L, Side<T>& R, T sg, const FluxParams<T>& P, T* F, T* dF, bool need_F, State&& state,
                       const T* W0n_lin = nullptr, const T* W0_lin = nullptr, const T* W0t_lin = nullptr)
{
    T W0[4], W0n[4], W0t[4], S3[4], S4[4], S5[4], N4[4], N5[4];
    Prim<T> pl, pr;
    state(0, L, pl);
    state(1, R, pr);
    side_terms<false, T, DIM, NONEQ, PRFIX>(L, pl, sg, P, W0, W0n, W0t, S3, S4, S5, N4, N5);
    side_terms<true, T, DIM, NONEQ, PRFIX>(R, pr, -sg, P, W0, W0n, W0t, S3, S4, S5, N4, N5);
    // the kinetic merge is also the density moment of the side terms (the
    // heat flux needs it even where W0 is replaced below)
    T W0k[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) W0k[i] = W0[i];
    if (P.merge == 1) {
        // arithmetic average of the two sides in place of the kinetic
        // weighting (Sec. 3.2, for smooth flow); the side terms stay
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            W0[i] = T(0.5) * (L.W[i] + R.W[i]);
            W0n[i] = T(0.5) * (L.Wn[i] + R.Wn[i]);
            W0t[i] = T(0.5) * (L.Wt[i] + R.Wt[i]);
        }
    }
    if (W0n_lin) {
#pragma unroll
        for (int i = 0; i < 4; ++i) W0n[i] = W0n_lin[i];
    }
    if (W0_lin) {
#pragma unroll
        for (int i = 0; i < 4; ++i) W0[i] = W0_lin[i];
    }
    if (W0t_lin) {
#pragma unroll
        for (int i = 0; i < 4; ++i) W0t[i] = W0t_lin[i];
    }

    Equilibrium<T> E;
    equilibrium<T, DIM, NONEQ>(W0, W0n, W0t, P, E);
    const T *F0 = E.F0, *F1 = E.F1, *F2 = E.F2;

    if (P.tau_mode == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            F[i] = F0[i];
            dF[i] = F2[i];
        }
        return;
    }
    T cF[6], cD[6];
    const T dt = P.dt, idt = T(1) / dt;
    const T is = tau_over_dt(P, pl.p, pr.p, E.p, idt);
    time_coeffs<T>(T(1) / is, is, cF, cD);
    // Prandtl correction: F_E += (1/Pr - 1) q, q the heat flux relative to
    // (U0, V0) expanded in raw moments of the same time-dependent f.
    // Density moments: rho0 <psi>_0 = W0, rho0 <(a_n u + a_t v) psi>_0 =
    // -W0_time, rho0 <A0 psi>_0 = W0_time; side terms W0k (the kinetic
    // merge), N4, N5.
    T W0time[4] = {T(0), T(0), T(0), T(0)};
    T cf = T(0), uk = T(0);
    const T U0 = E.U, V0 = E.V;
    if constexpr (PRFIX) {
        const Grad<T>& g = E.g;
        W0time[0] = g.r;
        W0time[1] = g.mU + U0 * g.r;
        W0time[2] = g.mV + V0 * g.r;
        W0time[3] = E.q * g.r + U0 * g.mU + V0 * g.mV + (P.cp - T(1)) * g.p;  // 1/(gamma - 1) = cp - 1
        cf = E.q + U0 * U0;
        uk = U0 * E.q;
    }
    auto combine = [&](const T* c, T s1, T s2, T* o) {
        // q_k = c_k s1 for p_k = 1 (k = 0, 3), c_k s2 for p_k = 2
        const T c0 = c[0] * s1, c1 = c[1] * s2, c2 = c[2] * s2, c3 = c[3] * s1, c4 = c[4] * s2, c5 = c[5] * s2;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            o[i] = fma(c0, F0[i], fma(c1, F1[i], fma(c2, F2[i], fma(c3, S3[i], fma(c4, S4[i], c5 * S5[i])))));
        if constexpr (PRFIX) {
            T Mo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                Mo[i] = c0 * W0[i] + (c2 - c1) * W0time[i] + c3 * W0k[i] + c4 * N4[i] + c5 * N5[i];
            o[3] += P.prfac * (o[3] - U0 * o[1] - V0 * o[2] + cf * o[0] + U0 * V0 * Mo[2] - U0 * Mo[3] - uk * Mo[0]);
        }
    };
    // qF_k = cF_k dt^{p_k - 1}, qD_k = 4 cD_k dt^{p_k - 2}
    if (need_F) combine(cF, T(1), dt, F);
    combine(cD, T(4) * idt, T(4), dF);
}

// the same for two physical sides
template <typename T, int DIM>
struct PlainState {
    T gm1;
    GKS_HD void operator()(int, Side<T>& S, Prim<T>& p) const { prim_state<T, DIM>(S.W, gm1, p); }
};
template <typename T, int DIM, bool NONEQ, bool PRFIX>
GKS_HD void point_flux(Side<T>& L, Side<T>& R, const FluxParams<T>& P, T* F, T* dF)
{
    point_flux<T, DIM, NONEQ, PRFIX>(L, R, T(1), P, F, dF, true, PlainState<T, DIM>{P.gm1});
}

}  // namespace gks
