// gks_adjoint.cu -- hand-written discrete adjoint of the 2-D S2O4 step
// (collision-free flux, tau = 0) with checkpointing (include/gks.h,
// gks_adjoint_* and gks_vjp_step).
//
// One step of the scheme (Sec. 2.2, dimension by dimension, fixed dt):
//   W*      = W^n - dt/h  d(F/2 + dt/8 dF)(W^n)     (both directions)
//   A       = W^n - dt/h  d(F + dt/6 dF)(W^n)
//   W^{n+1} = A   - dt/h  d(dt/3 dF)(W*)
// where d is the face difference and (F, dF) the Gauss-averaged face flux
// and its time derivative.  Given lam = dJ/dW^{n+1}, the adjoint step is
//   lam*  = [d dF/dW*]^T (dt^2/(3h) Delta lam)
//   lam^n = lam + lam* + [dF/dW^n]^T (dt/h Delta(lam + lam*/2))
//                      + [d dF/dW^n]^T (dt^2/h Delta(lam/6 + lam*/8))
// with Delta lam the difference of lam across a face (zero outside the
// interior).  The transposed flux Jacobian of one direction is applied by
// three kernels on the stage input:
//   k_adj_lines   normal TENO-D per cell -> face-line values and slopes
//                 (the forward sweep's phase 1)
//   k_adj_gauss   per face segment and Gauss point: tangential TENO-D to the
//                 Gauss point (forward), the reverse of the point flux, then
//                 the transposed tangential reconstruction; sums, per tile,
//                 the contributions to each line row, and writes the tile's
//                 own rows and the two rows beyond each of its edges
//   k_adj_normal  per cell: gathers the line cotangents of its two faces,
//                 applies the transposed normal reconstruction and sums what
//                 the cells of its neighbourhood contribute to it
// and the ghost layers are folded back onto the interior cells they copy
// (the transpose of the ghost fill).  TENO-D selections are recomputed from
// the same stage inputs as in the forward pass, i.e. frozen at the forward
// pass's choice.  Every sum is a gather in a fixed order, so the result does
// not depend on scheduling (only the positivity fallback, which smooth flows
// do not take, adds with atomics).
//
// Checkpointing: gks_adjoint_forward keeps W every k steps; the backward pass
// recomputes each k-step segment from its checkpoint, stage by stage, keeping
// W and W* of every step, and runs the segment's adjoint steps in reverse.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "../../include/gks.h"
#include "gks_adjoint.cuh"
#include "gks_ctx.h"

using namespace gks;

namespace {

constexpr int NQ = 16;  // line quantities per face segment: [vL, sL, vR, sR] x 4 variables

// One direction of one stage.  Orientation: dirn 0 = faces normal to x
// (normal index = x, unit stride), dirn 1 = faces normal to y.  Scratch
// arrays are laid out with the unit-stride grid direction fastest.
struct AdjDir {
    const double* src;    // stage input, float64 path (ghosts filled)
    const float* srcf;    // stage input, float32 path (float32 shadow, ghosts filled)
    const double* lam1;   // cotangent fields (ghosted; interior used)
    const double* lam2;   // may be null
    double cF1, cD1, cF2, cD2;
    // float32 copies of the scalars, converted on the host (a float64 ->
    // float32 conversion in every thread would run on the slow float64 pipe)
    float fcF1, fcD1, fcF2, fcD2, fihn, fiht;
    void* lines;          // [NQ][faces nn+1][rows nt+4]
    void* contrib;        // line cotangents: [NQ][faces nn+1][rows ntp], then [NQ][faces][tiles][4] edge rows
    double* gW;           // ghosted gradient accumulator
    int dirn, nn, nt;
    int tiles, ntp;       // Gauss-row tiles of adj_tile(dirn) rows, rows padded to whole tiles
    long long sn, st;     // element strides along normal / tangential
    double ihn, iht;
};

__device__ __forceinline__ int gvar_(int v, bool swap) { return (swap && (v == 1 || v == 2)) ? 3 - v : v; }

// scratch indices: faces f in [0, nn], line rows r in [-2, nt+2), Gauss rows
// in [0, nt), cells i in [-1, nn]
template <int D>
__device__ __forceinline__ long long lidx(const AdjDir& a, int f, int r)
{
    return D == 0 ? (long long)(r + 2) * (a.nn + 1) + f : (long long)f * (a.nt + 4) + (r + 2);
}
// A k_adj_gauss block holds 128 face segments (float64: 64, as a block's time
// is its share of the float64 pipe): 16 along the unit stride.  Rows of its
// tile along the tangential direction:
template <typename T> constexpr int ADJ_PAIRS = sizeof(T) == 4 ? 128 : 64;
__host__ __device__ constexpr int adj_tile(int dirn, bool f32) { return dirn == 0 ? (f32 ? 8 : 4) : 16; }
// line cotangents: own rows of a tile, and its edge rows e = 0, 1 (the two
// rows before it) and 2, 3 (after it)
template <int D>
__device__ __forceinline__ long long midx(const AdjDir& a, int f, int r)
{
    return D == 0 ? (long long)r * (a.nn + 1) + f : (long long)f * a.ntp + r;
}
template <int D>
__device__ __forceinline__ long long eidx(const AdjDir& a, int f, int tile, int e)
{
    return D == 0 ? (long long)(tile * 4 + e) * (a.nn + 1) + f : (long long)f * (a.tiles * 4) + tile * 4 + e;
}
// a direction scalar in the arithmetic type
template <typename T>
__device__ __forceinline__ T scal(double d, float f)
{
    if constexpr (sizeof(T) == 4) return f;
    else return d;
}

template <typename T>
__device__ __forceinline__ T load_src(const AdjDir& a, long long gi)
{
    if constexpr (sizeof(T) == 4) return a.srcf[gi];
    else return a.src[gi];
}

// map the launch to (normal index, tangential index): the unit-stride grid
// direction runs along threadIdx.x
template <int D>
__device__ __forceinline__ void map2(int& n, int& t, int n0, int t0)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (D == 0) { n = n0 + x; t = t0 + y; }
    else { n = n0 + y; t = t0 + x; }
}

// frozen selection as 4 bits: large, and the kept small stencils
template <typename T>
__device__ __forceinline__ unsigned sel_code(const TenoSel<T>& S)
{
    if (S.large) return 1u;
    return (S.w[0] > T(0) ? 2u : 0u) | (S.w[1] > T(0) ? 4u : 0u) | (S.w[2] > T(0) ? 8u : 0u);
}

template <typename T>
__device__ __forceinline__ void sel_decode(unsigned c, TenoSel<T>& S)
{
    S.large = (c & 1u) != 0;
    const T d0 = (c & 2u) ? T(1) : T(0), d1 = (c & 4u) ? T(1) : T(0), d2 = (c & 8u) ? T(1) : T(0);
    const T dsum = d0 + d1 + d2;
    const T inv = S.large ? T(0) : T(1) / dsum;  // as teno_select: d_k / sum d
    S.w[0] = d0 * inv;
    S.w[1] = d1 * inv;
    S.w[2] = d2 * inv;
}

// The forward's TENO-D of two stencils (qa, qb) in the forward's arithmetic:
// the float32 sweep reconstructs variable pairs (0, 1), (2, 3) and, per face
// side, the value and normal-slope streams as packed pairs, so the same
// pairs here reproduce its values and selections bit for bit.  Returns the
// two selection codes (qa in bits 0-3, qb in bits 4-7).
template <typename T>
__device__ __forceinline__ unsigned fwd_faces2(const T qa[5], const T qb[5], const TenoT<T>& P, T* vp, T* dp, T* vm,
                                               T* dm)
{
    if constexpr (sizeof(T) == 4) {
        f2 qq[5];
#pragma unroll
        for (int s = 0; s < 5; ++s) qq[s] = f2(qa[s], qb[s]);
        TenoSel2 S2;
        f2 a, b, c, d;
        const bool both = teno_select_x2(qq, P, S2);
        if (both) teno_faces_x2(S2, true, a, b, c, d);
        else teno_faces_x2(S2, false, a, b, c, d);
        vp[0] = a.x(); dp[0] = b.x(); vm[0] = c.x(); dm[0] = d.x();
        vp[1] = a.y(); dp[1] = b.y(); vm[1] = c.y(); dm[1] = d.y();
        return both ? 0x11u : sel_code_x(S2) | (sel_code_y(S2) << 4);
    } else {
        unsigned code = 0;
        const T* q[2] = {qa, qb};
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            TenoSel<T> S;
            teno_select(q[l], P, S);
            teno_faces(q[l], S, vp[l], dp[l], vm[l], dm[l]);
            code |= sel_code(S) << (4 * l);
        }
        return code;
    }
}
template <typename T>
__device__ __forceinline__ unsigned fwd_gauss2(const T qa[5], const T qb[5], const TenoT<T>& P, T gA, T gB, T* va,
                                               T* da, T* vb, T* db)
{
    if constexpr (sizeof(T) == 4) {
        f2 qq[5];
#pragma unroll
        for (int s = 0; s < 5; ++s) qq[s] = f2(qa[s], qb[s]);
        TenoSel2 S2;
        f2 a, b, c, d;
        const bool both = teno_select_x2(qq, P, S2);
        if (both) teno_gauss_pm_x2(S2, true, gB, a, b, c, d);  // gA = -gB
        else teno_gauss_pm_x2(S2, false, gB, a, b, c, d);
        va[0] = a.x(); da[0] = b.x(); vb[0] = c.x(); db[0] = d.x();
        va[1] = a.y(); da[1] = b.y(); vb[1] = c.y(); db[1] = d.y();
        return both ? 0x11u : sel_code_x(S2) | (sel_code_y(S2) << 4);
    } else {
        unsigned code = 0;
        const T* q[2] = {qa, qb};
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            TenoSel<T> S;
            teno_select(q[l], P, S);
            teno_gauss_pm(S, gB, va[l], da[l], vb[l], db[l]);  // gA = -gB, as the forward
            code |= sel_code(S) << (4 * l);
        }
        return code;
    }
}

// ---- phase 1: normal TENO-D of the stage input (as the forward sweep)
template <typename T, int D>
__global__ void __launch_bounds__(256) k_adj_lines(GridDev g, AdjDir a, TenoT<T> tn)
{
    int i, r;
    map2<D>(i, r, -1, -2);
    if (i > a.nn || r >= a.nt + 2) return;
    const bool swap = D != 0;
    const long long org = (long long)NG * g.pitch + NG;
    const long long LP = (long long)(a.nn + 1) * (a.nt + 4);
    T* L = static_cast<T*>(a.lines);
    const T ih = scal<T>(a.ihn, a.fihn);
    {
        const int vv = 2 * (int)blockIdx.z;  // variable pairs (0, 1), (2, 3), as the forward
        T q[2][5];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const long long base = (long long)gvar_(vv + l, swap) * g.plane + org + r * a.st;
#pragma unroll
            for (int s = 0; s < 5; ++s) q[l][s] = load_src<T>(a, base + (i - 2 + s) * a.sn);
        }
        T vp[2], dp[2], vm[2], dm[2];
        fwd_faces2(q[0], q[1], tn, vp, dp, vm, dm);
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const int v = vv + l;
            if (i + 1 <= a.nn) {
                L[(0 * 4 + v) * LP + lidx<D>(a, i + 1, r)] = vp[l];
                L[(1 * 4 + v) * LP + lidx<D>(a, i + 1, r)] = dp[l] * ih;
            }
            if (i >= 0) {
                L[(2 * 4 + v) * LP + lidx<D>(a, i, r)] = vm[l];
                L[(3 * 4 + v) * LP + lidx<D>(a, i, r)] = dm[l] * ih;
            }
        }
    }
}

// ---- Gauss points: forward tangential TENO-D, reverse point flux, transposed
// tangential TENO-D.  Two adjacent lanes hold the two Gauss points of one face
// segment; lane 0 finishes the left side's quantities, lane 1 the right's.
//
// A face segment contributes to the five line rows of its stencil.  Writing
// the five contributions of 16 quantities (80 values per segment, read once
// by k_adj_normal) was most of both kernels' memory traffic; the block's 128
// segments now add theirs up in shared memory, and 1.25 to 1.5 values per
// segment and quantity go out.
//
// Bound by its chain of dependent arithmetic at few warps per SM, so float32
// runs three blocks of 256 threads at 80 registers (some values spill) rather
// than two at 128, and a segment that keeps its large stencils throughout (one
// compare of its codes) skips the sub-stencils: with the direction a template
// parameter, 12 steps and their reverse on a 512^2 float32 plane 9.86 -> 9.07
// ms, 4 on a 96^2 float64 plane 5.45 -> 5.35 ms.
template <typename T, int D>
__global__ void __launch_bounds__(2 * ADJ_PAIRS<T>, (sizeof(T) == 4) ? 3 : 2)
k_adj_gauss(GridDev g, AdjDir a, FluxParams<T> fp, TenoT<T> tt)
{
    constexpr int NP = ADJ_PAIRS<T>;
    __shared__ T sc[8][5][NP];  // [side, variable][stencil position][segment]
    const int gp = threadIdx.x & 1;
    const int x = (blockIdx.x * blockDim.x + threadIdx.x) >> 1, y = blockIdx.y * blockDim.y + threadIdx.y;
    int f, r;
    if (D == 0) { f = x; r = y; }
    else { f = y; r = x; }
    const bool valid = f <= a.nn && r < a.nt;
    const int fc = valid ? f : 0, rc = valid ? r : 0;  // in-range indices for the idle lanes' loads
    const bool swap = D != 0;
    const long long org = (long long)NG * g.pitch + NG;
    const long long LP = (long long)(a.nn + 1) * (a.nt + 4);
    const T* Lq = static_cast<const T*>(a.lines);
    const T iht = scal<T>(a.iht, a.fiht);

    // forward, as the forward sweep: lane gp reconstructs side gp (0: left,
    // 1: right) at both Gauss points, keeps its own point and hands the other
    // point's values to its partner; L is the own side, R the partner's
    Side<T> L, R;
    unsigned codes = 0;  // selections of the own side: 4 bits per quantity kk * 4 + v
    const T gs = gp ? T(0.28867513459481288) : T(-0.28867513459481288);
    {
        const int ls = D == 0 ? a.nn + 1 : 1;  // element stride of line rows
        const T* Lp = Lq + (long long)(8 * gp) * LP + lidx<D>(a, fc, rc - 2);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            // the side's value and normal-slope streams as one pair, as the forward
            T q[2][5];
            T va[2], da[2], vb[2], db[2];
            const T *pv = Lp + v * LP, *ps = Lp + (4 + v) * LP;
#pragma unroll
            for (int s = 0; s < 5; ++s) {
                q[0][s] = pv[s * ls];
                q[1][s] = ps[s * ls];
            }
            const unsigned c2 = fwd_gauss2(q[0], q[1], tt, -gs, gs, vb, db, va, da);
            codes |= (c2 & 15u) << (4 * v);
            codes |= (c2 >> 4) << (4 * (4 + v));
            L.W[v] = va[0];
            R.W[v] = __shfl_xor_sync(0xffffffffu, vb[0], 1);
            L.Wt[v] = da[0] * iht;
            R.Wt[v] = __shfl_xor_sync(0xffffffffu, db[0], 1) * iht;
            L.Wn[v] = va[1];
            R.Wn[v] = __shfl_xor_sync(0xffffffffu, vb[1], 1);
        }
    }
    // positivity fallback, as the forward: the adjacent cell average, zero slopes
    const bool fbL = valid && !physical<T, 2>(L.W, fp.gm1);
    const bool fbR = valid && !physical<T, 2>(R.W, fp.gm1);
    const int cL = fc - 1 + gp, cR = fc - gp;  // normal index of the cell beside the face on the own / partner's side
    if (fbL || fbR) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const long long b = (long long)gvar_(v, swap) * g.plane + org + rc * a.st;
            if (fbL) { L.W[v] = load_src<T>(a, b + cL * a.sn); L.Wn[v] = L.Wt[v] = T(0); }
            if (fbR) { R.W[v] = load_src<T>(a, b + cR * a.sn); R.Wn[v] = R.Wt[v] = T(0); }
        }
    }
    // face cotangents (each Gauss point carries weight 1/2).  The
    // differences are taken in float64, the rest in the working precision;
    // the two lanes of a face split the variables (lane gp: 2 gp, 2 gp + 1)
    // and exchange them, so each float64 difference (the float64 pipe is the
    // slow one) is formed once per face
    T gF[4], gdF[4];
    {
        const T cF1 = scal<T>(a.cF1, a.fcF1), cF2 = scal<T>(a.cF2, a.fcF2);
        const T cD1 = scal<T>(a.cD1, a.fcD1), cD2 = scal<T>(a.cD2, a.fcD2);
        T mF[2], mD[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int v = 2 * gp + h;
            const long long b = (long long)gvar_(v, swap) * g.plane + org + rc * a.st;
            // lam of the cells on either side (zero outside the interior);
            // one float64 subtraction per difference
            const double p1 = fc < a.nn ? a.lam1[b + fc * a.sn] : 0.0;
            const double m1 = fc >= 1 ? a.lam1[b + (fc - 1) * a.sn] : 0.0;
            T e1 = from_f64<T>(p1 - m1), e2 = T(0);
            if (a.lam2) {
                const double p2 = fc < a.nn ? a.lam2[b + fc * a.sn] : 0.0;
                const double m2 = fc >= 1 ? a.lam2[b + (fc - 1) * a.sn] : 0.0;
                e2 = from_f64<T>(p2 - m2);
            }
            mF[h] = T(0.5) * (cF1 * e1 + cF2 * e2);
            mD[h] = T(0.5) * (cD1 * e1 + cD2 * e2);
        }
        const T oF0 = __shfl_xor_sync(0xffffffffu, mF[0], 1), oF1 = __shfl_xor_sync(0xffffffffu, mF[1], 1);
        const T oD0 = __shfl_xor_sync(0xffffffffu, mD[0], 1), oD1 = __shfl_xor_sync(0xffffffffu, mD[1], 1);
        gF[0] = gp ? oF0 : mF[0];
        gF[1] = gp ? oF1 : mF[1];
        gF[2] = gp ? mF[0] : oF0;
        gF[3] = gp ? mF[1] : oF1;
        gdF[0] = gp ? oD0 : mD[0];
        gdF[1] = gp ? oD1 : mD[1];
        gdF[2] = gp ? mD[0] : oD0;
        gdF[3] = gp ? mD[1] : oD1;
    }
    Side<T> gL, gR;
#pragma unroll
    for (int v = 0; v < 4; ++v) gL.W[v] = gL.Wn[v] = gL.Wt[v] = gR.W[v] = gR.Wn[v] = gR.Wt[v] = T(0);
    if (valid) point_flux_vjp(L, R, gp ? T(-1) : T(1), fp, gF, gdF, gL, gR);
    if (fbL || fbR) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const long long b = (long long)gvar_(v, swap) * g.plane + org + rc * a.st;
            if (fbL) {
                atomicAdd(&a.gW[b + cL * a.sn], (double)gL.W[v]);
                gL.W[v] = gL.Wn[v] = gL.Wt[v] = T(0);
            }
            if (fbR) {
                atomicAdd(&a.gW[b + cR * a.sn], (double)gR.W[v]);
                gR.W[v] = gR.Wn[v] = gR.Wt[v] = T(0);
            }
        }
    }
    // exchange: each lane keeps its own side and receives that side's
    // cotangents at the partner's point
    T oW[4], oWn[4], oWt[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        oW[v] = __shfl_xor_sync(0xffffffffu, gR.W[v], 1);
        oWn[v] = __shfl_xor_sync(0xffffffffu, gR.Wn[v], 1);
        oWt[v] = __shfl_xor_sync(0xffffffffu, gR.Wt[v], 1);
    }
    const int pair = threadIdx.y * 16 + (threadIdx.x >> 1), tid = threadIdx.y * 32 + threadIdx.x;
    const int TT = adj_tile(D, sizeof(T) == 4), NF = NP / TT;  // the tile's rows and faces
    const int tile = D == 0 ? blockIdx.y : blockIdx.x, f0 = (D == 0 ? blockIdx.x : blockIdx.y) * NF;
    const long long MP = (long long)(a.nn + 1) * a.ntp, EP = (long long)(a.nn + 1) * a.tiles * 4;
    T* M = static_cast<T*>(a.contrib);
    T* Eg = M + NQ * MP;
    const bool all_large = codes == 0x11111111u;
#pragma unroll 1
    for (int kk = 0; kk < 2; ++kk) {  // values, then normal slopes, of both sides
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            TenoSel<T> S;
            S.large = true;
            if (!all_large) sel_decode((codes >> (4 * (kk * 4 + v))) & 15u, S);
            T gq[5];
            if (kk == 0) teno_gauss_pm_T(S, gs, oW[v], oWt[v] * iht, gL.W[v], gL.Wt[v] * iht, gq);
            else teno_gauss_pm_T(S, gs, oWn[v], T(0), gL.Wn[v], T(0), gq);
#pragma unroll
            for (int s = 0; s < 5; ++s) sc[gp * 4 + v][s][pair] = valid ? gq[s] : T(0);
        }
        __syncthreads();
        // line row l - 2 of the tile from the segments of rows l - s; 16
        // segments of a row (dirn 0) or of a face (dirn 1) are adjacent
        for (int k = tid; k < 8 * (TT + 4) * NF; k += 2 * NP) {
            int l, fl, qq;
            if (D == 0) { fl = k % 16; l = (k / 16) % (NP / 16 + 4); qq = k / (NP + 64); }
            else { l = k % 20; fl = (k / 20) % (NP / 16); qq = k / (20 * (NP / 16)); }
            const int f2_ = f0 + fl;
            if (f2_ > a.nn) continue;
            T acc = T(0);
#pragma unroll
            for (int s = 0; s < 5; ++s) {
                const int rl = l - s;
                if (rl >= 0 && rl < TT) acc += sc[qq][s][D == 0 ? rl * 16 + fl : fl * 16 + rl];
            }
            const int qi = (2 * (qq >> 2) + kk) * 4 + (qq & 3);
            if (l >= 2 && l < TT + 2) M[qi * MP + midx<D>(a, f2_, tile * TT + l - 2)] = acc;
            else Eg[qi * EP + eidx<D>(a, f2_, tile, l < 2 ? l : l - TT)] = acc;
        }
        __syncthreads();
    }
}

// ---- per cell: line cotangents of its faces -> transposed normal TENO-D,
// and the sum of what the cells around hand it.  The block's cells lie along
// the normal (x faces: 128, y faces: 32 rows of 8); the contributions meet in
// shared memory, so only the inner cells (all but two at either end) are the
// block's own.  The five contributions of a cell through memory and a gather
// kernel of its own took 22 + 11 us on a 512^2 float32 plane
// (its gradient over 12 steps 9.07 -> 8.89 ms, 4 steps of a 96^2 float64
// plane 5.35 -> 5.19 ms).
template <int D> constexpr int ADJ_NX = D == 0 ? 128 : 8;  // block shape
template <int D> constexpr int ADJ_NY = 256 / ADJ_NX<D>;
template <int D> constexpr int ADJ_OWN = (D == 0 ? ADJ_NX<D> : ADJ_NY<D>) - 4;  // own cells along the normal

template <typename T, int D>
__global__ void __launch_bounds__(256) k_adj_normal(GridDev g, AdjDir a, TenoT<T> tn)
{
    __shared__ T part[2][5][256];
    const int tid = threadIdx.y * ADJ_NX<D> + threadIdx.x;
    // cell i (two before the block's first own cell onwards), line row r
    const int k = D == 0 ? threadIdx.x : threadIdx.y;
    const int i = (int)blockIdx.y * ADJ_OWN<D> - 5 + k;
    const int r = (int)(D == 0 ? blockIdx.x * ADJ_NY<D> + threadIdx.y : blockIdx.x * ADJ_NX<D> + threadIdx.x) - 2;
    const bool swap = D != 0;
    const long long org = (long long)NG * g.pitch + NG;
    const long long MP = (long long)(a.nn + 1) * a.ntp, EP = (long long)(a.nn + 1) * a.tiles * 4;
    const T* M = static_cast<const T*>(a.contrib);
    const T* Eg = M + NQ * MP;
    const T ih = scal<T>(a.ihn, a.fihn);
    // line row r: its tile's sum, and the edge rows of the tiles beside it
    const int TT = adj_tile(D, sizeof(T) == 4);
    int own = -1, e1 = -1, e2 = -1, t1 = 0, t2 = 0;  // own row; edge rows of tiles t1, t2
    if (r < 0) { t1 = 0; e1 = r + 2; }
    else if (r >= a.ntp) { t1 = a.tiles - 1; e1 = 2 + r - a.ntp; }
    else {
        const int tl = r / TT, m = r - tl * TT;
        own = r;
        if (m >= TT - 2 && tl + 1 < a.tiles) { t1 = tl + 1; e1 = m - (TT - 2); }
        if (m < 2 && tl > 0) { t2 = tl - 1; e2 = 2 + m; }
    }
    auto gline = [&](int q, int f) {
        T acc = T(0);
        if (e1 >= 0) acc += Eg[q * EP + eidx<D>(a, f, t1, e1)];
        if (own >= 0) acc += M[q * MP + midx<D>(a, f, own)];
        if (e2 >= 0) acc += Eg[q * EP + eidx<D>(a, f, t2, e2)];
        return acc;
    };
    const int vv = 2 * (int)blockIdx.z;  // variable pairs, as the forward's selection
    if (i < -1 || i > a.nn || r >= a.nt + 2) {
#pragma unroll
        for (int s = 0; s < 10; ++s) part[s / 5][s % 5][tid] = T(0);
    } else {
        T q[2][5];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const long long base = (long long)gvar_(vv + l, swap) * g.plane + org + r * a.st;
#pragma unroll
            for (int s = 0; s < 5; ++s) q[l][s] = load_src<T>(a, base + (i - 2 + s) * a.sn);
        }
        T fvp[2], fdp[2], fvm[2], fdm[2];
        const unsigned c2 = fwd_faces2(q[0], q[1], tn, fvp, fdp, fvm, fdm);
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const int v = vv + l;
            T gvp = T(0), gdp = T(0), gvm = T(0), gdm = T(0);
            if (i + 1 <= a.nn) {
                gvp = gline(0 * 4 + v, i + 1);
                gdp = gline(1 * 4 + v, i + 1) * ih;
            }
            if (i >= 0) {
                gvm = gline(2 * 4 + v, i);
                gdm = gline(3 * 4 + v, i) * ih;
            }
            TenoSel<T> S;
            sel_decode((c2 >> (4 * l)) & 15u, S);  // the forward's selection
            T gq[5] = {T(0), T(0), T(0), T(0), T(0)};
            teno_faces_T(S, gvp, gdp, gvm, gdm, gq);
#pragma unroll
            for (int s = 0; s < 5; ++s) part[l][s][tid] = gq[s];
        }
    }
    __syncthreads();
    if (k < 2 || k >= 2 + ADJ_OWN<D> || i > a.nn + 2 || r >= a.nt + 2) return;
    constexpr int step = D == 0 ? 1 : ADJ_NX<D>;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        T acc = T(0);
#pragma unroll
        for (int s = 0; s < 5; ++s) acc += part[l][s][tid + (2 - s) * step];  // cell i + 2 - s holds i at its position s
        a.gW[(long long)gvar_(vv + l, swap) * g.plane + org + i * a.sn + r * a.st] += to_f64(acc);
    }
}

// ---- transpose of the ghost fill: y ghost rows first (over the full ghosted
// width), then the x ghost columns of the interior rows.  One thread per
// (column or row, variable) walks its six ghost cells in a fixed order.
// The six ghosts and their source cells are read at once and added up in a
// fixed order in registers (one after the other through memory they cost a
// round trip each).  tang, norm: the line holds the tangential / the normal
// momentum of these ghosts.
__device__ __forceinline__ void fold_line(double* P, long long stride, int n, int bc0, int bc1, bool tang, bool norm)
{
    double x[2 * NG], s[2 * NG];
    int src[2 * NG];
#pragma unroll
    for (int k = 0; k < 2 * NG; ++k) {
        const int j = k < NG ? k : n + k;
        bool fn, fa;
        src[k] = ghost_src(k < NG ? bc0 : bc1, n, j, fn, fa);
        const double y = P[j * stride];
        x[k] = ((norm && (fn || fa)) || (tang && fa)) ? -y : y;
        s[k] = P[src[k] * stride];
    }
#pragma unroll
    for (int k = 0; k < 2 * NG; ++k) {
        s[k] += x[k];
#pragma unroll
        for (int m = k + 1; m < 2 * NG; ++m)
            if (src[m] == src[k]) s[m] = s[k];  // the same source again: go on from its sum
        P[src[k] * stride] = s[k];
        P[(k < NG ? k : n + k) * stride] = 0.0;
    }
}

__global__ void k_fold_y(GridDev g, double* gW)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int gx = g.nx + 2 * NG;
    if (idx >= 4 * gx) return;
    const int v = idx / gx, i = idx % gx;
    double* P = gW + (long long)v * g.plane + i;
    fold_line(P, g.pitch, g.ny, g.bc[2], g.bc[3], v == 1, v == 2);
}

__global__ void k_fold_x(GridDev g, double* gW)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 4 * g.ny) return;
    const int v = idx / g.ny, j = NG + idx % g.ny;
    double* P = gW + (long long)v * g.plane + (long long)j * g.pitch;
    fold_line(P, 1, g.nx, g.bc[0], g.bc[1], v == 2, v == 1);
}

// out = a + b + c (whole ghosted arrays)
__global__ void k_sum3(const double* __restrict__ a, const double* __restrict__ b, const double* __restrict__ c,
                       double* __restrict__ out, long long n)
{
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x) out[i] = a[i] + b[i] + c[i];
}

__global__ void k_shadow(const double* __restrict__ W, float* __restrict__ Wf, long long n)
{
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x) Wf[i] = narrow(W[i]);
}

int blocks_for(long long n) { return (int)std::min<long long>((n + 255) / 256, 4096); }

}  // namespace

struct gks_adjoint {
    gks_ctx* c = nullptr;
    int k = 1;
    int nsteps = 0;
    double dt = 0.0;
    bool have_forward = false;
    std::vector<double*> ckpt;   // W at steps 0, k, 2k, ... (ghosted)
    // the stage inputs W and W* of the segment being reversed, from the
    // recomputation, as the adjoint kernels read them: in the kernels'
    // precision, ghosts filled
    std::vector<void*> seg, segs;
    double* WN = nullptr;        // final state of the forward pass
    double *lam = nullptr, *lams = nullptr, *gacc = nullptr, *nxt = nullptr;
    void *lines = nullptr, *contrib = nullptr;
    long long launches = 0;
    // one full segment's recomputation and reverse sweep, captured once and
    // replayed for every full segment (fixed buffers; dt and the context's
    // parameters are baked in)
    cudaGraphExec_t seg_exec = nullptr;
    double seg_dt = 0.0;
    long long seg_version = -1, seg_kernels = 0, seg_ctx_kernels = 0;
    bool seg_eager = false;  // the segment does not return its buffers to place: no graph
};

namespace {

gks_status adj_alloc(gks_adjoint* A, double** p)
{
    gks_ctx* c = A->c;
    if (!*p) CK(cudaMalloc(p, c->arr_bytes));
    return GKS_OK;
}

gks_status adj_scratch(gks_adjoint* A)
{
    gks_ctx* c = A->c;
    if (A->lines) return GKS_OK;
    const long long nx = c->desc.nx, ny = c->desc.ny;
    const size_t es = c->desc.precision == GKS_FP32_FLUX ? 4 : 8;
    const long long lines = std::max((nx + 1) * (ny + 4), (ny + 1) * (nx + 4)) * NQ;
    long long contrib = 0;  // line cotangents: own rows of whole tiles and four edge rows per tile
    for (int d = 0; d < 2; ++d) {
        const long long nn = d == 0 ? nx : ny, nt = d == 0 ? ny : nx, tt = adj_tile(d, es == 4);
        const long long tiles = (nt + tt - 1) / tt;
        contrib = std::max(contrib, (nn + 1) * tiles * (tt + 4) * NQ);
    }
    CK(cudaMalloc(&A->lines, lines * es));
    CK(cudaMalloc(&A->contrib, contrib * es));
    gks_status s;
    if ((s = adj_alloc(A, &A->lam)) || (s = adj_alloc(A, &A->lams)) || (s = adj_alloc(A, &A->gacc)) ||
        (s = adj_alloc(A, &A->nxt)))
        return s;
    return GKS_OK;
}

// load a ghosted float64 state into the context's W (and its float32 shadow)
gks_status load_state(gks_adjoint* A, const double* Wg)
{
    gks_ctx* c = A->c;
    CK(cudaMemcpyAsync(c->W, Wg, c->arr_bytes, cudaMemcpyDeviceToDevice, c->stream));
    if (c->Wf) {
        const long long n = (long long)c->nv * c->g.plane;
        k_shadow<<<blocks_for(n), 256, 0, c->stream>>>(c->W, c->Wf, n);
        CK(cudaGetLastError());
        ++A->launches;
    }
    return GKS_OK;
}

template <typename T, int D>
gks_status sweep_vjp_t(gks_adjoint* A, AdjDir d)
{
    gks_ctx* c = A->c;
    const HostFlux hf = rt::host_flux(c);
    const FluxParams<T> fp = make_flux_params<T>(hf);
    const TenoT<T> tn = teno_t<T>(rt::teno_params(c, false)), tt = teno_t<T>(rt::teno_params(c, true));
    const GridDev& g = c->g;
    cudaStream_t st = c->stream;
    // launch shapes: x along the unit-stride direction
    auto grid_for = [&](int nnorm, int ntan, dim3 blk, int xmul) {
        const int ex = D == 0 ? nnorm : ntan, ey = D == 0 ? ntan : nnorm;
        return dim3((unsigned)((ex * xmul + blk.x - 1) / blk.x), (unsigned)((ey + blk.y - 1) / blk.y));
    };
    const dim3 b256(32, 8), bg(32, ADJ_PAIRS<T> / 16);
    // the per-cell kernels take the two variable pairs in blockIdx.z
    dim3 gcell = grid_for(d.nn + 2, d.nt + 4, b256, 1);
    gcell.z = 2;
    k_adj_lines<T, D><<<gcell, b256, 0, st>>>(g, d, tn);
    k_adj_gauss<T, D><<<grid_for(d.nn + 1, d.nt, bg, 2), bg, 0, st>>>(g, d, fp, tt);
    constexpr int across = D == 0 ? ADJ_NY<D> : ADJ_NX<D>;
    const dim3 gn((d.nt + 4 + across - 1) / across, (d.nn + 6 + ADJ_OWN<D> - 1) / ADJ_OWN<D>, 2);
    k_adj_normal<T, D><<<gn, dim3(ADJ_NX<D>, ADJ_NY<D>), 0, st>>>(g, d, tn);
    CK(cudaGetLastError());
    A->launches += 3;
    return GKS_OK;
}

// adds to A->gacc the transposed flux Jacobian of both directions at the
// stage input, with face cotangents from lam1, lam2
gks_status stage_vjp(gks_adjoint* A, const void* input, const double* lam1, const double* lam2, double cF1,
                     double cD1, double cF2, double cD2)
{
    gks_ctx* c = A->c;
    const bool f32 = c->desc.precision == GKS_FP32_FLUX;
    for (int dirn = 0; dirn < 2; ++dirn) {
        AdjDir d{};
        d.src = static_cast<const double*>(input);
        d.srcf = static_cast<const float*>(input);
        d.lam1 = lam1;
        d.lam2 = lam2;
        const double h = dirn == 0 ? c->g.dx : c->g.dy;
        d.cF1 = cF1 / h;
        d.cD1 = cD1 / h;
        d.cF2 = cF2 / h;
        d.cD2 = cD2 / h;
        d.lines = A->lines;
        d.contrib = A->contrib;
        d.gW = A->gacc;
        d.dirn = dirn;
        if (dirn == 0) {
            d.nn = c->desc.nx; d.nt = c->desc.ny; d.sn = 1; d.st = c->g.pitch;
            d.ihn = 1.0 / c->g.dx; d.iht = 1.0 / c->g.dy;
        } else {
            d.nn = c->desc.ny; d.nt = c->desc.nx; d.sn = c->g.pitch; d.st = 1;
            d.ihn = 1.0 / c->g.dy; d.iht = 1.0 / c->g.dx;
        }
        const int tt = adj_tile(dirn, f32);
        d.tiles = (d.nt + tt - 1) / tt;
        d.ntp = d.tiles * tt;
        d.fcF1 = (float)d.cF1;
        d.fcD1 = (float)d.cD1;
        d.fcF2 = (float)d.cF2;
        d.fcD2 = (float)d.cD2;
        d.fihn = (float)d.ihn;
        d.fiht = (float)d.iht;
        gks_status s = f32 ? (dirn == 0 ? sweep_vjp_t<float, 0>(A, d) : sweep_vjp_t<float, 1>(A, d))
                           : (dirn == 0 ? sweep_vjp_t<double, 0>(A, d) : sweep_vjp_t<double, 1>(A, d));
        if (s) return s;
    }
    const GridDev& g = c->g;
    k_fold_y<<<(4 * (g.nx + 2 * NG) + 127) / 128, 128, 0, c->stream>>>(g, A->gacc);
    k_fold_x<<<(4 * g.ny + 127) / 128, 128, 0, c->stream>>>(g, A->gacc);
    CK(cudaGetLastError());
    A->launches += 2;
    return GKS_OK;
}

// bytes of a state in the kernels' precision
size_t work_bytes(const gks_ctx* c)
{
    return (size_t)c->nv * c->g.plane * (c->Wsf ? sizeof(float) : sizeof(double));
}

// A->lam <- (dW^{n+1}/dW^n)^T A->lam at the ghosted state Wn with its stage
// state Ws (as the forward pass computed it)
gks_status adjoint_step(gks_adjoint* A, const void* Wn, const void* Ws)
{
    gks_ctx* c = A->c;
    const double dt = A->dt;
    gks_status s;
    // lam* = [d dF/dW*]^T (dt^2/(3h) Delta lam)
    CK(cudaMemsetAsync(A->gacc, 0, c->arr_bytes, c->stream));
    if ((s = stage_vjp(A, Ws, A->lam, nullptr, 0.0, dt * dt / 3.0, 0.0, 0.0))) return s;
    std::swap(A->lams, A->gacc);
    // stage 1 at W^n with the cotangents of A (lam) and of W* (lam*)
    CK(cudaMemsetAsync(A->gacc, 0, c->arr_bytes, c->stream));
    if ((s = stage_vjp(A, Wn, A->lam, A->lams, dt, dt * dt / 6.0, 0.5 * dt, dt * dt / 8.0))) return s;
    const long long n = (long long)c->nv * c->g.plane;
    k_sum3<<<blocks_for(n), 256, 0, c->stream>>>(A->lam, A->lams, A->gacc, A->nxt, n);
    CK(cudaGetLastError());
    ++A->launches;
    std::swap(A->lam, A->nxt);
    return GKS_OK;
}

// checkpoints for nsteps steps and the k segment states (W and W*), kept
// for the adjoint's lifetime
gks_status reserve(gks_adjoint* A, int nsteps)
{
    gks_ctx* c = A->c;
    const int ncp = (nsteps + A->k - 1) / A->k;
    while ((int)A->ckpt.size() < ncp) {
        double* p = nullptr;
        if (cudaMalloc(&p, c->arr_bytes) != cudaSuccess) {
            cudaGetLastError();
            return rt::fail(c, GKS_ENOMEM, "no device memory for %d checkpoints", ncp);
        }
        A->ckpt.push_back(p);
    }
    while ((int)A->seg.size() < A->k) {
        void *p = nullptr, *q = nullptr;
        if (cudaMalloc(&p, work_bytes(c)) != cudaSuccess || cudaMalloc(&q, work_bytes(c)) != cudaSuccess) {
            cudaFree(p);
            cudaGetLastError();
            return rt::fail(c, GKS_ENOMEM, "no device memory for a %d-step segment", A->k);
        }
        A->seg.push_back(p);
        A->segs.push_back(q);
    }
    return GKS_OK;
}

gks_status check_supported(gks_ctx* c)
{
    if (c->desc.dim != 2) return rt::fail(c, GKS_EUNSUPPORTED, "the adjoint is built for 2-D grids");
    if (c->sch.tau_mode != GKS_TAU_ZERO)
        return rt::fail(c, GKS_EUNSUPPORTED, "the adjoint is built for the collision-free flux (tau_mode = zero)");
    if (c->sch.recon != GKS_RECON_TENO_D || c->sch.charvars)
        return rt::fail(c, GKS_EUNSUPPORTED,
                        "the adjoint is built for component-wise TENO-D (frozen stencil selection)");
    for (int k = 0; k < 4; ++k)
        if (c->desc.bc[k] > GKS_BC_REFLECT)
            return rt::fail(c, GKS_EUNSUPPORTED, "the adjoint is built for the copying boundary rules");
    if (c->sch.merge != GKS_MERGE_KINETIC)
        return rt::fail(c, GKS_EUNSUPPORTED, "the adjoint is built for the kinetic merge");
    return GKS_OK;
}

gks_status sync_check(gks_ctx* c)
{
    gks_diag d;
    return gks_get_diagnostics(c, &d);
}

}  // namespace

// ====================================================================== C ABI
extern "C" {

gks_status gks_adjoint_create(gks_ctx* c, int checkpoint_every, gks_adjoint** out)
{
    if (!c || !out || checkpoint_every < 1) return GKS_EINVAL;
    *out = nullptr;
    gks_status s = check_supported(c);
    if (s) return s;
    gks_adjoint* A = new (std::nothrow) gks_adjoint();
    if (!A) return GKS_ENOMEM;
    A->c = c;
    A->k = checkpoint_every;
    if ((s = adj_scratch(A)) || (s = adj_alloc(A, &A->WN))) {
        gks_adjoint_destroy(A);
        cudaGetLastError();
        return s == GKS_ECUDA ? GKS_ENOMEM : s;
    }
    *out = A;
    return GKS_OK;
}

void gks_adjoint_destroy(gks_adjoint* A)
{
    if (!A) return;
    if (A->seg_exec) cudaGraphExecDestroy(A->seg_exec);
    for (double* p : A->ckpt) cudaFree(p);
    for (void* p : A->seg) cudaFree(p);
    for (void* p : A->segs) cudaFree(p);
    cudaFree(A->WN);
    cudaFree(A->lam);
    cudaFree(A->lams);
    cudaFree(A->gacc);
    cudaFree(A->nxt);
    cudaFree(A->lines);
    cudaFree(A->contrib);
    delete A;
}

gks_status gks_adjoint_forward(gks_adjoint* A, int nsteps, double dt)
{
    const NvtxRange range("gks_adjoint_forward");
    if (!A || nsteps < 1 || !(dt > 0.0) || !std::isfinite(dt)) return GKS_EINVAL;
    gks_ctx* c = A->c;
    gks_status s = check_supported(c);
    if (s) return s;
    if ((s = reserve(A, nsteps))) return s;
    A->have_forward = false;
    for (int n = 0; n < nsteps; ++n) {
        if (n % A->k == 0) CK(cudaMemcpyAsync(A->ckpt[n / A->k], c->W, c->arr_bytes, cudaMemcpyDeviceToDevice, c->stream));
        if ((s = gks_step(c, dt))) return s;
    }
    CK(cudaMemcpyAsync(A->WN, c->W, c->arr_bytes, cudaMemcpyDeviceToDevice, c->stream));
    if ((s = sync_check(c))) return s;
    A->nsteps = nsteps;
    A->dt = dt;
    A->have_forward = true;
    return GKS_OK;
}

namespace {

// recompute a segment of len steps from the state in the context, stage by
// stage (the same kernels and W as the forward pass's steps), keeping W and
// W* of every step, then reverse its steps
gks_status run_segment(gks_adjoint* A, int len)
{
    gks_ctx* c = A->c;
    gks_status s;
    const void* w = c->Wf ? static_cast<const void*>(c->Wf) : static_cast<const void*>(c->W);
    const void* ws = c->Wsf ? static_cast<const void*>(c->Wsf) : static_cast<const void*>(c->Ws);
    for (int n = 0; n < len; ++n) {
        CK(cudaMemcpyAsync(A->seg[n], w, work_bytes(c), cudaMemcpyDeviceToDevice, c->stream));
        if ((s = rt::fill_ghosts(c, A->seg[n], c->stream))) return s;
        if ((s = gks_stage(c, 1, A->dt))) return s;
        CK(cudaMemcpyAsync(A->segs[n], ws, work_bytes(c), cudaMemcpyDeviceToDevice, c->stream));
        if ((s = rt::fill_ghosts(c, A->segs[n], c->stream))) return s;
        if (n + 1 < len && (s = gks_stage(c, 2, A->dt))) return s;
    }
    for (int n = len - 1; n >= 0; --n)
        if ((s = adjoint_step(A, A->seg[n], A->segs[n]))) return s;
    return GKS_OK;
}

// capture run_segment(k) as a graph (once per dt and context parameters);
// leaves seg_exec null where the segment's buffer rotation does not return
// to its start (odd k) so that replays would read the wrong buffers
gks_status segment_graph(gks_adjoint* A)
{
    gks_ctx* c = A->c;
    if (A->seg_eager) return GKS_OK;
    if (A->seg_exec && A->seg_dt == A->dt && A->seg_version == c->param_version) return GKS_OK;
    if (A->seg_exec) {
        cudaGraphExecDestroy(A->seg_exec);
        A->seg_exec = nullptr;
    }
    if (!c->cap_stream) CK(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
    double* const before[4] = {A->lam, A->lams, A->gacc, A->nxt};
    const long long L0 = A->launches, C0 = c->launches;
    cudaStream_t keep = c->stream;
    c->stream = c->cap_stream;
    CK(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
    c->capturing = true;
    gks_status s = run_segment(A, A->k);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(c->cap_stream, &graph);
    c->capturing = false;
    c->stream = keep;
    A->seg_kernels = A->launches - L0;
    A->seg_ctx_kernels = c->launches - C0;
    A->launches = L0;  // captured, not launched
    c->launches = C0;
    const bool in_place = A->lam == before[0] && A->lams == before[1] && A->gacc == before[2] && A->nxt == before[3];
    A->lam = before[0], A->lams = before[1], A->gacc = before[2], A->nxt = before[3];
    if (s != GKS_OK || e != cudaSuccess || !in_place) {
        if (graph) cudaGraphDestroy(graph);
        cudaGetLastError();
        if (s != GKS_OK) return s;
        if (e != cudaSuccess) return rt::fail(c, GKS_ECUDA, "capturing the adjoint segment: %s", cudaGetErrorString(e));
        A->seg_eager = true;
        return GKS_OK;
    }
    e = cudaGraphInstantiate(&A->seg_exec, graph, 0);
    cudaGraphDestroy(graph);
    CK(e);
    A->seg_dt = A->dt;
    A->seg_version = c->param_version;
    return GKS_OK;
}

}  // namespace

gks_status gks_adjoint_backward(gks_adjoint* A, const double* gWN, double* gW0, int on_device)
{
    const NvtxRange range("gks_adjoint_backward");
    if (!A || !gWN || !gW0) return GKS_EINVAL;
    gks_ctx* c = A->c;
    if (!A->have_forward) return rt::fail(c, GKS_EINVAL, "gks_adjoint_backward needs a completed forward pass");
    // W and the device's dt change below, also where a replayed segment runs no
    // host code that would say so
    c->cfl_dt_ready = false;
    gks_status s;
    if ((s = reserve(A, A->nsteps))) return s;
    CK(cudaMemsetAsync(A->lam, 0, c->arr_bytes, c->stream));
    if ((s = rt::copy_interior(c, A->lam, gWN, on_device, true))) return s;
    const int ncp = (A->nsteps + A->k - 1) / A->k;
    for (int sgi = ncp - 1; sgi >= 0; --sgi) {
        const int n0 = sgi * A->k, n1 = std::min(n0 + A->k, A->nsteps);
        const NvtxRange seg_range("adjoint segment");
        if ((s = load_state(A, A->ckpt[sgi]))) return s;
        if (n1 - n0 == A->k) {
            if ((s = segment_graph(A))) return s;
            if (A->seg_exec) {
                CK(cudaGraphLaunch(A->seg_exec, c->stream));
                A->launches += A->seg_kernels;
                c->launches += A->seg_ctx_kernels;
                continue;
            }
        }
        if ((s = run_segment(A, n1 - n0))) return s;
    }
    if ((s = rt::copy_interior(c, A->lam, gW0, on_device, false))) return s;
    // leave the context at the forward pass's final state
    if ((s = load_state(A, A->WN))) return s;
    return sync_check(c);
}

long long gks_adjoint_launches(const gks_adjoint* A) { return A ? A->launches : 0; }

gks_status gks_adjoint_reserve(gks_adjoint* A, int nsteps)
{
    if (!A || nsteps < 1) return GKS_EINVAL;
    return reserve(A, nsteps);
}

gks_status gks_vjp_step(gks_ctx* c, const double* W, const double* gout, double* gin, double dt, int on_device)
{
    if (!c || !W || !gout || !gin || !(dt > 0.0) || !std::isfinite(dt)) return GKS_EINVAL;
    gks_adjoint* A = nullptr;
    gks_status s = gks_adjoint_create(c, 1, &A);
    if (s) return s;
    if (!(s = gks_set_state(c, W, on_device)) && !(s = gks_adjoint_forward(A, 1, dt)))
        s = gks_adjoint_backward(A, gout, gin, on_device);
    gks_adjoint_destroy(A);
    return s;
}

}  // extern "C"
