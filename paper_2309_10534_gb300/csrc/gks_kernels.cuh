// gks_kernels.cuh -- kernels of one S2O4 step of the TENO-D gas-kinetic scheme.
//
// Data layout (HBM): conserved variables, float64, SoA with three ghost
// layers: W[v][j][i], v < nvar, j < gy = ny + 6 (1-D: gy = 1), i < pitch
// (pitch >= nx + 6, a multiple of 16 doubles).  Interior cell (0, 0) sits at
// (j, i) = (3, 3) (1-D: i = 3).  Three such arrays live on the device:
//   W  -- the state W^n (and W^{n+1} after stage 2)
//   Ws -- the stage state W*
//   Ac -- the stage accumulator W^n - dt/dx d(F + dt/6 dF)   (Sec. 2.2)
// Kernels of one step (2-D): sweep-x s1, sweep-y s1, sweep-x s2, sweep-y s2
// (+ CFL reduction and commit).  1-D: stage 1, stage 2 (the same).  The blocks
// at the boundary load their ghost cells by the boundary rules, and the last
// block of a step's last kernel commits the step: four (two) launches a step
// instead of seven (five).  A sweep computes every face flux of its tile
// once, in shared memory, so both neighbours of a face apply bit-identical
// values and the update is conservative.
#pragma once

#include "gks_device.cuh"
#include "gks_pair.cuh"

namespace gks {

constexpr int NG = 3;

struct DevState {
    double t, dt, t_end, cfl;
    unsigned long long sigma;      // max over cells of the signal rate, as ordered bits
    unsigned long long fallbacks;  // positivity fallbacks taken
    long long steps, max_steps;
    unsigned int err;              // bit 0 non-physical update, bit 1 fallback failed
    unsigned int done;             // 1: t_end or max_steps reached; kernels return early
    unsigned int fixed_dt;         // 1: keep dt (caller-given), 0: CFL time step
    unsigned int ticket;           // blocks of a committing kernel that have finished
    long long steps0;              // steps before the present gks_advance_to
    unsigned int idle;             // 1: that call found t_end already reached
};

// state-setting boundary rules: conserved states (energy in slot 3) and the
// moving oblique shock x_s(y, t) = x0 + (y - oy) cot + vx t
struct BcStates {
    double in[4], pre[4];
    double x0, cot, vx;
};

struct GridDev {
    int dim, nx, ny, pitch, gy;
    long long plane;   // elements per variable plane = gy * pitch
    double dx, dy;
    int bc[4];
    double gamma, mu;
    double ox, oy;     // domain origin (cell centres at ox + (i + 1/2) dx)
    BcStates bs;
};

constexpr int BC_INFLOW = 5, BC_WALL_AFTER_X0 = 6, BC_MOVING_SHOCK = 7;

// the state a state-setting rule gives the ghost at interior coordinates
// (i, j): 1 the inflow state, 2 the pre-shock state, 0 where the rule copies
// from the interior.  The array's time is t + toff dt (0 for W, 1/2 for W*).
__device__ __forceinline__ int ghost_state(const GridDev& g, int bc, int i, int j, const DevState* ds, double toff)
{
    if (bc < BC_INFLOW) return 0;
    if (bc == BC_INFLOW) return 1;
    const double x = g.ox + (i + 0.5) * g.dx;
    if (bc == BC_WALL_AFTER_X0) return (x < g.bs.x0) ? 1 : 0;
    const double y = g.oy + (j + 0.5) * g.dy, t = ds ? ds->t + toff * ds->dt : 0.0;
    return (x < g.bs.x0 + (y - g.oy) * g.bs.cot + g.bs.vx * t) ? 1 : 2;
}

// ------------------------------------------------------------------ ghosts
// source index of ghost position g (ghosted coordinate) along a line of n
// interior cells, and the velocity flips the rule implies
__device__ __forceinline__ int ghost_src(int bc, int n, int g, bool& flip_n, bool& flip_all)
{
    flip_n = flip_all = false;
    if (g >= NG && g < NG + n) return g;
    const bool low = g < NG;
    switch (bc) {
    case 0:  // periodic
        return NG + (((g - NG) % n) + n) % n;
    case 1:  // zero gradient
        return low ? NG : NG + n - 1;
    case 3:  // no-slip adiabatic wall
        flip_all = true;
        return low ? 2 * NG - 1 - g : 2 * (NG + n) - 1 - g;
    default:  // symmetry / reflect
        flip_n = true;
        return low ? 2 * NG - 1 - g : 2 * (NG + n) - 1 - g;
    }
}

// Where the value of cell (i, j) (interior coordinates, -3 .. n + 2) comes
// from: a prescribed state, or an interior cell with the momenta's signs.  A
// y ghost row takes the y rule to pick an interior row, then an x ghost
// column the x rule (the same values as filling x first, then y over the full
// ghosted width).
struct CellSrc {
    int i, j;     // the interior cell copied
    int state;    // 0 copy, 1 inflow, 2 pre-shock state
    bool n1, n2;  // momentum 1 / 2 negated
};
template <bool D2>
__device__ __forceinline__ CellSrc cell_source(const GridDev& g, int i, int j, const DevState* ds, double toff)
{
    CellSrc s{i, j, 0, false, false};
    bool fn, fa;
    if (D2 && (j < 0 || j >= g.ny)) {
        const int by = g.bc[j >= g.ny ? 3 : 2];
        s.state = ghost_state(g, by, i, j, ds, toff);
        if (s.state) return s;
        s.j = ghost_src(by, g.ny, j + NG, fn, fa) - NG;
        s.n1 = fa;
        s.n2 = fn || fa;
    }
    if (i < 0 || i >= g.nx) {
        const int bx = g.bc[i >= g.nx ? 1 : 0];
        s.state = ghost_state(g, bx, i, j, ds, toff);
        if (s.state) return s;
        s.i = ghost_src(bx, g.nx, i + NG, fn, fa) - NG;
        s.n1 ^= fn || fa;
        s.n2 ^= fa;
    }
    return s;
}
// component v of a prescribed state
__device__ __forceinline__ double state_value(const GridDev& g, int state, int v)
{
    const int k = (v == g.dim + 1) ? 3 : v;
    return state == 1 ? g.bs.in[k] : g.bs.pre[k];
}

// ------------------------------------------------------------------ commit
// After the last kernel of a step: advance t by dt, pick the next dt
// (CFL from the reduced sigma, clipped to t_end), detect completion.
// init: only pick dt from sigma (before the first step).
__device__ __forceinline__ void commit_step(DevState* ds, bool init)
{
    if (ds->done) return;
    if (!init) {
        ds->t += ds->dt;
        ds->steps += 1;
    }
    const double sig = __longlong_as_double((long long)atomicExch(&ds->sigma, 0ull));
    double dt = ds->fixed_dt ? ds->dt : ds->cfl / sig;
    if (ds->t + dt > ds->t_end) dt = ds->t_end - ds->t;
    ds->dt = dt;
    if (!(ds->t < ds->t_end) || (ds->max_steps > 0 && ds->steps >= ds->max_steps)) ds->done = 1u;
}

// ------------------------------------------------------------------ CFL rate
// sigma = max((|U| + a)/h, 4 nu / h^2), dt = cfl / sigma  (Sec. 5), in the
// kernel's arithmetic type (the float32 path takes its time step in float32;
// only the state and its accumulation are float64)
// U^2 + V^2 with both products rounded before the sum (no fused
// multiply-add): the same bits for (U, V) and (V, U), so a sweep that holds
// the state in its local frame and the grid-order reduction pick the same
// time step
template <typename T>
__device__ __forceinline__ T speed2(T U, T V)
{
    if constexpr (sizeof(T) == 4) return __fmul_rn(U, U) + __fmul_rn(V, V);
    else return __dmul_rn(U, U) + __dmul_rn(V, V);
}

// division and square root rounded to nearest whatever the unit's float
// flags: the sweeps' units take fast float32 division and square root, the
// reduction before a call's first step (k_sigma) does not, and both must
// form the same time step
template <typename T>
__device__ __forceinline__ T div_rn(T a, T b)
{
    if constexpr (sizeof(T) == 4) return __fdiv_rn(a, b);
    else return __ddiv_rn(a, b);
}
template <typename T>
__device__ __forceinline__ T sqrt_rn(T a)
{
    if constexpr (sizeof(T) == 4) return __fsqrt_rn(a);
    else return __dsqrt_rn(a);
}

template <typename T, typename WT = double>
__device__ __forceinline__ T cell_sigma(const WT* w, int dim, T gamma, T mu, T h, unsigned int& err)
{
    const T r = (T)w[0], ir = div_rn(T(1), r);
    const T U = (T)w[1] * ir, V = (dim == 2) ? (T)w[2] * ir : T(0);
    const T E = (T)(dim == 2 ? w[3] : w[2]);  // no dynamic index: keeps w in registers
    const T q = speed2(U, V);
    const T p = (gamma - T(1)) * (E - T(0.5) * r * q);
    if (!(r > T(0) && p > T(0) && isfinite(p))) err |= 1u;
    const T a = sqrt_rn(gamma * p * ir);
    const T ih = div_rn(T(1), h);
    T s = (sqrt_rn(q) + a) * ih;
    if (mu > T(0)) s = fmax(s, T(4) * mu * ir * ih * ih);
    return s;
}

// maximum of a warp's non-negative values, NaN only where every lane holds
// NaN (as fmax has it); float32 by one integer reduction on the bits, which
// order like the values
__device__ __forceinline__ float warp_max(float s)
{
    const unsigned k = __reduce_max_sync(0xffffffffu, s != s ? 0u : __float_as_uint(s) + 1u);
    return k == 0u ? __uint_as_float(0x7fffffffu) : __uint_as_float(k - 1u);
}
__device__ __forceinline__ double warp_max(double s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
    return s;
}

// Block reduction of the CFL rate (only when with_sigma), the error word and
// the fallback count; one atomic of each per block.  commit: the last block
// to get here commits the step (every block has read dt and done by then).
template <int NT, typename T>
__device__ __forceinline__ void block_commit(T s, bool with_sigma, unsigned int err, unsigned int nfb, DevState* ds,
                                             bool commit)
{
    __shared__ T red_s[NT / 32];
    __shared__ unsigned int red_e[NT / 32], red_f[NT / 32];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (with_sigma) {
        const T m = warp_max(s);
        if (l == 0) red_s[w] = m;
    }
    // errors and fallbacks are rare: one vote says whether there are any
    const bool any = __syncthreads_or((err | nfb) != 0u);
    if (any) {
        err = __reduce_or_sync(0xffffffffu, err);
        nfb = __reduce_add_sync(0xffffffffu, nfb);
        if (l == 0) { red_e[w] = err; red_f[w] = nfb; }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (with_sigma) s = red_s[0];
        for (int k = 1; k < NT / 32; ++k) {
            if (with_sigma) s = fmax(s, red_s[k]);
            if (any) {
                err |= red_e[k];
                nfb += red_f[k];
            }
        }
        const double sd = (double)s;
        if (with_sigma && (sd > 0.0 || sd != sd))
            atomicMax(&ds->sigma, (unsigned long long)__double_as_longlong(sd));
        if (err) atomicOr(&ds->err, err);
        if (nfb) atomicAdd(&ds->fallbacks, (unsigned long long)nfb);
        if (commit) {
            __threadfence();  // this block's rate before its ticket
            if (atomicAdd(&ds->ticket, 1u) + 1u == gridDim.x * gridDim.y) {
                __threadfence();
                ds->ticket = 0;
                commit_step(ds, false);
            }
        }
    }
}

// ------------------------------------------------------------------ stage arithmetic
// Stage combinations of the face flux F and its time derivative dF
// (Sec. 2.2): stage 1: g0 = F/2 + dt/8 dF (for W*), g1 = F + dt/6 dF (for the
// accumulator); stage 2: g0 = dt/3 dF.  Explicit fused multiply-adds, here
// and in the updates below, give every kernel the same rounding.
template <typename T>
__device__ __forceinline__ void stage_comb(int stage, T F, T dF, T dt, T& g0, T& g1)
{
    if (stage == 1) {
        g0 = fma(T(0.125) * dt, dF, T(0.5) * F);
        g1 = fma(dt * T(1.0 / 6.0), dF, F);
    } else {
        g0 = (dt * T(1.0 / 3.0)) * dF;
        g1 = T(0);
    }
}
// float64 path: W* = W - cx dG0, A = W - cx dG1; stage 2: W = A - cx dG0
__device__ __forceinline__ double upd64(double w, double cx, double dG) { return fma(-cx, dG, w); }
// float32 path: W* = W - cx dG0 and the increment cx dG1 in float32; stage 2:
// W = W - (increment + cx dG0), the sum in float32, the update in float64
__device__ __forceinline__ float wstar32(float w, float cx, float dG) { return fmaf(-cx, dG, w); }
__device__ __forceinline__ double wnew32(double w, float inc, float cx, float dG)
{
    return w - widen(fmaf(cx, dG, inc));
}

// ------------------------------------------------------------------ 1-D stage
// float64 path: W* and the accumulator A are float64 arrays.
// float32 path (as the 2-D one): W* is only the stage-2 reconstruction input,
// so it is formed and kept in float32, and the accumulator is kept as the
// float32 increment dt/dx d(F + dt/6 dF); the only float64 arithmetic is the
// final update W^{n+1} = W^n - (increment + dt/dx d(dt/3 dF*)).
template <typename T> __device__ __forceinline__ T load_as(double x) { return from_f64<T>(x); }
template <typename T> __device__ __forceinline__ T load_as(float x) { return x; }
struct Stage1DArgs {
    const double* src;   // float64 reconstruction input (W; float64 path stage 2: W*)
    const float* srcf;   // float32 path: stage 1 the float32 shadow of W (or nullptr: src,
                         // converted), stage 2 W* (float32)
    double* out0;        // float64 path stage 1: W*; stage 2: the new state
    double* out1;        // float64 path stage 1: accumulator A
    const double* acc;   // float64 path stage 2: accumulator A
    float* out0f;        // float32 path stage 1: W*; stage 2: the new state's float32
                         // shadow (or nullptr)
    float* out1f;        // float32 path stage 1: accumulator increment
    const float* accf;   // float32 path stage 2: accumulator increment
    const double* base;  // float32 path stage 2: W^n
    int stage;
    int with_sigma;      // stage 2: reduce the CFL rate of the new state
    int commit;          // the last block commits the step
    double idx;          // 1 / dx
};

// cells i0 - 3 .. i0 + TN + 2 of a block at an end of the grid, ghosts by the
// boundary rules (out of line: the other blocks keep their registers)
template <typename T, int TN, typename E>
__device__ __noinline__ void load_edge_1d(T* sq, const E* src, const GridDev& g, int i0, const DevState* ds, int stage)
{
    const long long pl = g.plane;
    for (int k = threadIdx.x; k < 3 * (TN + 6); k += blockDim.x) {
        const int v = k / (TN + 6), c = k % (TN + 6) - NG;
        T val = T(0);
        if (c < g.nx - i0 + NG) {  // beyond: padding
            const int i = i0 + c;
            const CellSrc cs = cell_source<false>(g, i, 0, ds, stage == 1 ? 0.0 : 0.5);
            val = cs.state ? (T)state_value(g, cs.state, v) : load_as<T>(src[v * pl + NG + cs.i]);
            if (v == 1 && cs.n1) val = -val;
        }
        sq[k] = val;
    }
}

// 4- or 8-byte copies from global to shared memory that the thread waits for
// only when it reads them
template <int B>
__device__ __forceinline__ void copy_async(void* dst, const void* src)
{
    static_assert(B == 4 || B == 8, "cp.async size");
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (B == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the last N committed groups of this thread are done
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T, bool NONEQ, bool PRFIX, int TN, int REC = 0>
__global__ void __launch_bounds__(TN + 2, sizeof(T) == 4 ? 8 : 4) k1d_stage(const __grid_constant__ GridDev g, Stage1DArgs a,
                                                    FluxParams<T> fp, TenoT<T> tn, DevState* ds)
{
    if (ds->done) return;
    // TN cells per block, TN + 2 threads: the TN + 2 reconstructed cells,
    // TN + 1 faces and TN updated cells each take one pass of the block
    constexpr int NT = TN + 2;
    const double dt = ds->dt;
    // dt and dt/dx in the arithmetic type, converted once per block (a
    // float64 -> float32 conversion runs on the slow float64 pipe)
    __shared__ T s_scal[6];  // dt, dt/dx, 1/dx, gamma, mu, dx
    if (threadIdx.x == 0) {
        s_scal[0] = (T)dt;
        s_scal[1] = (T)(dt * a.idx);
        s_scal[2] = (T)a.idx;
        s_scal[3] = (T)g.gamma;
        s_scal[4] = (T)g.mu;
        s_scal[5] = (T)g.dx;
    }
    __shared__ T sq[3][TN + 6];
    // [var][value, slope][face], and one entry beyond each end that no face
    // reads, so that every cell stores both its faces' values
    __shared__ T sL[3][2][TN + 2], sR_[3][2][TN + 2];
    T(*sR)[2][TN + 2] = reinterpret_cast<T(*)[2][TN + 2]>(&sR_[0][0][1]);
    __shared__ T sG[2][3][TN + 1];                     // face fluxes for the update
    const int i0 = blockIdx.x * TN;
    const int tid = threadIdx.x;
    const int slot[3] = {0, 1, 3};

    // a 1-D plane is one ghosted row; three of them pass 2^31 elements from
    // 7.2e8 cells on, so a variable's offset is a 64-bit one (every comparison
    // with nx is of differences, which stay in range up to the largest grid)
    const long long pl = g.plane;
    const int uo = i0 + tid + NG;
    const bool own = tid < TN && tid < g.nx - i0;
    // one loop per source type: a per-element choice between the float32
    // and the converted float64 source was compiled as both, and every
    // element then paid a float64 -> float32 conversion on the slow float64
    // pipe whichever source it took
    const bool edge = i0 < NG || TN + NG > g.nx - i0;
    auto load = [&](auto src) {
        if (edge) {
            load_edge_1d<T, TN>(&sq[0][0], src, g, i0, ds, a.stage);
            return;
        }
        static_assert(TN + 6 - NT == 4, "four cells beyond one per thread");
        if constexpr (std::is_same<decltype(src), const T*>::value) {
#pragma unroll
            for (int v = 0; v < 3; ++v) copy_async<sizeof(T)>(&sq[v][tid], src + (v * pl + i0 + tid));
            if (tid < 12) copy_async<sizeof(T)>(&sq[tid >> 2][NT + (tid & 3)], src + ((tid >> 2) * pl + i0 + NT + (tid & 3)));
            return;
        }
#pragma unroll
        for (int v = 0; v < 3; ++v) sq[v][tid] = load_as<T>(src[v * pl + i0 + tid]);
        if (tid < 12) sq[tid >> 2][NT + (tid & 3)] = load_as<T>(src[(tid >> 2) * pl + i0 + NT + (tid & 3)]);
    };
    if constexpr (sizeof(T) == 4) {
        if (a.srcf) load(a.srcf);
        else load(a.src);
    } else {
        load(a.src);
    }
    copy_commit();
    // the update's other inputs, on their way while the stage computes: read in
    // the update they cost its warps a memory round trip each (four steps of a
    // 2^22-cell float32 tube 1541 -> 1465 us against reads at the update's or the
    // stage's start into registers, which also took 64 registers instead of 56)
    __shared__ double s_base[3][TN];
    __shared__ float s_acc[3][sizeof(T) == 4 ? TN : 1];
    if (own && (a.stage == 2 || sizeof(T) == 8)) {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            if constexpr (sizeof(T) == 4) {
                copy_async<8>(&s_base[v][tid], a.base + (v * pl + uo));
                copy_async<4>(&s_acc[v][tid], a.accf + (v * pl + uo));
            } else {
                copy_async<8>(&s_base[v][tid], (a.stage == 1 ? a.src : a.acc) + (v * pl + uo));
            }
        }
    }
    copy_commit();
    copy_wait<1>();  // the tile
    __syncthreads();
    fp.dt = s_scal[0];
    const T idx_ = s_scal[2];
    if constexpr (REC == REC_TENO_CHAR) {
        // phase 1 in characteristic variables: per face f (between interior
        // i0 + f - 1 and i0 + f), the six cells around it projected with the
        // face's basis, both sides reconstructed
        for (int f = tid; f <= TN; f += NT) {
            T w[6][4], vl[4], dl[4], vr[4], dr[4];
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                w[c][0] = sq[0][f + c];
                w[c][1] = sq[1][f + c];
                w[c][2] = T(0);
                w[c][3] = sq[2][f + c];
            }
            char_face<T, 1>(w, tn, fp.gm1, vl, dl, vr, dr);
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                sL[v][0][f] = vl[slot[v]];
                sL[v][1][f] = dl[slot[v]] * idx_;
                sR[v][0][f] = vr[slot[v]];
                sR[v][1][f] = dr[slot[v]] * idx_;
            }
        }
    } else {
        // phase 1: reconstruction per cell c (interior i0 - 1 + c), both faces
        for (int c = tid; c < TN + 2; c += NT) {
            T q[3][5], vp[3], dp[3], vm[3], dm[3];
#pragma unroll
            for (int v = 0; v < 3; ++v)
#pragma unroll
                for (int s = 0; s < 5; ++s) q[v][s] = sq[v][c + s];
            recon_cell3<REC>(q, tn, vp, dp, vm, dm);
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                sL[v][0][c] = vp[v];
                sL[v][1][c] = dp[v] * idx_;
                sR_[v][0][c] = vm[v];
                sR_[v][1][c] = dm[v] * idx_;
            }
        }
    }
    __syncthreads();
    // phase 2: flux at face f (between interior i0+f-1 and i0+f)
    unsigned int nfb = 0, err = 0;
    for (int f = tid; f <= TN; f += NT) {
        if (f > g.nx - i0) continue;  // padding past the last face
        Side<T> L, R;
#pragma unroll
        for (int k = 0; k < 4; ++k) { L.W[k] = L.Wn[k] = L.Wt[k] = R.W[k] = R.Wn[k] = R.Wt[k] = T(0); }
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            L.W[slot[v]] = sL[v][0][f];
            L.Wn[slot[v]] = sL[v][1][f];
            R.W[slot[v]] = sR[v][0][f];
            R.Wn[slot[v]] = sR[v][1][f];
        }
        auto state = [&](int side, Side<T>& S, Prim<T>& p) {
            if (prim_state<T, 1>(S.W, fp.gm1, p)) return;
#pragma unroll
            for (int v = 0; v < 3; ++v) { S.W[slot[v]] = sq[v][f + 2 + side]; S.Wn[slot[v]] = T(0); }
            ++nfb;
            if (!prim_state<T, 1>(S.W, fp.gm1, p)) err |= 2u;
        };
        T F[4], dF[4];
        if constexpr (rec_conventional(REC)) {
            // conventional path: equilibrium slope from the cell averages
            // i-1 .. i+2 around the face by the linear Eq. (3.12)
            T w0n[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
            for (int v = 0; v < 3; ++v)
                w0n[slot[v]] = (T(1.25) * (sq[v][f + 3] - sq[v][f + 2]) - T(1.0 / 12.0) * (sq[v][f + 4] - sq[v][f + 1]))
                             * idx_;
            point_flux<T, 1, NONEQ, PRFIX>(L, R, T(1), fp, F, dF, a.stage == 1, state, w0n);
        } else {
            point_flux<T, 1, NONEQ, PRFIX>(L, R, T(1), fp, F, dF, a.stage == 1, state);
        }
        const T tdt = s_scal[0];
#pragma unroll
        for (int v = 0; v < 3; ++v) stage_comb<T>(a.stage, F[slot[v]], dF[slot[v]], tdt, sG[0][v][f], sG[1][v][f]);
    }
    __syncthreads();
    // phase 3: update
    T sig = T(0);
    const double cx = dt * a.idx;
    const T cxt = s_scal[1];
    copy_wait<0>();
    if (own) {
        const int c = tid, o = uo;
        T w[4];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const T d0 = sG[0][v][c + 1] - sG[0][v][c];
            if constexpr (sizeof(T) == 4) {
                if (a.stage == 1) {
                    a.out0f[v * pl + o] = wstar32(sq[v][c + 3], cxt, d0);
                    a.out1f[v * pl + o] = cxt * (sG[1][v][c + 1] - sG[1][v][c]);
                } else {
                    const double r = wnew32(s_base[v][tid], s_acc[v][tid], cxt, d0);
                    a.out0[v * pl + o] = r;
                    w[v] = narrow(r);
                    if (a.out0f) a.out0f[v * pl + o] = w[v];
                }
            } else {
                const double r = upd64(s_base[v][tid], cx, (double)d0);
                a.out0[v * pl + o] = r;
                if (a.stage == 1) a.out1[v * pl + o] = upd64(s_base[v][tid], cx, (double)(sG[1][v][c + 1] - sG[1][v][c]));
                w[v] = (T)r;
            }
        }
        if (a.with_sigma) sig = cell_sigma<T, T>(w, 1, s_scal[3], s_scal[4], s_scal[5], err);
    }
    if (NT % 32 == 0) block_commit<NT, T>(sig, a.with_sigma != 0, err, nfb, ds, a.commit != 0);
}

// ------------------------------------------------------------------ 1-D stage, short grids
// The same stage for grids too short to fill the chip, where a step lasts as
// long as one warp's chain of operations (a dependent float64 operation takes
// over 100 cycles, a float32 stage ~1500 instructions): three warps on 30
// cells split the chain, so that no lane runs more than a third of it.
// Phase 1: warp v reconstructs variable v.  Phase 2: warps 0 and 1 the left
// and the right side's moments; then warp 0 the equilibrium fluxes while warp
// 1 forms the time coefficients; then warp v combines component v.  The
// heat-flux correction, the averaged merge and characteristic variables take
// k1d_stage.
constexpr int WIDE_TN = 30;

template <typename T, bool NONEQ, int REC>
__global__ void __launch_bounds__(96) k1d_stage_wide(const __grid_constant__ GridDev g, Stage1DArgs a,
                                                     FluxParams<T> fp, TenoT<T> tn, DevState* ds)
{
    if (ds->done) return;
    constexpr int TN = WIDE_TN, NS = 16;
    __shared__ T sq[3][TN + 6];
    __shared__ T sL[3][2][32], sR[3][2][32];  // [var][value, slope][face]
    __shared__ T sS[2][NS][32];               // a side's W0, W0n, S3, S4, S5 (3 each), pressure
    __shared__ T sF[3][3][32], sC[12][32];    // F0, F1, F2; time coefficients
    __shared__ T sG[2][3][32];
    __shared__ double s_cx;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * TN;
    const int pl = (int)g.plane;  // a short grid: three rows fit in 32 bits
    constexpr int slot[3] = {0, 1, 3};
    const double dt = ds->dt;
    fp.dt = (T)dt;
    const T ih = (T)a.idx;
    if (threadIdx.x == 0) s_cx = dt * a.idx;
    auto load = [&](auto src) {  // warp v loads variable v
        for (int c = lane; c < TN + 6; c += 32) {
            const int i = i0 - NG + c;
            T val = T(0);
            if (i >= 0 && i < g.nx) {
                val = load_as<T>(src[warp * pl + NG + i]);
            } else if (i < g.nx + NG) {  // a ghost; beyond: padding
                const CellSrc cs = cell_source<false>(g, i, 0, ds, a.stage == 1 ? 0.0 : 0.5);
                val = cs.state ? (T)state_value(g, cs.state, warp) : load_as<T>(src[warp * pl + NG + cs.i]);
                if (warp == 1 && cs.n1) val = -val;
            }
            sq[warp][c] = val;
        }
    };
    if constexpr (sizeof(T) == 4) {
        if (a.srcf) load(a.srcf);
        else load(a.src);
    } else {
        load(a.src);
    }
    // the update's other inputs, ahead of their use (warp 0: cell i0 + lane)
    const int i = i0 + lane, o = i + NG;
    const bool own = warp == 0 && lane < TN && i < g.nx;
    double base[3] = {0.0, 0.0, 0.0};
    T acc[3] = {T(0), T(0), T(0)};
    if (own) {
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            if constexpr (sizeof(T) == 4) {
                if (a.stage == 2) { base[v] = a.base[v * pl + o]; acc[v] = a.accf[v * pl + o]; }
            } else {
                base[v] = a.stage == 1 ? a.src[v * pl + o] : a.acc[v * pl + o];
            }
        }
    }
    __syncwarp();
    {
        T q[5], vp, dp, vm, dm;
#pragma unroll
        for (int s = 0; s < 5; ++s) q[s] = sq[warp][lane + s];
        if constexpr (sizeof(T) == 4 && REC == 0) {
            // as recon_cell3: (rho, rho u) in the packed form, E in the scalar one
            if (warp < 2) {
                f2 qq[5], x, y, z, w;
#pragma unroll
                for (int s = 0; s < 5; ++s) qq[s] = f2(q[s]);
                packed_faces<0, false>(qq, tn, x, y, z, w);
                vp = x.x(), dp = y.x(), vm = z.x(), dm = w.x();
            } else {
                TenoSel<T> S;
                teno_select<false>(q, tn, S);
                teno_faces(q, S, vp, dp, vm, dm);
            }
        } else {
            TenoSel<T> S;
            rec_select<REC, false>(q, tn, S);
            rec_faces<REC>(q, S, vp, dp, vm, dm);
        }
        sL[warp][0][lane] = vp;
        sL[warp][1][lane] = dp * ih;
        if (lane >= 1) {
            sR[warp][0][lane - 1] = vm;
            sR[warp][1][lane - 1] = dm * ih;
        }
    }
    __syncthreads();
    // phase 2: face lane between interior cells i0 + lane - 1 and i0 + lane
    const bool face = lane <= TN && i0 + lane <= g.nx;
    unsigned int nfb = 0, err = 0;
    if (warp < 2 && face) {
        const int f = lane;
        Side<T> S;
#pragma unroll
        for (int k = 0; k < 4; ++k) S.W[k] = S.Wn[k] = S.Wt[k] = T(0);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            S.W[slot[v]] = warp ? sR[v][0][f] : sL[v][0][f];
            S.Wn[slot[v]] = warp ? sR[v][1][f] : sL[v][1][f];
        }
        Prim<T> p;
        if (!prim_state<T, 1>(S.W, fp.gm1, p)) {
#pragma unroll
            for (int v = 0; v < 3; ++v) { S.W[slot[v]] = sq[v][f + 2 + warp]; S.Wn[slot[v]] = T(0); }
            ++nfb;
            if (!prim_state<T, 1>(S.W, fp.gm1, p)) err |= 2u;
        }
        T W0[4], W0n[4], W0t[4], S3[4], S4[4], S5[4];
        side_terms<false, T, 1, NONEQ, false>(S, p, warp ? T(-1) : T(1), fp, W0, W0n, W0t, S3, S4, S5, nullptr, nullptr);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            sS[warp][v][f] = W0[slot[v]];
            sS[warp][3 + v][f] = W0n[slot[v]];
            if constexpr (NONEQ) {
                sS[warp][6 + v][f] = S3[slot[v]];
                sS[warp][9 + v][f] = S4[slot[v]];
                sS[warp][12 + v][f] = S5[slot[v]];
            }
        }
        sS[warp][15][f] = p.p;
    }
    __syncthreads();
    if (warp < 2 && face) {
        const int f = lane;
        T W0[4] = {sS[0][0][f] + sS[1][0][f], sS[0][1][f] + sS[1][1][f], T(0), sS[0][2][f] + sS[1][2][f]};
        if (warp == 0) {
            T W0n[4] = {T(0), T(0), T(0), T(0)}, W0t[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                if constexpr (rec_conventional(REC))  // Eq. (3.12), as k1d_stage
                    W0n[slot[v]] = (T(1.25) * (sq[v][f + 3] - sq[v][f + 2])
                                    - T(1.0 / 12.0) * (sq[v][f + 4] - sq[v][f + 1])) * ih;
                else W0n[slot[v]] = sS[0][3 + v][f] + sS[1][3 + v][f];
            }
            Equilibrium<T> E;
            equilibrium<T, 1, NONEQ>(W0, W0n, W0t, fp, E);
#pragma unroll
            for (int v = 0; v < 3; ++v) {
                sF[0][v][f] = E.F0[slot[v]];
                sF[1][v][f] = E.F1[slot[v]];
                sF[2][v][f] = E.F2[slot[v]];
            }
        } else if (fp.tau_mode != 0) {
            T p0 = T(1);
            if (fp.tau_mode == 2) p0 = fp.gm1 * (W0[3] - T(0.5) * W0[1] * W0[1] / W0[0]);
            T cF[6], cD[6];
            const T is = tau_over_dt(fp, sS[0][15][f], sS[1][15][f], p0, T(1) / fp.dt);
            time_coeffs<T>(T(1) / is, is, cF, cD);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                sC[k][f] = cF[k];
                sC[6 + k][f] = cD[k];
            }
        }
    }
    __syncthreads();
    if (face) {
        const int f = lane, v = warp;
        T F = T(0), dF;
        if (fp.tau_mode == 0) {
            F = sF[0][v][f];
            dF = sF[2][v][f];
        } else {
            const T x[6] = {sF[0][v][f], sF[1][v][f], sF[2][v][f], sS[0][6 + v][f] + sS[1][6 + v][f],
                            sS[0][9 + v][f] + sS[1][9 + v][f], sS[0][12 + v][f] + sS[1][12 + v][f]};
            const T tdt = fp.dt, i4 = T(4) / tdt;
            // q_k = c_k s1 for p_k = 1 (k = 0, 3), c_k s2 for p_k = 2
            auto combine = [&](int c, T s1, T s2) {
                T r = (sC[c + 5][f] * s2) * x[5];
                r = fma(sC[c + 4][f] * s2, x[4], r);
                r = fma(sC[c + 3][f] * s1, x[3], r);
                r = fma(sC[c + 2][f] * s2, x[2], r);
                r = fma(sC[c + 1][f] * s2, x[1], r);
                return fma(sC[c][f] * s1, x[0], r);
            };
            if (a.stage == 1) F = combine(0, T(1), tdt);
            dF = combine(6, i4, T(4));
        }
        stage_comb<T>(a.stage, F, dF, fp.dt, sG[0][v][f], sG[1][v][f]);
    }
    __syncthreads();
    T sig = T(0);
    if (own) {
        const double cx = s_cx;
        const T cxt = (T)cx;
        const int c = lane;
        T w[4];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const T d0 = sG[0][v][c + 1] - sG[0][v][c];
            if constexpr (sizeof(T) == 4) {
                if (a.stage == 1) {
                    a.out0f[v * pl + o] = wstar32(sq[v][c + 3], cxt, d0);
                    a.out1f[v * pl + o] = cxt * (sG[1][v][c + 1] - sG[1][v][c]);
                } else {
                    const double r = wnew32(base[v], acc[v], cxt, d0);
                    a.out0[v * pl + o] = r;
                    w[v] = narrow(r);
                    if (a.out0f) a.out0f[v * pl + o] = w[v];
                }
            } else {
                const double r = upd64(base[v], cx, (double)d0);
                a.out0[v * pl + o] = r;
                if (a.stage == 1) a.out1[v * pl + o] = upd64(base[v], cx, (double)(sG[1][v][c + 1] - sG[1][v][c]));
                w[v] = (T)r;
            }
        }
        if (a.with_sigma) sig = cell_sigma<T, T>(w, 1, (T)g.gamma, (T)g.mu, (T)g.dx, err);
    }
    block_commit<96, T>(sig, a.with_sigma != 0, err, nfb, ds, a.commit != 0);
}

// ------------------------------------------------------------------ 2-D sweep
// One stage = x sweep (pass 0) then y sweep (pass 1).  The x sweep stores its
// flux-divergence increments dt/dx dG in the kernel's arithmetic type (inc0,
// inc1); the y sweep adds its own.
// float64 path (one float64 update per value):
//   stage 1: W* = W - (inc0 + dt/dy dG1),  A = W - (inc1 + dt/dy dG2)
//   stage 2: W  = A - (inc0 + dt/dy dG)
// float32 path: W* is only the stage-2 reconstruction input, so it is formed
// in float32 from the float32 shadow of W, and the accumulator stays an
// increment; the only float64 arithmetic is the final update of W:
//   stage 1: W*f = Wf - (inc0 + dt/dy dG1),  inc1 <- inc1 + dt/dy dG2
//   stage 2: W   = W - (inc1 + inc0 + dt/dy dG)   (and its shadow Wf)
struct SweepArgs {
    const double* src;   // reconstruction input (W or W*)
    const float* srcf;   // float32 path: float32 shadow of src
    const float* basef;  // float32 path, y sweep of stage 1: float32 shadow of W
    const double* base;  // y sweep: W (stage 1) or A (stage 2)
    double* out0;        // y sweep, stage 1: W*; stage 2: W
    float* out0f;        // float32 path, y sweep: float32 shadow of out0
    double* out1;        // y sweep, stage 1: A
    void* inc0;          // increments, arithmetic type, same ghosted layout
    void* inc1;          // (stage 1 only)
    int stage, pass;     // pass 0: x sweep (first), 1: y sweep (second)
    int dirn;            // 0: faces normal to x, 1: faces normal to y
    int nn, nt;          // cells along the normal / tangential direction
    long long sn, st;    // element strides along normal / tangential
    double ihn, iht;     // inverse cell sizes along normal / tangential
    double hmin;         // min(dx, dy) for the CFL rate
    int with_sigma;
    int commit;          // the last block commits the step
    int sms;             // multiprocessors of the device (tile choice)
    int tall;            // more rows of tiles than a grid's y extent takes: rows along x (sweep_tall)
};

// global variable index of local variable v (swap: faces normal to y)
__device__ __forceinline__ int gvar(int v, bool swap) { return (swap && (v == 1 || v == 2)) ? 3 - v : v; }

// Tiles that can lie with their rows along the grid's x extent: the float64
// ones and the lowest float32 ones, which the tallest grids take.  The choice
// costs the taller float32 tiles, which spill, 1.5 % (2048 x 1024 viscous
// 3209 -> 3257 us for two steps); 64^2 float32 254 us either way.
template <typename T>
__host__ __device__ constexpr bool sweep_tall(int rows) { return sizeof(T) == 8 || rows == 4; }

template <typename T> struct alignas(2 * sizeof(T)) Pair2 {
    T v, s;
};

template <typename T, int TN, int TT, bool CONV, bool STAGED> struct SweepSmem {
    T w[4][TT + 4][TN + 6];           // cells: tangential rows t0-2.., normal n0-3..
    Pair2<T> rec[2][4][TT + 4][TN + 1];  // [side][var][row][face]: value and normal slope
    T flux[8 * (TN + 1) * (TT + 1)];  // face fluxes for the update (layout: sfi)
    // y sweep: the update's inputs, copied while the sweep computes
    double base[STAGED ? 4 : 1][STAGED ? TN * TT : 1];  // W or A (float32 stage 1: its float32 shadow, in the first half)
    T inc[2][STAGED ? 4 : 1][STAGED ? TN * TT : 1];     // the x sweep's increments
    // conventional path: line-averaged equilibrium state and its normal
    // slope per face and row (Step 2)
    T w0[CONV ? 2 : 1][4][CONV ? TT + 4 : 1][CONV ? TN + 1 : 1];
};

// MB blocks of a kernel with this struct fit an SM's 228 KB (1 KB of a block is
// the system's, half a KB its static arrays)
template <typename Smem>
__host__ __device__ constexpr bool sweep_resident(int MB) { return MB * (sizeof(Smem) + 1536) <= 228 * 1024; }

// The update's inputs go through shared memory where the tile keeps the MB
// resident blocks its register budget is for: 16 rows of the conventional path
// do not (122 KB a block, 91 without; one step of a float32 plane with one
// resident block and with two: 768^2 TENO5 546 -> 459 us, WENO5-Z 467 -> 397,
// 1024^2 965 -> 816 and 818 -> 697).
template <typename T, int TN, int TT, int MB, bool CONV>
__host__ __device__ constexpr bool sweep_staged() { return sweep_resident<SweepSmem<T, TN, TT, CONV, true>>(MB); }
template <typename T, int TN, int TT, int MB, bool CONV>
using SweepShared = SweepSmem<T, TN, TT, CONV, sweep_staged<T, TN, TT, MB, CONV>()>;

// the cells of a tile that reaches past the boundary, ghosts by the boundary
// rules (out of line: the other tiles keep their registers)
template <typename T, int TN, int TT>
__device__ __noinline__ void load_edge_2d(T* w, const GridDev& g, const SweepArgs& a, int n0, int t0,
                                          const DevState* ds)
{
    constexpr int CN = TN + 6, CT = TT + 4;
    const bool swap = a.dirn != 0;
    for (int k = threadIdx.x; k < 4 * CN * CT; k += blockDim.x) {
        const int v = k / (CN * CT), e = k % (CN * CT);
        const int ct = swap ? e % CT : e / CN, cn = swap ? e / CT : e % CN;
        const int in = n0 - NG + cn, it = t0 - 2 + ct;
        T val = T(0);
        if (in < a.nn + NG && it < a.nt + 2) {  // beyond: padding
            const int gv = gvar(v, swap);
            const CellSrc cs = cell_source<true>(g, swap ? it : in, swap ? in : it, ds, a.stage == 1 ? 0.0 : 0.5);
            const long long off = (long long)gv * g.plane + (long long)(cs.j + NG) * g.pitch + cs.i + NG;
            if (cs.state) val = (T)state_value(g, cs.state, gv);
            else if constexpr (sizeof(T) == 4) val = a.srcf[off];
            else val = a.src[off];
            if ((gv == 1 && cs.n1) || (gv == 2 && cs.n2)) val = -val;
        }
        w[(v * CT + ct) * CN + cn] = val;
    }
}

template <typename T, bool NONEQ, bool PRFIX, int TN, int TT, int NT, int MB, int REC = 0>
__global__ void __launch_bounds__(NT, MB)
k2d_sweep(const __grid_constant__ GridDev g, const __grid_constant__ SweepArgs a, FluxParams<T> fp, TenoT<T> tnn, TenoT<T> tnt, DevState* ds)
{
    if (ds->done) return;
    constexpr int NF = TN + 1;           // faces per tile row
    constexpr int NW = NT / 32;
    constexpr bool CONV = rec_conventional(REC);
    constexpr int RB = rec_base(REC);  // the tangential (per-quantity) reconstruction
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool STAGED = sweep_staged<T, TN, TT, MB, CONV>();
    using Shared = SweepShared<T, TN, TT, MB, CONV>;
    static_assert(sweep_resident<Shared>(MB), "the MB blocks of the launch bounds fit an SM's shared memory");
    Shared& sm = *reinterpret_cast<Shared*>(smem_raw);
    // face fluxes for the update: [k][row][face] for x faces; [k][face][row]
    // (rows padded) for y faces, so that phase 3 runs along the unit-stride x
    // direction in both sweeps
    T* sF = sm.flux;
    const bool fy = a.dirn != 0;
    auto sfi = [&](int k, int r, int f) { return fy ? (k * NF + f) * (TT + 1) + r : (k * TT + r) * NF + f; };

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the stage's scalars in the arithmetic type, converted once per block
    // (a float64 -> float32 conversion runs on the slow float64 pipe):
    // dt, dt/h_n, 1/h_n, 1/h_t, gamma, mu, min(h_n, h_t); visible after the
    // load phase's barrier
    __shared__ T s_scal[7];
    if (tid == 0) {
        const double dt = ds->dt;
        s_scal[0] = (T)dt;
        s_scal[1] = (T)(dt * a.ihn);
        s_scal[2] = (T)a.ihn;
        s_scal[3] = (T)a.iht;
        s_scal[4] = (T)g.gamma;
        s_scal[5] = (T)g.mu;
        s_scal[6] = (T)a.hmin;
    }
    const bool tall = sweep_tall<T>(TT) && a.tall;
    const int n0 = (tall ? blockIdx.y : blockIdx.x) * TN, t0 = (tall ? blockIdx.x : blockIdx.y) * TT;
    static_assert(TN == 31, "lanes of a warp along the tile's faces");
    // local frame: normal momentum first; y faces swap the two momentum components
    const bool swap = a.dirn != 0;
    // offsets within one variable plane fit in 32 bits; each variable's plane
    // is reached through its own base pointer
    const int org = NG * g.pitch + NG;  // interior (0,0)
    const int sn = (int)a.sn, st = (int)a.st;
    const long long pv1 = (long long)gvar(1, swap) * g.plane, pv2 = (long long)gvar(2, swap) * g.plane;
    const long long pv3 = 3 * g.plane;

    // load cells (normal n0-3 .. n0+TN+2, tangential t0-2 .. t0+TT+1); the
    // thread index runs fastest along the unit-stride direction; tiles that
    // reach past the boundary take their ghosts by the boundary rules
    {
        constexpr int CN = TN + 6, CT = TT + 4;
        const bool edge = n0 < NG || n0 + TN + NG > a.nn || t0 < 2 || t0 + TT + 2 > a.nt;
        const T* base;
        if constexpr (sizeof(T) == 4) base = a.srcf + (org + (n0 - NG) * sn + (t0 - 2) * st);
        else base = a.src + (org + (n0 - NG) * sn + (t0 - 2) * st);
        auto cell = [&](int v, int cn, int ct) {
            const long long pv = v == 0 ? 0 : (v == 1 ? pv1 : (v == 2 ? pv2 : pv3));
            copy_async<sizeof(T)>(&sm.w[v][ct][cn], (base + pv) + (cn * sn + ct * st));
        };
        if (edge) load_edge_2d<T, TN, TT>(&sm.w[0][0][0], g, a, n0, t0, ds);
        else for (int k = tid; k < 4 * CN * CT; k += NT) {
            const int v = k / (CN * CT), e = k % (CN * CT);
            if (!fy) cell(v, e % CN, e / CN);
            else cell(v, e / CT, e % CT);
        }
    }
    copy_commit();
    // y sweep: start copying the update's inputs (read in the update, they
    // cost its warps a memory round trip: four steps of a 64^2 float32 plane
    // 292 -> 281 us, two of a 1024^2 plane the same)
    const bool base_f = sizeof(T) == 4 && a.stage == 1;
    if (STAGED && a.pass == 1) {
        for (int k = tid; k < TN * TT; k += NT) {
            const int r = fy ? k % TT : k / TN, c = fy ? k / TT : k % TN;
            const int in = n0 + c, it = t0 + r;
            if (in < a.nn && it < a.nt) {
                const int o = org + in * sn + it * st;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const long long go = (v == 0 ? 0 : (v == 1 ? pv1 : (v == 2 ? pv2 : pv3))) + o;
                    if (base_f) copy_async<4>(reinterpret_cast<float*>(sm.base[v]) + k, a.basef + go);
                    else copy_async<8>(&sm.base[v][k], a.base + go);
                    copy_async<sizeof(T)>(&sm.inc[0][v][k], static_cast<const T*>(a.inc0) + go);
                    if (a.stage == 1 || sizeof(T) == 4)
                        copy_async<sizeof(T)>(&sm.inc[1][v][k], static_cast<const T*>(a.inc1) + go);
                }
            }
        }
    }
    copy_commit();
    copy_wait<1>();  // the tile
    __syncthreads();
    fp.dt = s_scal[0];

    // The last tiles of a line or column do only their own work.  float64,
    // whose blocks' time is their work on the slow pipe, counts through the
    // tile's nf faces and nr rows alone (4 steps and their reverse on 96^2,
    // four tiles of 31 where the last holds 3 cells: 5.18 -> 4.60 ms).  float32
    // skips the warps that lie outside (two steps of 2048 x 1024 viscous cells
    // 3213 -> 3182 us); counting costs it registers (1024^2 1316 -> 1344 us).
    constexpr bool COUNT = sizeof(T) == 8;
    const int nf = COUNT ? min(NF, a.nn - n0 + 1) : NF, nr = COUNT ? min(TT, a.nt - t0) : TT;
    const bool whole = !COUNT || nf == NF;

    // phase 1: normal TENO-D per (cell, row, var): cell c <-> normal n0-1+c
    if constexpr (REC == REC_TENO_CHAR) {
        // characteristic variables: per (face, row), the six cells around
        // face f (between normal n0-1+f and n0+f) projected with the face's
        // basis, both sides reconstructed
        const T ih = s_scal[2];
        constexpr int NR = TT + 4;
        for (int k = tid; k < NF * NR; k += NT) {
            const int r = k / NF, f = k % NF;
            T w[6][4], vl[4], dl[4], vr[4], dr[4];
#pragma unroll
            for (int c = 0; c < 6; ++c)
#pragma unroll
                for (int v = 0; v < 4; ++v) w[c][v] = sm.w[v][r][f + c];
            char_face<T, 2>(w, tnn, fp.gm1, vl, dl, vr, dr);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                sm.rec[0][v][r][f] = {vl[v], dl[v] * ih};
                sm.rec[1][v][r][f] = {vr[v], dr[v] * ih};
            }
        }
    } else if constexpr (sizeof(T) == 4 && REC <= 1) {
        // float32 TENO-D / WENO5-AO: variables (0, 1) and (2, 3) as packed pairs
        const float ih = s_scal[2];
        // a warp takes one (row, pair): cells 0..31 along the lanes; the 33rd
        // cells of all rows come last, one per lane
        constexpr int NL = 2 * (TT + 4);
        for (int k = warp; k < NL + (NL + 31) / 32; k += NW) {
            const bool line = k < NL;
            const int e = line ? k : (k - NL) * 32 + lane, c = line ? lane : 32;
            if (e >= NL) continue;
            const int vv = 2 * (e & 1), r = e >> 1;
            if (t0 - 2 + r > a.nt + 1) continue;  // no Gauss point reads this row
            f2 q[5];
#pragma unroll
            for (int s = 0; s < 5; ++s) q[s] = f2(sm.w[vv][r][c + s], sm.w[vv + 1][r][c + s]);
            f2 vp, dp, vm, dm;
            packed_faces<REC>(q, tnn, vp, dp, vm, dm);
            const f2 dpi = dp * f2(ih), dmi = dm * f2(ih);
            if (c <= TN) {
                sm.rec[0][vv][r][c] = {vp.x(), dpi.x()};
                sm.rec[0][vv + 1][r][c] = {vp.y(), dpi.y()};
            }
            if (c >= 1) {
                sm.rec[1][vv][r][c - 1] = {vm.x(), dmi.x()};
                sm.rec[1][vv + 1][r][c - 1] = {vm.y(), dmi.y()};
            }
        }
    } else {
        const T ih = s_scal[2];
        // (row, variable) lines as above; narrow tiles count through their cells
        const int NL = 4 * (nr + 4), NK = whole ? 32 * (NL + (NL + 31) / 32) : NL * (nf + 1);
        for (int k = tid; k < NK; k += NT) {
            const int w = k >> 5;
            const bool line = w < NL;
            int e = line ? w : (w - NL) * 32 + lane, c = line ? lane : 32;
            if (!whole) {
                e = k / (nf + 1);
                c = k - e * (nf + 1);
            }
            if (e >= NL) continue;
            const int v = e & 3, r = e >> 2;
            if (t0 - 2 + r > a.nt + 1) continue;
            T q[5];
#pragma unroll
            for (int s = 0; s < 5; ++s) q[s] = sm.w[v][r][c + s];
            TenoSel<T> S;
            rec_select<REC>(q, tnn, S);
            T vp, dp, vm, dm;
            rec_faces<REC>(q, S, vp, dp, vm, dm);
            if (c <= TN) sm.rec[0][v][r][c] = {vp, dp * ih};
            if (c >= 1) sm.rec[1][v][r][c - 1] = {vm, dm * ih};
        }
    }
    __syncthreads();

    unsigned int nfb = 0, err = 0;
    if constexpr (CONV) {
        // phase 1b (conventional path, Step 2): per face and row, the
        // line-averaged equilibrium state by the kinetic merge of the face
        // values (a non-physical side takes its adjacent cell average), and
        // its normal slope by Eq. (3.12) on the row's cell averages
        const T ih = s_scal[2];
        for (int k = tid; k < NF * (TT + 4); k += NT) {
            const int r = k / NF, f = k % NF;
            // faces n0+f <= nn on rows t0-2+r <= nt+1 (ghosted extent) exist;
            // the rest of the tile is padding that no Gauss point reads
            if (n0 + f > a.nn || t0 - 2 + r > a.nt + 1) continue;
            T wl[4], wr[4], w0[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) { wl[v] = sm.rec[0][v][r][f].v; wr[v] = sm.rec[1][v][r][f].v; }
            if (!physical<T, 2>(wl, fp.gm1)) {
#pragma unroll
                for (int v = 0; v < 4; ++v) wl[v] = sm.w[v][r][f + 2];
                if (!physical<T, 2>(wl, fp.gm1)) err |= 2u;
            }
            if (!physical<T, 2>(wr, fp.gm1)) {
#pragma unroll
                for (int v = 0; v < 4; ++v) wr[v] = sm.w[v][r][f + 3];
                if (!physical<T, 2>(wr, fp.gm1)) err |= 2u;
            }
            merge_values<T, 2>(wl, wr, fp, w0);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                sm.w0[0][v][r][f] = w0[v];
                sm.w0[1][v][r][f] = (T(1.25) * (sm.w[v][r][f + 3] - sm.w[v][r][f + 2])
                                     - T(1.0 / 12.0) * (sm.w[v][r][f + 4] - sm.w[v][r][f + 1])) * ih;
            }
        }
        __syncthreads();
    }

    // phase 2: per (face segment, Gauss point): tangential TENO-D of the line
    // averages to the Gauss point, then merge + flux.  The two lanes of a face
    // segment split the work: lane gpi reconstructs side gpi (0: left, 1:
    // right) at both Gauss points, keeps its own point (xi = -g for lane 0, +g
    // for lane 1: one signed g, no selection) and hands the other point's
    // values to its partner.  A lane's own side goes first into the flux,
    // whose sign says which of the two that is; after it they average
    // (weights 1/2).
    const T tdt = s_scal[0];
    const T iht = s_scal[3];
    const T gA = T(-0.28867513459481288), gB = T(0.28867513459481288);  // -+1/(2 sqrt 3)
    const int np = nr * nf;
#pragma unroll 1
    for (int task = tid; (task & ~31) < 2 * np; task += NT) {  // whole warps
        // lanes past the last pair repeat it
        const int pair = COUNT ? min(task >> 1, np - 1) : task >> 1, gpi = task & 1;
        const int r = whole ? pair / NF : pair / nf, f = pair - r * nf;
        // faces n0+f <= nn on rows t0+r < nt exist; the rest of the tile is padding
        const bool valid = COUNT || ((n0 + f <= a.nn) && (t0 + r < a.nt));
        if (!COUNT && !__any_sync(0xffffffffu, valid)) continue;
        const T gs = gpi ? gB : gA;
        Side<T> L, R;  // own side, partner's side
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            // line averages of the side's value (W) and normal slope (Wn) at
            // the own (a) and the partner's (b) Gauss point: value and
            // tangential derivative of W, value of Wn
            T wa, wda, wb, wdb, na, nb;
            if constexpr (sizeof(T) == 4 && RB <= 1) {
                // both streams as one packed pair (x: W, y: Wn)
                f2 q[5];
#pragma unroll
                for (int s = 0; s < 5; ++s) {
                    const Pair2<T> p = sm.rec[gpi][v][r + s][f];
                    q[s] = f2(p.v, p.s);
                }
                f2 va, da, vb, db;
                packed_gauss<RB>(q, tnt, -gs, gs, vb, db, va, da);
                wa = va.x(), wda = da.x(), wb = vb.x(), wdb = db.x(), na = va.y(), nb = vb.y();
            } else {
                T q[5], qs[5];
                TenoSel<T> S;
                T dn;
#pragma unroll
                for (int s = 0; s < 5; ++s) {
                    const Pair2<T> p = sm.rec[gpi][v][r + s][f];
                    q[s] = p.v;
                    qs[s] = p.s;
                }
                rec_select<RB>(q, tnt, S);
                rec_gauss_pm<RB>(S, gs, wb, wdb, wa, wda);
                rec_select<RB>(qs, tnt, S);
                rec_gauss_pm<RB>(S, gs, nb, dn, na, dn);
            }
            L.W[v] = wa;
            R.W[v] = __shfl_xor_sync(0xffffffffu, wb, 1);
            L.Wt[v] = wda * iht;
            R.Wt[v] = __shfl_xor_sync(0xffffffffu, wdb, 1) * iht;
            L.Wn[v] = na;
            R.Wn[v] = __shfl_xor_sync(0xffffffffu, nb, 1);
        }
        T F[4] = {T(0), T(0), T(0), T(0)}, dF[4] = {T(0), T(0), T(0), T(0)};
        if (valid) {
            auto state = [&](int k, Side<T>& S, Prim<T>& p) {
                if (prim_state<T, 2>(S.W, fp.gm1, p)) return;
                const int side = k ^ gpi;  // 0: left, 1: right
#pragma unroll
                for (int v = 0; v < 4; ++v) { S.W[v] = sm.w[v][r + 2][f + 2 + side]; S.Wn[v] = S.Wt[v] = T(0); }
                nfb += task < 2 * np;
                if (!prim_state<T, 2>(S.W, fp.gm1, p)) err |= 2u;
            };
            if constexpr (CONV) {
                // Step 4: the equilibrium state and slopes at this lane's Gauss
                // point, linear (quartic) reconstructions of the rows' merges
                T w0g[4], w0t[4], w0n[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    T q[5], dd;
#pragma unroll
                    for (int s = 0; s < 5; ++s) q[s] = sm.w0[0][v][r + s][f];
                    quartic_gauss(q, gs, w0g[v], dd);
                    w0t[v] = dd * iht;
#pragma unroll
                    for (int s = 0; s < 5; ++s) q[s] = sm.w0[1][v][r + s][f];
                    quartic_gauss(q, gs, w0n[v], dd);
                }
                // a non-physical linear state (the quartic across a
                // discontinuity) falls back to the kinetic merge at the point
                if (physical<T, 2>(w0g, fp.gm1)) {
                    point_flux<T, 2, NONEQ, PRFIX>(L, R, gpi ? T(-1) : T(1), fp, F, dF, a.stage == 1, state, w0n, w0g, w0t);
                } else {
                    nfb += task < 2 * np;
                    point_flux<T, 2, NONEQ, PRFIX>(L, R, gpi ? T(-1) : T(1), fp, F, dF, a.stage == 1, state);
                }
            } else {
                point_flux<T, 2, NONEQ, PRFIX>(L, R, gpi ? T(-1) : T(1), fp, F, dF, a.stage == 1, state);
            }
        }
        // the stage's combinations at both points, averaged (weights 1/2): each
        // lane finishes half of the face's values, one shuffle per value
        // stage 1: lane 0 the four W* combinations, lane 1 the accumulator's;
        // stage 2: variables 2 gpi and 2 gpi + 1
        T g0[4], g1[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) stage_comb<T>(a.stage, F[v], dF[v], tdt, g0[v], g1[v]);
        if (a.stage == 1) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const T got = __shfl_xor_sync(0xffffffffu, gpi ? g0[v] : g1[v], 1);
                sF[sfi(4 * gpi + v, r, f)] = T(0.5) * ((gpi ? g1[v] : g0[v]) + got);
            }
        } else {
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const T got = __shfl_xor_sync(0xffffffffu, gpi ? g0[v] : g0[v + 2], 1);
                sF[sfi(2 * gpi + v, r, f)] = T(0.5) * ((gpi ? g0[v + 2] : g0[v]) + got);
            }
        }
    }
    __syncthreads();

    // phase 3: flux divergence; the y sweep updates the float64 state.  Each
    // thread reads the inputs it copied itself
    copy_wait<0>();
    T sig = T(0);
    const T cn = s_scal[1];
    auto base64 = [&](int v, int k, long long go) {
        if constexpr (STAGED) return sm.base[v][k];
        else return a.base[go];
    };
    auto basef = [&](int v, int k, long long go) {
        if constexpr (STAGED) return reinterpret_cast<const float*>(sm.base[v])[k];
        else return a.basef[go];
    };
    auto inc = [&](int q, int v, int k, long long go) {
        if constexpr (STAGED) return sm.inc[q][v][k];
        else return static_cast<const T*>(q ? a.inc1 : a.inc0)[go];
    };
#pragma unroll 1
    for (int k = tid; k < TN * TT; k += NT) {
        // x faces: the normal (x) index fastest; y faces: the tangential (x) index
        const int r = fy ? k % TT : k / TN, c = fy ? k / TT : k % TN;
        const int in = n0 + c, it = t0 + r;
        if (in < a.nn && it < a.nt) {
            const int o = org + in * sn + it * st;
            T* inc0 = static_cast<T*>(a.inc0);
            T* inc1 = static_cast<T*>(a.inc1);
            double wn[4];
            T wf[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const long long go = (v == 0 ? 0 : (v == 1 ? pv1 : (v == 2 ? pv2 : pv3))) + o;
                const T d0 = cn * (sF[sfi(v, r, c + 1)] - sF[sfi(v, r, c)]);
                const T d1 = (a.stage == 1)
                           ? cn * (sF[sfi(4 + v, r, c + 1)] - sF[sfi(4 + v, r, c)])
                           : T(0);
                if (a.pass == 0) {
                    inc0[go] = d0;
                    if (a.stage == 1) inc1[go] = d1;
                } else if constexpr (sizeof(T) == 4) {
                    if (a.stage == 1) {
                        a.out0f[go] = basef(v, k, go) - (inc(0, v, k, go) + d0);
                        inc1[go] = inc(1, v, k, go) + d1;
                    } else {
                        const double res = base64(v, k, go) - widen(inc(1, v, k, go) + inc(0, v, k, go) + d0);
                        a.out0[go] = res;
                        wf[v] = narrow(res);  // local order; the CFL rate only needs |U|
                        a.out0f[go] = wf[v];
                    }
                } else if (a.stage == 1) {
                    const double w = base64(v, k, go);
                    a.out0[go] = w - (double)(inc(0, v, k, go) + d0);
                    a.out1[go] = w - (double)(inc(1, v, k, go) + d1);
                } else {
                    const double res = base64(v, k, go) - (double)(inc(0, v, k, go) + d0);
                    a.out0[go] = res;
                    wn[v] = res;  // local order; the CFL rate only needs |U|
                }
            }
            if (a.with_sigma) {
                if constexpr (sizeof(T) == 4) sig = fmax(sig, cell_sigma<T, T>(wf, 2, s_scal[4], s_scal[5], s_scal[6], err));
                else sig = fmax(sig, cell_sigma<T>(wn, 2, s_scal[4], s_scal[5], s_scal[6], err));
            }
        }
    }
    block_commit<NT, T>(sig, a.with_sigma != 0, err, nfb, ds, a.commit != 0);
}

}  // namespace gks
