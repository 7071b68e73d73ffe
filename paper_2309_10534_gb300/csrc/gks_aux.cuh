// gks_aux.cuh -- small kernels of the step loop: ghost-layer filling, the
// CFL-rate reduction of a state, and the device-side time commit.  Included
// by the runtime translation unit only.
#pragma once

#include "gks_kernels.cuh"

namespace gks {

// ------------------------------------------------------------------ ghosts
// The ghost layers in memory, for callers that read them there (the adjoint,
// the selection count); the stage kernels form their own, and no step writes
// these, so they are filled whether or not a run is marked as finished.  One
// thread per ghost cell (cell_source).
template <typename E>
__global__ void k_fill_ghosts(const __grid_constant__ GridDev g, E* __restrict__ W, const DevState* ds)
{
    const int gx = g.nx + 2 * NG;
    const int nv = g.dim + 2;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    int i, j;  // ghosted position
    if (g.dim == 1) {
        if (idx >= 2 * NG) return;
        j = 0;
        i = idx < NG ? idx : g.nx + idx;  // 0,1,2 and nx+3.. nx+5
    } else {
        const int band = 2 * NG * gx;
        if (idx < band) {
            j = idx / gx;
            i = idx % gx;
            if (j >= NG) j = g.ny + j;  // rows ny+3 .. ny+5
        } else {
            idx -= band;
            if (idx >= 2 * NG * g.ny) return;
            j = NG + idx / (2 * NG);
            int k = idx % (2 * NG);
            i = k < NG ? k : g.nx + k;
        }
    }
    const int r0 = g.dim == 2 ? NG : 0;  // ghost rows below the interior
    const CellSrc s = g.dim == 2 ? cell_source<true>(g, i - NG, j - NG, ds, 0.0)
                                 : cell_source<false>(g, i - NG, 0, ds, 0.0);
    for (int v = 0; v < nv; ++v) {
        E val = s.state ? (E)state_value(g, s.state, v)
                        : W[(long long)v * g.plane + (long long)(s.j + r0) * g.pitch + s.i + NG];
        if ((v == 1 && s.n1) || (v == 2 && g.dim == 2 && s.n2)) val = -val;
        W[(long long)v * g.plane + (long long)j * g.pitch + i] = val;
    }
}

// honour_done: nothing where the run is finished (a call that finds its end
// time passed)
template <typename T>
__global__ void __launch_bounds__(256) k_sigma(GridDev g, const double* __restrict__ W, DevState* ds, bool honour_done)
{
    if (honour_done && ds->done) return;
    T s = T(0);
    unsigned int err = 0;
    const int nv = g.dim + 2;
    const double h = (g.dim == 2) ? fmin(g.dx, g.dy) : g.dx;
    const T gamma = (T)g.gamma, mu = (T)g.mu, th = (T)h;
    const unsigned ncell = (unsigned)((long long)g.nx * (g.dim == 2 ? g.ny : 1));  // at most 2^31
    for (unsigned c = blockIdx.x * 256u + threadIdx.x; c < ncell; c += 256u * gridDim.x) {
        const unsigned j = g.dim == 2 ? c / (unsigned)g.nx : 0u, i = c - j * (unsigned)g.nx;
        const long long off = (long long)(g.dim == 2 ? j + NG : 0) * g.pitch + i + NG;
        T w[4];
        for (int v = 0; v < nv; ++v) w[v] = from_f64<T>(W[(long long)v * g.plane + off]);
        s = fmax(s, cell_sigma<T, T>(w, g.dim, gamma, mu, th, err));
    }
    block_commit<256, T>(s, true, err, 0u, ds, false);
}

// float64 views of the float32 path's stage buffers (gks_get_buffer):
// W* from its float32 form, the accumulator from W and its increment
__global__ void k_widen(const float* __restrict__ src, double* __restrict__ dst, long long n)
{
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x) dst[i] = widen(src[i]);
}
__global__ void k_accumulator(const double* __restrict__ W, const float* __restrict__ inc, double* __restrict__ A,
                              long long n)
{
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += 256ll * gridDim.x) A[i] = W[i] - widen(inc[i]);
}

// the first dt of a call, from k_sigma's rate
__global__ void k_commit(DevState* ds)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) commit_step(ds, true);
}

}  // namespace gks
