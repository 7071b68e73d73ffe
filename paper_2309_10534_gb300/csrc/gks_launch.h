// gks_launch.h -- host-side launchers of the stage kernels, one translation
// unit per precision so the heavy instantiations compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include "../../include/gks.h"
#include "gks_kernels.cuh"

namespace gks {

// tile of the 2-D sweep: TN cells along the face normal (TN + 1 faces, the
// lanes of a warp) x rows by the grid's size (gks_k2d_select.cu)
constexpr int SWEEP_TN = 31;
// cells per block of the 1-D stage (TN + 2 = 128 threads: one per
// reconstructed cell, face and updated cell)
constexpr int STAGE1D_TN = 126;
// Up to 160 cells per SM a 1-D stage takes k1d_stage_wide: its tiles of 30
// cells and three warps have a third of the chain of a 126-cell tile and fill
// the SMs sooner, but reconstruct 32 cells for 30; once several blocks share
// every SM, the 126-cell tiles move more cells.  One step, us (wide / 126), in
// float64 TENO-D, float64 WENO5-AO and float32 TENO-D: 400 cells 37 / 76,
// 43 / 96, 12.2 / 15.7; 12 000 cells 51 / 71, 69 / 95, 13.5 / 15.3; 24 000
// cells 86 / 98, 130 / 156, 14.6 / 16.9; 28 000 cells 101 / 96, 154 / 157,
// 15.5 / 15.4; 128 000 cells 353 / 316, 573 / 525, 37 / 20.
constexpr int STAGE1D_WIDE_NX = 152 * 160;

struct HostFlux {
    double gamma, K, ntot, c1, c2, mu, prfac;
    int tau_mode;
    int merge = 0;
};

cudaError_t launch_sweep_f32(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                             const TenoParams& tt, DevState* ds, cudaStream_t st);
cudaError_t launch_sweep_f64(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                             const TenoParams& tt, DevState* ds, cudaStream_t st);
// raise the dynamic shared-memory limit of every 2-D sweep instantiation
// (current device); call once before the first launch
cudaError_t prepare_sweep_f32();
cudaError_t prepare_sweep_f64();
cudaError_t launch_stage1d(int fp32, const GridDev& g, const Stage1DArgs& a, const HostFlux& hf,
                           const TenoParams& tn, DevState* ds, cudaStream_t st);

// Range checks of a gks_scheme shared by every entry point that takes one
// (gks_set_scheme, gks_batch_set_scheme, gks_step1d_noalloc).  Returns
// nullptr when the scheme is valid, else the reason, with *code set to the
// status to return.  The CFL number is checked only where it is used
// (check_cfl != 0).
const char* scheme_problem(const gks_scheme* s, int check_cfl, gks_status* code);

template <typename T>
inline FluxParams<T> make_flux_params(const HostFlux& h)
{
    FluxParams<T> p;
    p.gm1 = (T)(h.gamma - 1.0);
    p.K = (T)h.K;
    p.dt = (T)0;
    p.c1 = (T)h.c1;
    p.c2 = (T)h.c2;
    p.mu = (T)h.mu;
    p.prfac = (T)h.prfac;
    p.hkv = (T)(0.5 * (h.ntot - 1.0));
    p.cp = (T)(0.5 * (h.ntot + 2.0));
    p.tau_mode = h.tau_mode;
    p.merge = h.merge;
    return p;
}

}  // namespace gks
