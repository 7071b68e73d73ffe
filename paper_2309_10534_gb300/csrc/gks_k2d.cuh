// gks_k2d.cuh -- launcher of the 2-D sweep for one tile shape; each
// translation unit instantiates the shapes it names.
#pragma once

#include "gks_launch.h"

namespace gks {

// tiles of TT rows, NT threads, MB blocks resident per SM
template <typename T, int TT, int NT, int MB>
struct SweepTile {
    template <bool NONEQ, bool PRFIX, int REC>
    static cudaError_t one(const GridDev& g, SweepArgs a, const FluxParams<T>& fp, const TenoParams& tn,
                           const TenoParams& tt, DevState* ds, cudaStream_t st)
    {
        constexpr int TN = SWEEP_TN;
        const size_t smem = sizeof(SweepShared<T, TN, TT, MB, rec_conventional(REC)>);
        const unsigned cols = (a.nn + TN - 1) / TN, rows = (a.nt + TT - 1) / TT;
        // a grid's y extent ends at 65535 (a plane that tall has few columns)
        a.tall = sweep_tall<T>(TT) && rows > 65535;
        const dim3 grid(a.tall ? rows : cols, a.tall ? cols : rows);
        k2d_sweep<T, NONEQ, PRFIX, TN, TT, NT, MB, REC><<<grid, NT, smem, st>>>(g, a, fp, teno_t<T>(tn), teno_t<T>(tt), ds);
        return cudaGetLastError();
    }
    template <int REC>
    static cudaError_t rec(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                           const TenoParams& tt, DevState* ds, cudaStream_t st)
    {
        const FluxParams<T> fp = make_flux_params<T>(hf);
        if (hf.tau_mode == 0) return one<false, false, REC>(g, a, fp, tn, tt, ds, st);
        if (hf.prfac != 0.0 && hf.tau_mode == 2) return one<true, true, REC>(g, a, fp, tn, tt, ds, st);
        return one<true, false, REC>(g, a, fp, tn, tt, ds, st);
    }
    static cudaError_t launch(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                              const TenoParams& tt, DevState* ds, cudaStream_t st)
    {
        switch (tn.recon) {
        case 1: return rec<1>(g, a, hf, tn, tt, ds, st);
        case 2: return rec<2>(g, a, hf, tn, tt, ds, st);
        case 3: return rec<3>(g, a, hf, tn, tt, ds, st);
        case REC_TENO_CHAR: return rec<REC_TENO_CHAR>(g, a, hf, tn, tt, ds, st);
        default: return rec<0>(g, a, hf, tn, tt, ds, st);
        }
    }
    // raise the dynamic shared-memory limit (current device)
    template <bool NONEQ, bool PRFIX, int REC>
    static cudaError_t smem()
    {
        return cudaFuncSetAttribute(k2d_sweep<T, NONEQ, PRFIX, SWEEP_TN, TT, NT, MB, REC>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(SweepShared<T, SWEEP_TN, TT, MB, rec_conventional(REC)>));
    }
    template <int REC>
    static cudaError_t smem_rec()
    {
        cudaError_t e = smem<false, false, REC>();
        if (e == cudaSuccess) e = smem<true, false, REC>();
        if (e == cudaSuccess) e = smem<true, true, REC>();
        return e;
    }
    static cudaError_t prepare()
    {
        cudaError_t e = smem_rec<0>();
        if (e == cudaSuccess) e = smem_rec<1>();
        if (e == cudaSuccess) e = smem_rec<2>();
        if (e == cudaSuccess) e = smem_rec<3>();
        if (e == cudaSuccess) e = smem_rec<REC_TENO_CHAR>();
        return e;
    }
};

}  // namespace gks
