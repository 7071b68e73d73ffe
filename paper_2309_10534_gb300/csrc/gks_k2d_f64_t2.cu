// gks_k2d_f64_t2.cu -- the 2-D sweep in double, tiles of 2 rows.
#include "gks_k2d.cuh"

namespace gks {

cudaError_t sweep_f64_t2_prepare()
{
    return SweepTile<double, 2, 128, 2>::prepare();
}
cudaError_t sweep_f64_t2(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                        const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    return SweepTile<double, 2, 128, 2>::launch(g, a, hf, tn, tt, ds, st);
}

}  // namespace gks
