// gks_k2d_f32_t4.cu -- the 2-D sweep in float, tiles of 4 rows.
#include "gks_k2d.cuh"

namespace gks {

cudaError_t sweep_f32_t4_prepare()
{
    return SweepTile<float, 4, 256, 4>::prepare();
}
cudaError_t sweep_f32_t4(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                        const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    return SweepTile<float, 4, 256, 4>::launch(g, a, hf, tn, tt, ds, st);
}

}  // namespace gks
