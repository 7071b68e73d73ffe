// gks_k2d_f32_t16.cu -- the 2-D sweep in float, tiles of 16 rows.
#include "gks_k2d.cuh"

namespace gks {

cudaError_t sweep_f32_t16_prepare()
{
    return SweepTile<float, 16, 512, 2>::prepare();
}
cudaError_t sweep_f32_t16(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                        const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    return SweepTile<float, 16, 512, 2>::launch(g, a, hf, tn, tt, ds, st);
}

}  // namespace gks
