// gks_k2d_select.cu -- which tile shape a 2-D sweep takes.
//
// Tiles hold 31 cells along the normal.  The rows of a tile trade its halo
// (two rows on either side are reconstructed again) and its share of the
// block's fixed costs against how evenly the blocks fill the chip.
#include <algorithm>

#include "gks_launch.h"

namespace gks {

#define GKS_SWEEP(name)                                                                                        \
    cudaError_t name##_prepare();                                                                              \
    cudaError_t name(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,           \
                     const TenoParams& tt, DevState* ds, cudaStream_t st);
GKS_SWEEP(sweep_f32_t16)
GKS_SWEEP(sweep_f32_t8)
GKS_SWEEP(sweep_f32_t4)
GKS_SWEEP(sweep_f64_t4)
GKS_SWEEP(sweep_f64_t2)
#undef GKS_SWEEP

namespace {
// A sweep's time by its most loaded SM: the blocks it gets times a block's
// time when the SM is shared, and what the launch and the first block's chain
// add (relative units; the measurements stand at each use)
int sweep_time(const SweepArgs& a, int rows, int per_block, int fixed)
{
    const long long blocks = (long long)((a.nn + SWEEP_TN - 1) / SWEEP_TN) * ((a.nt + rows - 1) / rows);
    const long long sms = std::max(1, a.sms), load = (blocks + sms - 1) / sms;
    return (int)std::min<long long>(load, 1 << 20) * per_block + fixed;
}
}  // namespace

cudaError_t prepare_sweep_f32()
{
    cudaError_t e = sweep_f32_t16_prepare();
    if (e == cudaSuccess) e = sweep_f32_t8_prepare();
    if (e == cudaSuccess) e = sweep_f32_t4_prepare();
    return e;
}
cudaError_t prepare_sweep_f64()
{
    const cudaError_t e = sweep_f64_t4_prepare();
    return e == cudaSuccess ? sweep_f64_t2_prepare() : e;
}

// float32: 16 rows (512 threads, two face points per thread, two blocks per
// SM) reconstruct the least halo, 8 rows (512 threads, one point per thread)
// and 4 rows (256 threads) spread a grid over more SMs.  One step, us (16 / 8
// / 4 rows), by which the times below are taken: 64^2 72 / 47 / 45, 128^2 73 /
// 48 / 50, 192^2 72 / 64 / 58, 256^2 73 / 65 / 68, 320^2 103 / 91 / 102, 400^2
// 145 / 127 / 134, 512^2 182 / 184 / 199, 1024^2 595 / 627 / 695.
cudaError_t launch_sweep_f32(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                             const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    // more 16-row tiles than a grid's y extent takes (1 048 560 rows): the
    // tiles whose rows can lie along x
    if ((a.nt + 15) / 16 > 65535) return sweep_f32_t4(g, a, hf, tn, tt, ds, st);
    const int t16 = sweep_time(a, 16, 385, 320), t8 = sweep_time(a, 8, 208, 240), t4 = sweep_time(a, 4, 117, 260);
    if (t4 < t8 && t4 < t16) return sweep_f32_t4(g, a, hf, tn, tt, ds, st);
    return t8 < t16 ? sweep_f32_t8(g, a, hf, tn, tt, ds, st) : sweep_f32_t16(g, a, hf, tn, tt, ds, st);
}

// float64: 4 rows (128 threads at 210 registers, two face points per thread,
// two blocks per SM, which cover each other's barriers) or 2 rows (one point
// per thread) where those even out the SMs' loads.  One step, us (4 / 2 rows),
// by which the times below are taken: 64^2 353 / 208, 96^2 350 / 338, 128^2
// 592 / 416, 200^2 997 / 870, 400^2 2532 / 2718, 1024^2 15 670 / 16 918.
cudaError_t launch_sweep_f64(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                             const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    if (sweep_time(a, 2, 151, 40) < sweep_time(a, 4, 280, 70)) return sweep_f64_t2(g, a, hf, tn, tt, ds, st);
    return sweep_f64_t4(g, a, hf, tn, tt, ds, st);
}

}  // namespace gks
