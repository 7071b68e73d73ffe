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
long long blocks(const SweepArgs& a, int tt) { return (long long)((a.nn + SWEEP_TN - 1) / SWEEP_TN) * ((a.nt + tt - 1) / tt); }
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
// SM) move the most cells per second, 8 rows (512 threads, one point per
// thread) take 0.6 of their time per block and half the cells, 4 rows half of
// that again.  So 16 rows win where the chip is filled many times over and
// the others where a last wave would be nearly empty or the grid does not
// fill the chip at all.  One step, ms (16 / 8 / 4 rows): 64^2 0.083 / 0.053 /
// 0.048, 256^2 0.089 / 0.080 / 0.087, 400^2 0.182 / 0.168 / 0.170, 512^2
// 0.228 / 0.246 / 0.254, 1024^2 0.750 / 0.833 / 0.893.
cudaError_t launch_sweep_f32(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                             const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    const long long sms = std::max(1, a.sms), b16 = blocks(a, 16), b8 = blocks(a, 8);
    if (blocks(a, 4) <= sms) return sweep_f32_t4(g, a, hf, tn, tt, ds, st);
    // waves of two blocks per SM, weighted by a block's time
    const long long w16 = 10 * ((b16 + 2 * sms - 1) / (2 * sms)), w8 = 6 * ((b8 + 2 * sms - 1) / (2 * sms));
    return w16 <= w8 || a.nt > 65535 * 8 ? sweep_f32_t16(g, a, hf, tn, tt, ds, st) : sweep_f32_t8(g, a, hf, tn, tt, ds, st);
}

// float64: 4 rows (128 threads at 210 registers, two blocks per SM, which
// cover each other's barriers); 2 rows where even those leave SMs idle (a last
// column of less than 8 cells is a small part of a block's work).  One step,
// ms (8 rows in one 256-thread block / 4 / 2), when the last tiles of a line
// were whole: 64^2 0.83 / 0.55 / 0.37, 400^2 3.11 / 2.89 / 3.09, 1024^2 16.8 /
// 16.5 / 18.0; since they do only their own work (4 / 2): 96^2 0.350 / 0.337,
// 100^2 0.348 / 0.336, and 64^2 0.209, 400^2 2.53 with the choice made here.
cudaError_t launch_sweep_f64(const GridDev& g, const SweepArgs& a, const HostFlux& hf, const TenoParams& tn,
                             const TenoParams& tt, DevState* ds, cudaStream_t st)
{
    const long long full = std::max(1ll, ((long long)a.nn + SWEEP_TN - 8) / SWEEP_TN) * ((a.nt + 1ll) / 2);
    if (full <= std::max(1, a.sms)) return sweep_f64_t2(g, a, hf, tn, tt, ds, st);
    return sweep_f64_t4(g, a, hf, tn, tt, ds, st);
}

}  // namespace gks
