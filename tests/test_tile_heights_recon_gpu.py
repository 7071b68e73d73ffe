"""Every reconstruction and merge on every tile height of the 2-D sweep (float32
16, 8 and 4 rows, float64 4 and 2), in both directions, against the FP64
oracle: strips of two tile columns that are periodic copies of a 33 x 53 (53 x
33) plane, whose step the oracle gives; 53 rows put every copy elsewhere in its
tiles.  A strip takes a height by its length (gks_k2d_select.cu): on 152 SMs
1166 rows the 8- (float64 4-) row tiles, 3604 the 16-row ones; its other
direction the 4- (2-) and the 8-row ones.

Tolerances are those of one step in the parity tests: 1e-12 relative L1 for
float64 and 1e-5 for the float32-flux path."""
import numpy as np
import pytest

import oracle as O
from paper_2309_10534_gb300 import workloads as WL

pytestmark = pytest.mark.gpu
VARIANTS = {
    "teno_d": {}, "ns": dict(tau="ns", mu=0.002, Pr=0.73), "weno_ao": dict(recon="weno_ao"),
    "weno_z": dict(recon="weno_z"), "teno5": dict(recon="teno5"), "charvars": dict(charvars=1),
    "average": dict(merge="average"),
}


@pytest.mark.parametrize("along_y", [True, False])
@pytest.mark.parametrize("variant", sorted(VARIANTS))
def test_every_variant_on_every_tile_height(along_y, variant):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks
    build.build()
    nx, ny = (33, 53) if along_y else (53, 33)
    kw = dict(bc=("periodic",) * 4, **VARIANTS[variant])
    W = WL.random_smooth_2d(nx, ny, seed=nx, kmax=3)
    P = O.make_problem(2, nx, ny, lx=nx / 32.0, ly=ny / 32.0, **kw)
    dt = 0.4 * O.dt(P, W)
    ref = O.step(P, W, dt)
    for k in (1, 22, 68):
        kx, ky = (1, k) if along_y else (k, 1)
        want = np.tile(ref, (1, ky, kx))
        for precision, tol in (("fp64", 1e-12), ("fp32", 1e-5)):
            S = gks.Solver(2, nx * kx, ny * ky, lx=nx * kx / 32.0, ly=ny * ky / 32.0, precision=precision, **kw)
            S.set_state(np.tile(W, (1, ky, kx)))
            S.step(dt)
            assert float(np.abs(S.get_state() - want).sum() / np.abs(want).sum()) < tol, (k, precision)
