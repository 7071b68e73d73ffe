"""Planes with more rows of tiles than a grid's y extent takes, in both
precisions: every height and orientation that a context accepts runs."""
import pytest

from paper_2309_10534_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-7), ("fp64", 1e-14)])
@pytest.mark.parametrize("along_y", [True, False])
def test_strip_of_copies_stays_one(along_y, precision, tol):
    """A periodic strip made of 1000 copies of a short one takes the short
    strip's values, 1.1 million cells long (65535 rows of 16-row tiles hold
    1 048 560).  A copy lies in other tiles, so the bound is the rounding of
    a step: 1e-7 float32, 1e-14 float64."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks
    build.build()
    k, n = 1000, 1100
    nx, ny = (3, n) if along_y else (n, 3)
    W = torch.from_numpy(WL.random_smooth_2d(nx, ny, seed=9, kmax=1)).cuda()
    rep = (1, k, 1) if along_y else (1, 1, k)
    kw = dict(bc=("periodic",) * 4, precision=precision)
    a = gks.Solver(2, nx, ny, lx=float(nx), ly=float(ny), **kw)
    nx, ny = (nx, ny * k) if along_y else (nx * k, ny)
    b = gks.Solver(2, nx, ny, lx=float(nx), ly=float(ny), **kw)
    a.set_state(W)
    big = W.repeat(rep)
    b.set_state(big)
    for _ in range(2):
        a.step(0.2)
        b.step(0.2)
    a.get_state(W)
    got = b.get_state(torch.empty_like(big))
    b.diagnostics()
    want = W.repeat(rep)
    assert float((got - want).abs().sum() / want.abs().sum()) < tol
