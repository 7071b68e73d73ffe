"""A 1-D grid whose three variables hold more than 2^31 elements: offsets that
do not fit in 32 bits, in the stages, the copies, the rate and the selection
count."""
import numpy as np
import pytest

from paper_2309_10534_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-7), ("fp64", 1e-14)])
def test_tube_of_copies_stays_one(precision, tol):
    """A periodic tube of 7.2e8 cells made of copies of a 28800-cell one (both
    take the 126-cell tiles) keeps the short tube's values.  A copy lies in
    other tiles, so the bound is the rounding of a step."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks
    build.build()
    n, k = 28800, 25000
    if torch.cuda.mem_get_info()[0] < 150e9:
        pytest.skip("needs 150 GB of device memory")
    x = 2 * np.pi * (np.arange(n) + 0.5) / n
    W0 = WL.conserved_1d((1 + 0.2 * np.sin(40 * x)) * np.where(x > np.pi, 1.5, 1.0), 0.3 + 0.1 * np.cos(30 * x),
                         1 + 0.1 * np.sin(50 * x + 1), 1.4)[:, None, :]
    kw = dict(bc=("periodic",) * 4, precision=precision)
    a, b = gks.Solver(1, n, lx=float(n), **kw), gks.Solver(1, n * k, lx=float(n) * k, **kw)
    W = torch.from_numpy(W0).cuda()
    big = W.repeat(1, 1, k)
    a.set_state(W)
    b.set_state(big)
    fa, fb = a.selection_flips(), b.selection_flips()
    assert fb == {name: k * v for name, v in fa.items()}
    assert a.compute_dt() == b.compute_dt()
    a.step(0.2)
    b.step(0.2)
    a.get_state(W)
    b.get_state(big)
    b.diagnostics()
    b.close()
    err = float(big.view(3, k, n).sub_(W.view(3, 1, n)).abs_().sum()) / (k * float(W.abs().sum()))
    del big
    torch.cuda.empty_cache()
    assert err < tol
