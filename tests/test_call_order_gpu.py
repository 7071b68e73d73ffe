"""Calls in orders where what one call leaves behind decides what the next one
does: each against a fresh context that is given the same state."""
import numpy as np
import pytest

from paper_2309_10534_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gks():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks as G
    build.build()
    return G


# ------------------------------------------------------------ selection counts
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,bc", [(1, ("reflect", "zerograd", "zerograd", "zerograd")), (2, ("periodic",) * 4),
                                    (2, ("reflect", "noslip", "symmetry", "zerograd"))])
def test_selection_counts_after_a_finished_run(gks, dim, bc, precision):
    """The counter reads W's ghost layers in memory, which no step writes: it
    fills them itself, also where advance_to has marked the run as finished."""
    n = 40
    if dim == 1:
        W = WL.sod(n).W
        kw = dict(bc=bc, precision=precision)
    else:
        W = WL.riemann2d(n, split=0.8).W if bc[0] == "periodic" else WL.random_smooth_2d(n, n, seed=7)
        kw = dict(bc=bc, precision=precision)
    S = gks.Solver(dim, n, n if dim == 2 else 1, **kw)
    S.set_state(W)
    assert S.advance_to(1e9, max_steps=6)[0] == 6
    fresh = gks.Solver(dim, n, n if dim == 2 else 1, **kw)
    fresh.set_state(S.get_state())
    assert S.selection_flips() == fresh.selection_flips()
