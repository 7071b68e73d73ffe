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


# ------------------------------------------------------------ steps the library did not launch itself
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_advance_after_steps_replayed_from_a_callers_graph(gks, precision):
    """gks_step only launches, so a caller can capture it and replay it.  Time
    and step count are the device's: advance_to goes on from there, whatever
    the library last read back."""
    import torch
    s = WL.riemann2d(24, split=0.8)
    S, ref = gks.solver_for(s, precision), gks.solver_for(s, precision)
    dt = 0.5 * S.compute_dt()
    S.step(dt)       # every kernel is loaded before the capture
    S.diagnostics()  # and that step is done before the stream changes
    st = torch.cuda.Stream()
    S.set_stream(st.cuda_stream)
    S.set_state(s.W)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        S.step(dt)
    assert S.diagnostics().steps == 0
    with torch.cuda.stream(st):
        for _ in range(3):
            g.replay()
    n, t = S.advance_to(1e9, max_steps=2)
    for _ in range(3):
        ref.step(dt)
    nr, tr = ref.advance_to(1e9, max_steps=2)
    assert (n, t) == (nr, tr) == (2, t) and S.diagnostics().steps == ref.diagnostics().steps == 5
    assert np.array_equal(S.get_state(), ref.get_state())
    with torch.cuda.stream(st):
        g.replay()
    st.synchronize()
    # a time already passed: nothing runs
    W = S.get_state()
    assert S.advance_to(0.5 * t) == (0, S.diagnostics().t) and np.array_equal(S.get_state(), W)


# ------------------------------------------------------------ the time step after a gradient
def test_cfl_step_after_a_replayed_gradient(gks):
    """backward leaves the context at the forward pass's final state; the CFL
    step after it takes its time step from that state, also when every
    segment of the pass was a replayed graph."""
    s = WL.isentropic_vortex(24, seed=None)
    S = gks.solver_for(s, "fp64", tau="zero")
    dt = 0.25 * S.compute_dt()
    A = gks.Adjoint(S, 2)
    A.forward(4, dt)
    WN = S.get_state()
    g = np.ones_like(s.W)
    A.backward(g)  # captures the segment
    S.step(0.0)    # leaves the next CFL time step on the device
    A.backward(g)
    assert np.array_equal(S.get_state(), WN)
    S.step(0.0)
    fresh = gks.solver_for(s, "fp64", tau="zero")
    fresh.set_state(WN)
    fresh.step(0.0)
    assert np.array_equal(S.get_state(), fresh.get_state())
