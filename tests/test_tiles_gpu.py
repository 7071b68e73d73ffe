"""The shapes a stage kernel chooses by the grid's size, at the edges of their
ranges: 1-D short and long grids, the 2-D tile heights, the adjoint's tiles and
the step graphs of advance_to, each against the FP64 oracle.

Tolerances are those of one step in the parity tests: 1e-12 relative L1 for
float64 and 1e-5 for the float32-flux path."""
import numpy as np
import pytest

import oracle as O
from paper_2309_10534_gb300 import workloads as WL

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 1e-5}
STATES = dict(bc_in=(1.2, 0.48, 0.1, 3.4), bc_pre=(1.4, 0.0, 0.0, 2.5), shock_x0=0.3, shock_theta=1.1,
              shock_speed=4.0)


@pytest.fixture(scope="module")
def gks():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks as G
    build.build()
    return G


def rel_l1(a, b):
    a = np.asarray(a).reshape(a.shape[0], -1)
    b = np.asarray(b).reshape(b.shape[0], -1)
    return float(np.abs(a - b).sum() / np.abs(b).sum())


def _tube(n, seed):
    """Cell-to-cell noise on both sides of a jump: every selection occurs."""
    rng = np.random.default_rng(seed)
    rho = np.exp(rng.uniform(-0.3, 0.3, n)) * (1.0 + 0.5 * (np.arange(n) > n // 2))
    return WL.conserved_1d(rho, rng.uniform(-0.2, 0.2, n), np.exp(rng.uniform(-0.3, 0.3, n)), 1.4)[:, None, :]


def _check_stage_and_step(gks, dim, nx, ny, W, states=None, **kw):
    P = O.make_problem(dim, nx, ny, **kw, **(states or {}))
    dt = 0.4 * O.dt(P, W)
    ref1, ref = O.stage1(P, W, dt), O.step(P, W, dt)
    for precision, tol in TOL.items():
        S = gks.Solver(dim, nx, ny, precision=precision, **kw)
        if states:
            S.set_boundary_states(**states)
        S.set_state(W)
        S.stage(1, dt)
        assert rel_l1(S.get_buffer(1), ref1) < tol, precision
        S.set_state(W)
        S.step(dt)
        assert rel_l1(S.get_state(), ref) < tol, precision
        # the rate that the step left behind gives the next dt
        assert abs(S.compute_dt() - O.dt(P, ref)) < 10 * tol * O.dt(P, ref), precision


@pytest.mark.parametrize("nx", [3, 4, 29, 30, 31, 59, 60, 61, 127, 24320, 24321, 24337])
@pytest.mark.parametrize("recon,bc", [("teno_d", ("periodic",) * 2), ("teno_d", ("reflect", "zerograd")),
                                      ("weno_ao", ("zerograd", "noslip"))])
def test_1d_grids_at_tile_edges(gks, nx, recon, bc):
    """Warp-split tiles of 30 cells up to 24320 cells, 126-cell tiles above."""
    _check_stage_and_step(gks, 1, nx, 1, _tube(nx, nx), bc=bc + ("zerograd",) * 2, recon=recon)


@pytest.mark.parametrize("recon", ["weno_z", "teno5"])
@pytest.mark.parametrize("nx", [60, 61, 24321])
def test_1d_weno_family_at_tile_edges(gks, nx, recon):
    x = (np.arange(nx) + 0.5) / nx
    W = WL.conserved_1d(1.0 + 0.2 * np.sin(2 * np.pi * x), 0.3 + 0.1 * np.cos(2 * np.pi * x),
                        1.0 + 0.1 * np.sin(2 * np.pi * x + 1.0), 1.4)[:, None, :]
    _check_stage_and_step(gks, 1, nx, 1, W, bc=("periodic",) * 4, recon=recon)


# both sides of every choice of a tile height, in both directions (float32 4,
# 8, 16 rows; float64 2, 4), with remainders along the line and across it
SIZES_2D = [(3, 3), (31, 9), (32, 33), (64, 64), (5, 303), (5, 617), (617, 5), (95, 62), (96, 96), (4, 1300), (128, 80),
            (9700, 3)]
TAU_BC = [("euler", ("periodic",) * 4), ("zero", ("zerograd", "reflect", "symmetry", "noslip")),
          ("ns", ("inflow", "zerograd", "wall_after_x0", "moving_shock"))]


@pytest.mark.parametrize("nx,ny,tau,bc", [(nx, ny, tau, bc) for nx, ny in SIZES_2D for tau, bc in TAU_BC
                                          if nx * ny < 20000 or tau == "zero"])
def test_2d_grids_at_tile_edges(gks, nx, ny, tau, bc):
    W = WL.random_smooth_2d(nx, ny, seed=nx + ny, kmax=2)
    rng = np.random.default_rng(nx)
    W = W * np.where(np.arange(nx) > nx // 2, 1.5, 1.0) * (1.0 + 0.02 * rng.uniform(-1, 1, W.shape[1:]))
    ns = tau == "ns"
    _check_stage_and_step(gks, 2, nx, ny, W, STATES if ns else None, bc=bc, tau=tau,
                          mu=0.002 if ns else 0.0, Pr=0.73 if ns else 1.0)


@pytest.mark.parametrize("dim,nx,ny", [(1, 61, 1), (2, 33, 21)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_step_counts_around_the_graph_length(gks, dim, nx, ny, precision):
    """advance_to launches captured groups of steps and single ones for the
    rest: any limit, reached in one call or in several, gives the steps of
    step(dt=0)."""
    W = _tube(nx, 5) if dim == 1 else WL.random_smooth_2d(nx, ny, seed=5, kmax=2)
    kw = dict(bc=("periodic",) * 4, precision=precision)
    for limits in ([1], [7], [8], [9], [17], [3, 8, 1, 5]):
        S, ref = gks.Solver(dim, nx, ny, **kw), gks.Solver(dim, nx, ny, **kw)
        S.set_state(W)
        ref.set_state(W)
        for m in limits:
            assert S.advance_to(1e9, max_steps=m)[0] == m
        for _ in range(sum(limits)):
            ref.step(0.0)
        assert rel_l1(S.get_state(), ref.get_state()) < TOL[precision], limits
        assert S.diagnostics().steps == ref.diagnostics().steps == sum(limits)
    # the last step ends on the time asked for
    S.set_state(W)
    n, t = S.advance_to(0.01)
    assert abs(t - 0.01) < 1e-15 and n > 0


@pytest.mark.parametrize("nx,ny", [(8, 67), (33, 13), (64, 9), (95, 31)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-7), ("fp32", 2e-5)])
def test_vjp_at_tile_remainders(gks, nx, ny, precision, tol):
    """One step's VJP against the oracle's directional derivative (the bounds
    of the adjoint's own tests), on grids that leave remainders in every tile
    of the reverse kernels."""
    W = WL.random_smooth_2d(nx, ny, seed=21, kmax=1)
    bc = ("reflect", "zerograd", "noslip", "symmetry")
    kw = dict(lx=nx / 16.0, ly=ny / 16.0, bc=bc, tau="zero")
    P = O.make_problem(2, nx, ny, **kw)
    dt = 0.4 * O.dt(P, W)
    S = gks.Solver(2, nx, ny, precision=precision, **kw)
    g = np.random.default_rng(4).standard_normal(W.shape)
    d = WL.random_smooth_2d(nx, ny, seed=100, kmax=1) - WL.random_smooth_2d(nx, ny, seed=200, kmax=1)
    gin = gks.vjp_step(S, W, g, dt)
    h = 1e-6
    fd = (O.step(P, W + h * d, dt) - O.step(P, W - h * d, dt)) / (2 * h)
    assert abs(float((gin * d).sum()) - float((g * fd).sum())) <= tol * float(np.abs(g * fd).sum())


@pytest.mark.parametrize("nx,ny", [(3, 264000), (264000, 3)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_more_rows_of_tiles_than_a_grid_extent_takes(gks, nx, ny, precision):
    """A long periodic strip made of copies of a short one stays that: every
    copy takes the short strip's values (the same cells in other tiles)."""
    k = 2000
    sx, sy = (nx, ny // k) if ny > nx else (nx // k, ny)
    W = WL.random_smooth_2d(sx, sy, seed=9, kmax=1)
    kw = dict(bc=("periodic",) * 4, precision=precision)
    a = gks.Solver(2, sx, sy, lx=float(sx), ly=float(sy), **kw)
    b = gks.Solver(2, nx, ny, lx=float(nx), ly=float(ny), **kw)
    a.set_state(W)
    b.set_state(np.tile(W, (1, k, 1) if ny > nx else (1, 1, k)))
    a.step(0.2)
    b.step(0.2)
    ref = a.get_state()
    assert rel_l1(b.get_state(), np.tile(ref, (1, k, 1) if ny > nx else (1, 1, k))) < (1e-14 if precision == "fp64" else 1e-7)
