"""State copies in and out at the widths where the copy kernel changes its
block shape, and their float32 shadow."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,nx,ny", [(1, n, 1) for n in (3, 255, 256, 257, 70000)] +
                         [(2, n, 41) for n in (3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 65)] + [(2, 3, 70000)])
def test_state_copies_at_the_edges_of_block_shapes(dim, nx, ny, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks
    build.build()
    S = gks.Solver(dim, nx, ny, precision=precision)
    rng = np.random.default_rng(nx)
    W = rng.uniform(0.9, 1.1, S.shape)
    S.set_state(W)
    assert np.array_equal(S.get_state(), W)
    t = torch.from_numpy(W).cuda()
    S.set_state(t)
    assert torch.equal(S.get_state(torch.empty_like(t)), t)
    # a uniform state in one cell's place: the stages read the copy that was set
    W = np.broadcast_to(np.array([1.0, 0.0, 2.5] if dim == 1 else [1.0, 0.0, 0.0, 2.5])[:, None, None], S.shape)
    S.set_state(np.array(W))
    S.step(1e-3)
    assert float(np.abs(S.get_state() - W).max()) < (1e-14 if precision == "fp64" else 1e-6)
