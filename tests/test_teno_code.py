"""The float64 kernels' TENO-D selection decided in float32 (where float32 can
decide it) against the selection in float64: same code for every stencil that
float32 decides, over scales, powers, cut-offs and special values (CPU)."""
import numpy as np
import pytest

from test_host_replica import G  # noqa: F401  (builds the library)


def _stencils(rng, n):
    """Jumps, waves, noise and constant runs over many scales."""
    x = np.arange(5)
    for _ in range(n):
        amp, base = 10.0 ** rng.uniform(-18, 3), 10.0 ** rng.uniform(-3, 3)
        kind = rng.integers(5)
        if kind == 0:
            q = base + amp * rng.standard_normal(5)
        elif kind == 1:
            q = base + amp * np.sin(rng.uniform(0.01, 2) * x + rng.uniform(0, 6))
        elif kind == 2:  # a jump over a small wave
            q = base * np.where(x < rng.integers(1, 5), 1.0, rng.uniform(0.1, 10)) + amp * rng.standard_normal(5)
        elif kind == 3:  # differences spread over decades: ratios near the cut-offs
            q = base + amp * np.cumsum(10.0 ** rng.uniform(-2, 0, 5) * rng.choice([-1, 1], 5))
        else:  # constant runs
            q = np.where(x < rng.integers(0, 6), base, base + amp)
        yield q


@pytest.mark.parametrize("q_pow", [1, 6, 7, 32])
@pytest.mark.parametrize("ct1,ct2", [(1e-7, 1e-5), (1e-4, 1e-5), (0.3, 0.2), (0.0, 1e-5)])
def test_float32_decision_is_the_float64_selection(G, q_pow, ct1, ct2):
    rng = np.random.default_rng(100 * q_pow + int(1e3 * ct1))
    decided = total = 0
    for q in _stencils(rng, 2500):
        c64, c32 = G.host_teno_code(q, q_pow=q_pow, ct1=ct1, ct2=ct2)
        assert c32 in (0, c64), (q.tolist(), c64, c32)
        decided += c32 != 0
        total += 1
    if ct1 > 0.0:  # a zero cut-off is never decided in float32
        assert decided > 0.7 * total


@pytest.mark.parametrize("q", [[1.0] * 5, [0.0] * 5, [0, 0, 0, 0, 1e-320], [0, 0, 1e-200, 0, 0], [1, 1, 1, 1, 2],
                               [1e300, -1e300, 1e300, 0, 0], [1, 2, np.inf, 3, 4], [1, 2, np.nan, 3, 4],
                               [1, 1 + 2e-16, 1, 1, 1], [0, 1e150, 0, 0, 0], [0, 0, 1e-17, 2e-17, 1.0]])
@pytest.mark.parametrize("eps", [1e-40, 0.0, 1e-8, 1.0])
def test_special_values(G, q, eps):
    c64, c32 = G.host_teno_code(np.array(q, dtype=float), eps=eps)
    assert c32 in (0, c64)


def test_constant_stencil_is_decided(G):
    """The most common stencil of a quiescent region takes no float64."""
    assert G.host_teno_code(np.full(5, 1.25)) == (1, 1)
