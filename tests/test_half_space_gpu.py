"""The start of the half-space moments, erfc(-z)/2 and exp(-z^2), as the device
forms it: the kinetic merge and the side terms scale every moment of a side by
these two, and where both sides move apart nothing else is left."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gks():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_10534_gb300 import build, gks as G
    build.build()
    return G


def test_float64_keeps_its_relative_accuracy_in_the_vanishing_half(gks):
    """Bounds in units of 2^-53, from the documented errors of exp (1 ulp = 2
    units) and erfcx (4 ulp): exp(-z^2) 2 + 1 (the correction's rounding), the
    half 3 + 8 + 1, and 2 more where it is subtracted from one."""
    mp = pytest.importorskip("mpmath")
    rng = np.random.default_rng(1)
    z = np.concatenate([rng.uniform(-26, -4, 400), rng.uniform(-4, 6, 400), [0.0, -0.0, 1e-300, -1e-9]])
    h, g = gks.eval_half_space(z, "fp64")
    with mp.workdps(40):
        zz = [mp.mpf(float(x)) for x in z]
        eh = [abs(mp.mpf(float(a)) / (mp.erfc(-x) / 2) - 1) * 2**53 for a, x in zip(h, zz)]
        eg = [abs(mp.mpf(float(a)) / mp.exp(-x * x) - 1) * 2**53 for a, x in zip(g, zz)]
        assert max(eg) <= 3 and max(eh) <= 14, (float(max(eg)), float(max(eh)))
