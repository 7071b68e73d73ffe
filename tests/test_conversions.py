"""The float32 kernels' integer float32 <-> float64 conversions give the bits
of the hardware's (round to nearest even), float32 denormals as zero (CPU)."""
import numpy as np

from test_host_replica import G  # noqa: F401  (builds the library)


def test_conversions_are_the_ieee_ones(G):
    rng = np.random.default_rng(1)
    n = 200000
    bits = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    y = bits.view(np.float32).copy()  # every exponent, infinities and NaN among them
    x = np.concatenate([
        rng.integers(0, 1 << 64, n // 4, dtype=np.uint64).view(np.float64),
        y[:n // 4].astype(np.float64),                                        # exact
        y[:n // 4].astype(np.float64) * (1 + 2.0 ** -24),                     # ties and near ties
        rng.standard_normal(n - 3 * (n // 4)) * 10.0 ** rng.uniform(-45, 40, n - 3 * (n // 4))])
    x[:8] = [0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235677973366e38, 3.40282346e38, 1.0 + 2.0 ** -24]
    with np.errstate(all="ignore"):
        want = x.astype(np.float32)
        got, wide = G.host_convert(x, y)
        tiny = np.abs(want) <= np.float32(1.1754944e-38)  # denormal, or rounded up to the smallest normal
        assert np.array_equal(np.isnan(got), np.isnan(want))
        ok = ~tiny & ~np.isnan(want)
        assert np.array_equal(got[ok].view(np.uint32), want[ok].view(np.uint32))
        assert np.all(np.abs(got[tiny]) <= np.float32(1.1754944e-38))
        wy = np.where(np.abs(y) < np.float32(1.1754944e-38), np.copysign(np.float32(0), y), y).astype(np.float64)
    assert np.array_equal(np.isnan(wide), np.isnan(wy))
    ok = ~np.isnan(wy)
    assert np.array_equal(wide[ok].view(np.uint64), wy[ok].view(np.uint64))
