"""The bound behind the FP32 chord direction (device.cuh, chord_direction): a chord's length and
the direction along it taken from one reciprocal square root, itself one unit in the last
place off (the bound of CUDA's rsqrt), stay within 5 units in the last place of the square root
and the divisions, so that a 29-bit cut 16 units from either end is the same."""
import numpy as np
import pytest


@pytest.mark.parametrize("scale", [1e-12, 1e-3, 1.0, 1e3, 1e12])
def test_quotients_from_one_reciprocal_square_root(scale):
    rng = np.random.default_rng(9)
    d = rng.normal(size=(200000, 3)) * 2.0 ** rng.integers(-20, 1, (200000, 3)) * scale
    l2 = (d * d).sum(axis=1)
    exact = np.sqrt(l2)
    y = (1.0 / np.sqrt(l2.astype(np.longdouble))).astype(np.float64)

    def ulps(a, b):
        return np.abs(np.abs(a).view(np.int64) - np.abs(b).view(np.int64)).max()

    for off in (-1, 0, 1):
        z = (y.view(np.int64) + off).view(np.float64)
        assert ulps(l2 * z, exact) <= 5
        for k in range(3):
            assert ulps(d[:, k] * z, d[:, k] / exact) <= 5
