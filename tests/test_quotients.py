"""Markstein's quotient (device.cuh, Over<float>) against the division, in float32 emulated in
float64, where the product of two floats, the remainder x - q d and the last sum's product are
exact: with y the correctly rounded 1/d, q + (x - q d) y is the correctly rounded x / d."""
import numpy as np
import pytest


@pytest.mark.parametrize("name", ["any", "grid", "one"])
def test_quotient_is_the_correctly_rounded_one(name):
    rng = np.random.default_rng(12)
    n = 2_000_000
    d = np.ldexp(rng.integers(1 << 23, 1 << 24, n).astype(np.float32), rng.integers(-40, 0, n)).astype(np.float32)
    x = np.ldexp(rng.integers(1 << 23, 1 << 24, n).astype(np.float32), rng.integers(-60, 10, n)).astype(np.float32)
    if name == "grid":  # the significand's low bits over its top 24 (the energy grid's position)
        d = (rng.integers(0, 1 << 23, n).astype(np.float32) * np.float32(2.0 ** -23) + np.float32(1.0)).astype(np.float32)
        x = (rng.integers(0, 1 << 29, n).astype(np.float32) * np.float32(2.0 ** -52)).astype(np.float32)
        half = d > np.float32(1.41421356)
        d[half] *= np.float32(0.5)
        x[half] *= np.float32(0.5)
    if name == "one":
        d[:] = np.float32(0.51099895)
    f8 = np.float64
    y = (1.0 / d.astype(f8)).astype(np.float32)
    q = (x * y).astype(np.float32)
    r = x.astype(f8) - q.astype(f8) * d.astype(f8)
    got = (q.astype(f8) + r * y.astype(f8)).astype(np.float32)
    np.testing.assert_array_equal(got, x / d)
