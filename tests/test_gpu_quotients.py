"""The split form's quotients by one number and its chord directions, as the device computes
them, bit for bit against the divisions and the square root they stand for: the reciprocal they
start from is the hardware's, whose error only the device can show."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    need_gpu()
    tr = make(W.slab_calorimeter(), precision=1, arena_bytes=256 << 20)
    yield tr
    tr.close()


def significands(rng, n):
    return (rng.integers(0, 1 << 23, n).astype(np.uint32) | np.uint32(127 << 23)).view(np.float32)


def same_quotients(ctx, d, x):
    from paper_2209_15445_gb300 import adept as A
    rc, got, ref = A.adept_probe_quotient(ctx.h, d, x)
    assert rc == A.OK
    np.testing.assert_array_equal(ref, x / d)  # numpy's division rounds correctly too
    bad = np.nonzero(got.view(np.uint32) != ref.view(np.uint32))[0]
    assert len(bad) == 0, (len(bad), d[bad[:5]], x[bad[:5]], got[bad[:5]], ref[bad[:5]])


# every significand of the divisor, at the ends and in the middle of the stated range of divisors,
# with quotients up to its ends (the residual x - q d needs x above 2^-100 to be exact)
@pytest.mark.parametrize("exponent", [-100, -37, -1, 0, 1, 50, 99])
def test_every_divisor_significand(ctx, exponent):
    rng = np.random.default_rng(100 + exponent)
    d = np.ldexp((np.arange(1 << 23, dtype=np.uint32) | np.uint32(127 << 23)).view(np.float32), exponent)
    assert d.dtype == np.float32
    lo, hi = max(-100, exponent - 100), min(100, exponent + 100)
    x = np.ldexp(significands(rng, len(d)), rng.integers(lo, hi, len(d))).astype(np.float32)
    x *= rng.choice(np.float32([-1.0, 1.0]), len(d))
    same_quotients(ctx, d, x)
    # quotients next to a number and next to the middle of two: x = q d and (q + half an ulp) d, rounded
    q = significands(rng, len(d)).astype(np.float64)
    e = rng.integers(lo, hi - 1, len(d)) - exponent
    for half in (0.0, 2.0 ** -24):
        x = np.ldexp((q + half) * d.astype(np.float64), e).astype(np.float32)
        same_quotients(ctx, d, x)


def test_the_transport_s_quotients(ctx):
    rng = np.random.default_rng(5)
    n = 1 << 22
    m = (rng.integers(0, 1 << 23, n).astype(np.uint32) | np.uint32(127 << 23)).view(np.float32)
    low = (rng.integers(0, 1 << 29, n).astype(np.float32) * np.float32(2.0 ** -52)).astype(np.float32)
    half = m > np.float32(1.41421356)
    m[half] *= np.float32(0.5)
    low[half] *= np.float32(0.5)
    same_quotients(ctx, m, low)  # the energy grid's position
    x = np.ldexp(significands(rng, n), rng.integers(-10, 21, n)).astype(np.float32)
    same_quotients(ctx, np.full(n, 0.51099895, np.float32), x)  # a photon's energy over the electron's mass
    zeros = np.zeros(1 << 10, np.float32)
    same_quotients(ctx, significands(rng, 1 << 10), zeros)


def test_chord_directions(ctx):
    from paper_2209_15445_gb300 import adept as A
    rng = np.random.default_rng(6)

    def check(v):
        rc, got, ref = A.adept_probe_chord_direction(ctx.h, v)
        assert rc == A.OK
        bad = np.nonzero((got.view(np.uint64) != ref.view(np.uint64)).any(axis=1))[0]
        assert len(bad) == 0, (len(bad), v[bad[:3]], got[bad[:3]], ref[bad[:3]])
        return ref

    for scale in (1e-14, 1e-3, 1.0, 1e3, 1e14):
        check(rng.normal(size=(1 << 19, 3)) * 2.0 ** rng.integers(-20, 1, (1 << 19, 3)) * scale)
    # lengths within forty units in the last place of a cut, along an axis and off it: vectors
    # whose length is a whole multiple of a component's
    f = np.ldexp(significands(rng, 1 << 16).astype(np.float64), rng.integers(-20, 20, 1 << 16))
    for k in range(-40, 41):
        g = (f.view(np.int64) + k).view(np.float64)
        for a in ((1.0, 0.0, 0.0), (0.0, 0.0, -1.0), (2.0, -3.0, 6.0), (0.0, 3.0, 4.0)):
            check(g[:2048, None] * np.array(a) / (7.0 if a[0] == 2.0 else 5.0 if a[1] == 3.0 else 1.0))
    # components that are zero (of either sign), that the cut flushes, and lengths past the fast form's range
    edge = np.array([[0.0, 0.0, 0.0], [-0.0, 0.0, 1.0], [1e-200, 1.0, -0.0], [1e-39, 2.0, 1.0], [1e-320, 0.0, 3.0],
                     [1e-15, 0.0, 0.0], [1.1e-15, 0.0, 0.0], [1e15, 0.0, 0.0], [0.9e15, 1.0, 0.0], [1e-170, 0.0, 0.0],
                     [1e20, 1e20, 1e20], [1e-20, -1e-20, 1e-20]])
    ref = check(edge)
    assert (ref[0] == 0.0).all() and ref[1, 3] == 1.0
