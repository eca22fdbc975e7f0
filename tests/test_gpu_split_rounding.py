"""The split form's FP64 -> FP32 conversion and back, bit for bit, through the one probe whose
result is a bare conversion: in a slab a track at height z heading straight down (direction
-z) is z above plane 0, and the FP32 distance is the FP64 difference with its significand cut
to 24 bits: smaller than the smallest normal float gives 0, and past the float range the
walls' 1e30 stands in."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu


def truncate(x):
    b = np.asarray(x, np.float64).view(np.uint64) & np.uint64(0xFFFFFFFFE0000000)
    y = b.view(np.float64).copy()
    y[y < 2.0 ** -126] = 0.0
    y[y > 1e30] = np.float64(np.float32(1e30))
    return y


def test_distance_is_the_truncated_height():
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    rng = np.random.default_rng(8)
    edge = 2.0 ** -126
    z = np.concatenate([
        np.ldexp(rng.uniform(1.0, 2.0, 4000), rng.integers(-140, 99, 4000)),
        2.0 ** np.arange(-1022.0, 99.0),
        np.nextafter(2.0 ** np.arange(-130.0, 99.0), 0.0),
        [0.0, 5e-324, 1e-300, edge, np.nextafter(edge, 0.0), np.nextafter(edge, 1.0), 1e38, 3.5e38, 1e39, 1e300]])
    n = len(z)
    pos, d = np.zeros((n, 3)), np.zeros((n, 3))
    pos[:, 2], d[:, 2] = z, -1.0
    tr = make(W.slab_calorimeter(), precision=1)
    rc, s, nxt = A.adept_probe_distance(tr.h, 1, pos, d, np.zeros(n, np.int32), np.full(n, 1.0), np.zeros(n, np.int32))
    tr.close()
    assert rc == 0
    np.testing.assert_array_equal(s, truncate(z))
    assert (nxt == -1).all()
