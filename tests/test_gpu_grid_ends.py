"""Table lookups at and past the ends of the energy grid, and at energies that are not finite: the
first and the last interval's line carried on (FP64)."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu

NTAB = [(0, 3), (1, 4), (2, 5)]


def test_lookup_past_the_grid():
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    tr = make(W.slab_calorimeter(), precision=0, arena_bytes=256 << 20)
    n = A.NNODE
    lo, step = np.log(1e-3), np.log(10.0) / 32
    E = np.array([0.0, np.inf, 5e-324, 1e-300, 1e-9, 0.9e-3, 0.9999e-3, 1.0001e6, 1.1e6, 1e9, 1e300, -1.0, np.nan])
    with np.errstate(all="ignore"):
        x = (np.log(E) - lo) / step
    k = np.where(x < 1.0, 0, n - 2)
    for s, nt in NTAB:
        for t in range(nt):
            rc, v = A.adept_get_table(tr.h, s, t, 0, 0)
            assert rc == A.OK
            with np.errstate(all="ignore"):
                slope = v[k + 1] - v[k]
                want = v[k] + slope * (x - k)
            rc, got = A.adept_probe_interp(tr.h, s, t, 0, 0, E)
            assert rc == A.OK
            # (the line's sum loses at most a few units in the last place of its larger term)
            scale = np.abs(v[k]) + np.abs(slope) * np.where(np.isfinite(x), np.abs(x - k), 0.0)
            fin = np.isfinite(want)
            assert (np.abs(got[fin] - want[fin]) <= 1e-12 * scale[fin]).all(), (s, t, got, want)
            np.testing.assert_array_equal(got[~fin], want[~fin])  # infinities by their sign, and NaN
    tr.close()
