"""Slab distances around the test that spares the wall distances (adept_probe_distance): points
in the middle, near and on the walls, tiny coordinates and directions along an axis, against
the distances to all planes in numpy.

FP32: a wall distance is (H - x) / u from x cut to 24 bits, so it is off by at most
2^-23 H / |u| = 2.4e-5 / |u| mm and a few 2^-24 of itself; the plane distance by a few 2^-24
of itself (the truncation, the fast reciprocal)."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu

H, DEPTH = 200.0, 8.0


def points(rng, n):
    edge = np.array([0.0, 1e-300, -1e-40, 2.0 ** -126, 0.5, -197.9, 197.98, 198.0, 199.0, -199.9, 199.99999, H, -H])
    xy = np.where(rng.random((n, 2)) < 0.5, rng.uniform(-H, H, (n, 2)), rng.choice(edge, (n, 2)))
    d = rng.normal(size=(n, 3)) * np.where(rng.random((n, 1)) < 0.5, [[1.0, 1.0, 1.0]], [[1e-3, 1.0, 1e-3]])
    d[rng.random((n, 3)) < 0.1] = 0.0
    d[np.abs(d).sum(axis=1) == 0.0] = [0.0, 0.0, 1.0]
    d /= np.linalg.norm(d, axis=1)[:, None]
    return xy, d.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("prec", [0, 1])
def test_nearest_plane_or_wall(prec):
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    rng = np.random.default_rng(5)
    geom = W.slab_calorimeter()
    planes = np.concatenate([[0.0], np.cumsum(np.tile(geom.sub_thickness, geom.n_layers))])
    n = 20000
    xy, d = points(rng, n)
    vol = rng.integers(0, len(planes) - 1, n).astype(np.int32)
    z = planes[vol] + rng.uniform(0.01, 0.99, n) * (planes[vol + 1] - planes[vol])
    pos = np.concatenate([xy, z[:, None]], axis=1)
    tr = make(geom, precision=prec)
    rc, s, nxt = A.adept_probe_distance(tr.h, prec, pos, d, vol, np.full(n, 1.0), np.zeros(n, np.int32))
    tr.close()
    assert rc == 0
    with np.errstate(divide="ignore", invalid="ignore"):
        sz = np.where(d[:, 2] > 0, (planes[vol + 1] - z) / d[:, 2], np.where(d[:, 2] < 0, (planes[vol] - z) / d[:, 2], np.inf))
        sw = np.where(d[:, :2] > 0, (H - xy) / d[:, :2], np.where(d[:, :2] < 0, (-H - xy) / d[:, :2], np.inf))
    u = np.where(np.isfinite(sw), np.abs(d[:, :2]), 1.0)
    tol_z = 1e-6 * np.where(np.isfinite(sz), sz, 0.0) if prec else 1e-13 * np.where(np.isfinite(sz), sz, 0.0)
    tol_w = np.where(np.isfinite(sw), 2.4e-5 / u + 1e-6 * np.abs(np.where(np.isfinite(sw), sw, 0.0)), 0.0) if prec else 1e-13 * H / u
    ref = np.minimum(sz, sw.min(axis=1))
    tol = np.maximum(tol_z, tol_w.max(axis=1))
    finite = np.isfinite(ref)
    assert (np.abs(s - ref) <= tol)[finite].all()
    step = np.where(d[:, 2] > 0, vol + 1, vol - 1)
    up = np.where((step >= 0) & (step < len(planes) - 1), step, -1)
    clear = finite & (np.abs(sz - sw.min(axis=1)) > 2 * tol)
    np.testing.assert_array_equal(nxt[clear], np.where(sz < sw.min(axis=1), up, -1)[clear])
