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


@pytest.mark.parametrize("charge,tol", [(0, 1e-11), (-1, 1e-9)])
def test_tubes_near_and_far_from_the_end_caps(charge, tol):
    """FP64 tube distances, straight and along a helix, around the test that spares the distance
    to the end caps, against the oracle (tolerances of the other tube distances)."""
    need_gpu()
    import oracle
    from paper_2209_15445_gb300 import adept as A
    rng = np.random.default_rng(6)
    geom = W.barrel_calorimeter()
    orc = oracle.Oracle(geom, field_T=3.8)
    n = 4000
    r, phi = rng.uniform(10.0, 1790.0, n), rng.uniform(0.0, 2 * np.pi, n)
    cap = 3000.0 - rng.choice([1e-9, 0.01, 1.0, 2.0, 2.3, 2.4, 50.0, 1000.0], n)
    z = np.where(rng.random(n) < 0.5, cap, -cap)
    c = np.where(rng.random(n) < 0.3, rng.choice([0.0, 1.0, -1.0, 0.9999], n), rng.uniform(-1.0, 1.0, n))
    f = rng.uniform(0.0, 2 * np.pi, n)
    s = np.sqrt(1.0 - c * c)
    pos = np.stack([r * np.cos(phi), r * np.sin(phi), z], 1)
    d = np.stack([s * np.cos(f), s * np.sin(f), c], 1)
    vol = np.array([orc.locate(p, u) for p, u in zip(pos, d)], np.int32)
    T = np.exp(rng.uniform(np.log(0.05), np.log(5e3), n))
    q = np.full(n, charge, np.int32)
    tr = make(geom, precision=0, field_T=3.8)
    rc, got, nxt = A.adept_probe_distance(tr.h, 0, pos, d, vol, T, q)
    tr.close()
    assert rc == 0
    ref = [orc.helix_distance(t, charge, p, u, v) if charge else orc.distance(p, u, v) for p, u, v, t in zip(pos, d, vol, T)]
    rs, rn = np.array([x[0] for x in ref]), np.array([x[1] for x in ref])
    agree = np.abs(got - rs) <= tol * np.maximum(1.0, rs)
    assert agree.mean() > 0.999
    np.testing.assert_array_equal(nxt[agree], rn[agree])
