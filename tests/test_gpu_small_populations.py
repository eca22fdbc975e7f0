"""Which kernels step a small population, and that they agree: the tail kernel from its first
generation (tail_tracks = 0, the default), or a launch per species and generation, or one for
all species, in chunks of a fixed length (tail_tracks < 0). The number of launches shows which
ran: two a tail chunk, and in a fixed chunk four and those of its generations."""
import numpy as np
import pytest

import oracle
from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu
from test_gpu_transport import SINGLE, compare_generations

pytestmark = pytest.mark.gpu

SLAB, BARREL = W.slab_calorimeter, W.barrel_calorimeter
SMALL = 1e-6  # tracks_per_MeV: a request counts as its primaries only


def launched(tr, before):
    """kernels per generation since `before`, the admission's two left out"""
    st = tr.stats()
    return (st.launches - before.launches - 2) / (st.generations - before.generations)


@pytest.mark.parametrize("tail", [-1, 0])
@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("name,pdg,E,mask", SINGLE)
def test_single_interactions_in_every_kernel(name, pdg, E, mask, fused, tail):
    need_gpu()
    geom = SLAB()
    tr = make(geom, precision=0, process_mask=mask, graph_generations=8, tail_tracks=tail, tracks_per_MeV=SMALL, fused=fused,
              tuned=False)
    n = 200
    prim = W.Primaries(np.full(n, pdg, np.int32), np.full(n, E), np.zeros((n, 3)), np.tile([0.0, 0.0, 1.0], (n, 1)),
                       np.arange(n, dtype=np.uint32))
    s0 = tr.stats()
    compare_generations(tr, oracle.Oracle(geom), prim, mask)
    if tail < 0:
        assert launched(tr, s0) >= (1 if fused else 3)
    tr.close()


@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
def test_small_showers_run_in_the_tail_kernel(precision, fused):
    need_gpu()
    tr = make(SLAB(), precision=precision, graph_generations=8, fused=fused, tuned=False)
    for n, E in ((1, 500.0), (2, 1000.0)):
        s0 = tr.stats()
        tr.run(W.electrons(n, E))
        assert launched(tr, s0) < 0.5  # two launches for eight generations
    tr.close()


@pytest.mark.parametrize("fused,tail", [(0, 60), (1, 60), (0, 100)])
def test_tail_chunks_below_their_bound_only(fused, tail):
    """In the tail kernel from the first track, out of it at twice the bound, in it again below
    the bound: the oracle's queue sizes in every generation, and launches of both kinds."""
    need_gpu()
    geom = SLAB()
    prim = W.mixed(5, seed=31)
    prim.E[:] = np.minimum(prim.E, 600.0)
    tr = make(geom, precision=0, graph_generations=8, fused=fused, tail_tracks=tail, tracks_per_MeV=SMALL, tuned=False)
    s0 = tr.stats()
    compare_generations(tr, oracle.Oracle(geom), prim, 0)
    fixed = (1 if fused else 3) + 4 / 8  # kernels per generation in fixed chunks of 8 alone
    assert 0.5 < launched(tr, s0) < fixed
    tr.close()


# the variants of the fused kernel, and the species kernels beside them, in a field
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name,geom_fn,opts", [("fused_field", BARREL, dict(fused=1, field_T=3.8)),
                                               ("fused_slab_field", SLAB, dict(fused=1, field_T=1.0)),
                                               ("fused_barrel", BARREL, dict(fused=1)),
                                               ("barrel_no_field", BARREL, {}),
                                               ("chords_slab", SLAB, dict(field_T=1.0, field_max_iterations=50, max_steps=300))])
def test_fused_and_field_kernels_equal_their_tail_kernel(name, geom_fn, opts, precision):
    """The same histories: only the order of a bin's sum may differ, over at most a few thousand
    terms, 1e-11 of the event's energy."""
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    geom = geom_fn()
    prim = W.barrel_primaries(8, seed=31) if geom.kind else W.mixed(8, seed=31)
    prim.E[:] = np.minimum(prim.E, 800.0)
    runs = []
    for tail in (-1, 0, 60):
        tr = make(geom, precision=precision, graph_generations=24, tail_tracks=tail, tracks_per_MeV=SMALL, tuned=False, **opts)
        s0 = tr.stats()
        edep, meta = tr.run(prim)
        per = launched(tr, s0)
        n, log = A.adept_get_generation_log(tr.h)
        log = log[: int(np.nonzero(log.sum(axis=1))[0].max()) + 1]
        runs.append((edep, log, (meta.leaked_MeV, meta.killed_MeV), list(tr.stats().steps), per))
        tr.close()
    ref = runs[0]
    assert ref[4] > 1.0 and runs[1][4] < 0.5 and runs[2][4] < ref[4]
    assert ref[1].sum(axis=1).max() > 120
    for r in runs[1:]:
        np.testing.assert_array_equal(r[1], ref[1])
        np.testing.assert_allclose(r[0], ref[0], rtol=0, atol=1e-11 * 800.0)
        np.testing.assert_allclose(r[2], ref[2], rtol=1e-11, atol=1e-11 * 800.0)
        assert r[3] == ref[3]


def test_optional_physics_has_no_tail_kernel():
    need_gpu()
    for physics in (1, 3):
        tr = make(SLAB(), precision=1, graph_generations=8, physics=physics, tuned=False)
        s0 = tr.stats()
        tr.run(W.electrons(1, 500.0))
        assert launched(tr, s0) >= 3
        tr.close()
