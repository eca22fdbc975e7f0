"""The tail kernel (the generations of a small population in one launch) against the chunks of
one launch per species and generation, for every variant of the step and both forms: the same
events with tail chunks off (tail_tracks < 0) and on give the same queue sizes in every
generation and the same deposits. The histories are the same, so deposits differ only by the
order of their sums: at most a few thousand terms a bin, 1e-11 of the event's energy."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu

SLAB, BARREL = W.slab_calorimeter, W.barrel_calorimeter


def EIGHT():
    """eight materials: in FP64 their tables do not fit a block's shared memory beside its rings"""
    mats = [W.PB, W.LAR, W.SI, W.FE, W.PBWO4, W.PB, W.FE, W.SI]
    return W.Geometry(kind=0, n_layers=12, materials=mats, sub_materials=list(range(8)),
                      sub_thickness=[2.0, 3.0, 0.3, 2.0, 2.0, 1.0, 1.0, 4.0], half_xy=200.0)


VARIANTS = [("plain", SLAB, {}), ("field", SLAB, dict(field_T=1.0)), ("barrel", BARREL, dict(field_T=3.8)),
            ("msc", SLAB, dict(physics=1)), ("msc_fluct_field", BARREL, dict(physics=3, field_T=3.8)),
            ("chords", BARREL, dict(field_T=3.8, field_max_iterations=100, max_steps=300)),
            ("chords_msc", BARREL, dict(field_T=3.8, field_max_iterations=50, physics=1, max_steps=300)),
            ("histogram", SLAB, dict(flags=8)), ("histogram_field", BARREL, dict(flags=8, field_T=3.8)),
            ("fused", SLAB, dict(fused=1)), ("eight_materials", EIGHT, {})]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name,geom_fn,opts", VARIANTS)
def test_tail_kernel_equals_fixed_chunks(name, geom_fn, opts, precision):
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    geom = geom_fn()
    prim = W.barrel_primaries(5, seed=31) if geom.kind else W.mixed(5, seed=31)
    prim.E[:] = np.minimum(prim.E, 600.0)
    runs = []
    # off; on from the first track; on with its end inside the shower (it ends at 120 tracks)
    for tail in (-1, 0, 60):
        tr = make(geom, precision=precision, graph_generations=24, tail_tracks=tail, tracks_per_MeV=1e-6, tuned=False, **opts)
        edep, meta = tr.run(prim)
        n, log = A.adept_get_generation_log(tr.h)
        log = log[: int(np.nonzero(log.sum(axis=1))[0].max()) + 1]
        runs.append((edep, log, (meta.leaked_MeV, meta.killed_MeV), list(tr.stats().steps), list(tr.stats().secondaries),
                     A.adept_get_step_histogram(tr.h)[1]))
        tr.close()
    ref = runs[0]
    assert ref[1].sum(axis=1).max() > 200
    for r in runs[1:]:
        np.testing.assert_array_equal(r[1], ref[1])
        np.testing.assert_allclose(r[0], ref[0], rtol=0, atol=1e-11 * 600.0)
        np.testing.assert_allclose(r[2], ref[2], rtol=1e-11, atol=1e-11 * 600.0)
        assert r[3] == ref[3] and r[4] == ref[4]
        np.testing.assert_array_equal(r[5], ref[5])
