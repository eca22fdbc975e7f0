"""Several contexts in one process whose transports run the same kernels with tables of different
sizes: what adept_init sets for one of them must not take anything from another."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu

SLAB, BARREL = W.slab_calorimeter, W.barrel_calorimeter


def LAYERS(n, materials):
    mats = [W.PB, W.LAR, W.SI, W.FE][:materials]
    return W.Geometry(kind=0, n_layers=n, materials=mats, sub_materials=list(range(materials)),
                      sub_thickness=[2.0] * materials, half_xy=200.0)


# (the kernel, the larger context, the smaller one)
PAIRS = [("plain", lambda: LAYERS(40, 4), lambda: LAYERS(10, 1), {}),
         ("field", BARREL, SLAB, dict(field_T=3.8)),
         ("fused_field", BARREL, SLAB, dict(field_T=3.8, fused=1)),
         ("chords", BARREL, SLAB, dict(field_T=3.8, field_max_iterations=30, max_steps=200)),
         ("histogram", lambda: LAYERS(40, 4), SLAB, dict(flags=8))]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name,large,small,opts", PAIRS)
def test_a_smaller_context_leaves_a_larger_one_as_it_was(name, large, small, opts, precision):
    need_gpu()
    runs = {}

    def transport(which, geom, tr):
        prim = W.barrel_primaries(2, seed=5) if geom.kind else W.electrons(2, 300.0)
        prim.E[:] = 300.0
        edep, _ = tr.run(prim)
        ref = runs.setdefault(which, edep)
        # the same histories each time: only the order of a bin's sum may change
        np.testing.assert_allclose(edep, ref, rtol=0, atol=1e-11 * 300.0)

    ga, gb = large(), small()
    a = make(ga, precision=precision, tuned=False, **opts)
    transport("a", ga, a)
    b = make(gb, precision=precision, tuned=False, **opts)
    for _ in range(2):
        transport("b", gb, b)
        transport("a", ga, a)
    a.close()
    transport("b", gb, b)
    b.close()
