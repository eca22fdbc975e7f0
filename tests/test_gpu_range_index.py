"""The indexed inversion of the range table (adept_probe_inverse_range) over every interval of
the table, at the nodes and past both ends, against a search of the node row itself.

An entry that is one interval off shows at the interval's middle: the range rises by 7 % or
more from node to node, so a neighbour's line, continued over half an interval, is off by
the change of slope, well above the tolerances. FP64: the difference r - a of nodes 7 % apart
loses four bits, so t is good to about 16 eps and E to 16 eps x 0.07; 1e-12 covers exp's own
argument (14 eps). FP32: lo + t is rounded at up to 288 (1.5e-5 x 0.072 = 1.1e-6), the
argument of exp at up to 14 (5e-7), t by 16 eps x 0.072 (7e-8), and the fast exp adds about
2e-6: 1e-5."""
import numpy as np
import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu

LN_EMIN, DLOG = np.log(1e-3), np.log(10.0) / 32.0
GAS = W.Material("Ar gas", 18, 39.948, 1.66e-3, 188.0)


@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)])
def test_every_interval_and_both_ends(prec, tol):
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    geom = W.Geometry(kind=0, n_layers=2, materials=[W.PB, W.SI, GAS, W.PBWO4], sub_materials=[0, 1, 2, 3],
                      sub_thickness=[1.0, 1.0, 1.0, 1.0], half_xy=10.0)
    tr = make(geom, precision=prec)
    for m in range(4):
        for s in (1, 2):
            rc, nodes = A.adept_get_table(tr.h, s, 1, m, prec)
            assert rc == 0
            a, b = nodes[:-1], nodes[1:]
            r = np.concatenate([a, a + 0.25 * (b - a), a + 0.5 * (b - a), a + 0.75 * (b - a), nodes * (1 + 1e-6),
                                nodes * (1 - 1e-6)])
            if prec:
                r = r.astype(np.float32).astype(np.float64)
            ends = np.array([0.0, 0.5 * nodes[0], nodes[-1], 1.5 * nodes[-1], 1e30])
            r = r[(r >= nodes[0]) & (r < nodes[-1])]
            lo = np.searchsorted(nodes, r, side="right") - 1
            E = np.exp(LN_EMIN + (lo + (r - nodes[lo]) / (nodes[lo + 1] - nodes[lo])) * DLOG)
            rc, got = A.adept_probe_inverse_range(tr.h, s, m, prec, r)
            assert rc == 0
            np.testing.assert_allclose(got, E, rtol=tol, atol=0)
            rc, got = A.adept_probe_inverse_range(tr.h, s, m, prec, ends)
            assert rc == 0
            np.testing.assert_array_equal(got, [0.0, 0.0, 1e6, 1e6, 1e6])
    tr.close()
