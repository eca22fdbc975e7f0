"""The timing flags over a transport of any size: every generation counts among the timed ones,
and the times are those of kernels that ran within the call."""
import time

import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import make, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,E", [(1, 200.0), (4, 1000.0), (40, 2000.0)])
@pytest.mark.parametrize("precision,fused,species", [(1, 0, 0), (0, 0, 0), (1, 1, 0), (0, 1, 0), (1, 0, 1), (0, 0, 1)])
def test_every_generation_is_timed(precision, fused, species, n, E):
    need_gpu()
    from paper_2209_15445_gb300 import adept as A
    flags = A.FLAG_TIME_SPECIES if species else A.FLAG_TIME_STEPS
    tr = make(W.slab_calorimeter(), precision=precision, fused=fused, flags=flags, tuned=False)
    prim = W.electrons(n, E)
    last = tr.stats()
    for _ in range(2):
        t0 = time.perf_counter()
        tr.run(prim)
        wall = 1e3 * (time.perf_counter() - t0)
        st = tr.stats()
        ran = st.generations - last.generations
        ms = st.step_kernel_ms - last.step_kernel_ms
        assert ran > 10 and st.step_launches - last.step_launches == ran
        assert 1e-3 * ran < ms < wall  # a generation takes more than a microsecond
        one = [st.species_ms[k] - last.species_ms[k] for k in range(3)]
        if species:
            assert max(one) <= ms * (1 + 1e-9) and min(one) > 0.0
        else:
            assert one == [0.0, 0.0, 0.0]
        last = st
    tr.close()
