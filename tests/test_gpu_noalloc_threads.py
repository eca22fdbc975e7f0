"""adept_build_tables_noalloc called from two host threads on one stream: the stream runs the
calls one after the other, so each must leave what it leaves alone, whichever way the threads'
launches fall."""
import threading

import pytest

from paper_2209_15445_gb300 import workloads as W

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def test_two_threads_on_one_stream_get_their_own_tables():
    torch = need_gpu()
    from paper_2209_15445_gb300 import adept as A
    sets = [[W.PB, W.LAR], [W.FE, W.SI]]
    calls = 1000
    stream = torch.cuda.Stream()

    def buffers(n):
        f8 = dict(dtype=torch.float64, device="cuda")
        return torch.zeros((n, 2, 12, A.NNODE), **f8), torch.zeros((n, 2, 2), **f8)

    def build(k, out, cuts, i):
        return A.adept_build_tables_noalloc(sets[k], 0.7, out[i].data_ptr(), cuts[i].data_ptr(), stream.cuda_stream)

    alone = [buffers(1) for _ in sets]
    got = [buffers(calls) for _ in sets]
    torch.cuda.synchronize()
    for k in range(2):
        assert build(k, *alone[k], 0) == A.OK
    stream.synchronize()
    start = threading.Barrier(2)
    rc = [[], []]

    def work(k):
        start.wait()
        for i in range(calls):
            rc[k].append(build(k, *got[k], i))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for k in range(2):
        assert rc[k] == [A.OK] * calls
        for a, b in zip(alone[k], got[k]):
            wrong = (b != a).flatten(1).any(1).sum().item()
            assert wrong == 0, f"{wrong} of {calls} calls of thread {k}"
