"""Two host threads that search two indexes at the same time. A kernel's
shared-memory limit is one setting for the whole process, so the launches of one index must not
depend on what the other one asked for."""
import ctypes
import threading

import numpy as np
import pytest

from paper_2307_10479_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _index(n, dim, seed):
    import paper_2307_10479_gb300 as deg
    i = np.arange(n, dtype=np.int32)[:, None]
    adj = ((i + np.array([-37, -2, 2, 37], np.int32)) % n).astype(np.int32)
    idx = deg.Index.from_arrays(synth.uniform(n, dim, seed), adj)
    idx.upload()
    return idx


@pytest.mark.parametrize("sizes,nq,ks,times", [
    ((600_000, 2_000), 2, (10, 10), 20_000),     # a block per query: the bitmap of C follows n
    ((2_000, 3_000), 700, (1_000, 1), 2_000),    # a warp per query: the result list follows k
])
def test_two_threads_two_indexes(sizes, nq, ks, times):
    import paper_2307_10479_gb300 as deg
    made = [_index(n, 16, s) for s, n in enumerate(sizes)]
    queries = [torch.from_numpy(synth.uniform(nq, 16, 10 + s)).cuda() for s in range(2)]
    want = [i.search(q, k=k, eps=0.0, max_hops=2) for i, q, k in zip(made, queries, ks)]
    got = [[torch.empty_like(t) for t in w] for w in want]
    torch.cuda.synchronize()
    failed, start = [], threading.Barrier(2)

    def work(t):
        try:
            # the call itself, with everything made beforehand: little time outside it
            params = deg.SearchParams(ks[t], 0.0, 0, 0, 2, 0, 0, 0, 0)
            args = (made[t]._h, ctypes.byref(params), queries[t].data_ptr(), None, 0, nq, got[t][0].data_ptr(),
                    got[t][1].data_ptr(), None, None, None)
            call = deg.lib().deg_search_ex
            start.wait()
            bad = sum(call(*args) != deg.DEG_OK for _ in range(times))
            torch.cuda.synchronize()
            assert bad == 0, f"{bad} of {times} searches refused"
            for g, w in zip(got[t], want[t]):
                assert torch.equal(g, w)
        except BaseException as e:                  # shown by the main thread
            failed.append(f"thread {t}: {e!r}")

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
