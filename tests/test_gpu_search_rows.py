"""The two forms of the search front on rows of more than 2,048 bytes, whose kernels are short of registers."""
import numpy as np
import pytest

from paper_2307_10479_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ms(f):
    for _ in range(3):
        f()
    best = np.inf
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 5)
    return best


@pytest.mark.parametrize("dim", [520, 960])
def test_wide_rows_unsorted_front(dim):
    # the front is unsorted below eps = 0.02 and sorted from there on: the same walks, nearly, so much
    # the same time. The sorted one is up to 13% faster on long walks; the limit leaves room for another 20%.
    import paper_2307_10479_gb300 as deg
    base = synth.mixture(8_000, synth.mixture_centres(40, dim, 7), 0.4, 1)
    idx = deg.Index.build_device(base, 20, 40, 0.2, batch_div=64)
    idx.upload()
    q = torch.from_numpy(synth.mixture(3_000, synth.mixture_centres(40, dim, 7), 0.4, 2)).cuda()
    how = dict(k=10, entry="pivot", with_trace=True)
    ids, _, trace = idx.search(q, eps=0.0199, **how)
    ids2, _, trace2 = idx.search(q, eps=0.0201, **how)
    assert (ids == ids2).float().mean() > 0.99
    assert trace2[:, 0].float().mean() < 1.1 * trace[:, 0].float().mean()
    assert _ms(lambda: idx.search(q, eps=0.0199, **how)) < 1.35 * _ms(lambda: idx.search(q, eps=0.0201, **how))
