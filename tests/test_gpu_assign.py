"""The tensor-core assignment of many rows to a few (k-means, locality layout) against plain NumPy k-means
on integer rows, where every float32 distance and cluster sum is exact."""
import numpy as np
import pytest

from paper_2307_10479_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ring(n):
    i = np.arange(n, dtype=np.int32)[:, None]
    return ((i + np.array([-2, -1, 1, 2], np.int32)) % n).astype(np.int32)


def _assign(x, c):
    """Labels and squared distances in float32, summed in dimension order, ties to the lower index."""
    t = torch.from_numpy(x).cuda()
    labels, best = [], []
    for lo in range(0, len(x), 2_048):
        d2 = torch.zeros((min(2_048, len(x) - lo), len(c)), dtype=torch.float64, device="cuda")
        cc = torch.from_numpy(c).cuda().double()
        for d in range(x.shape[1]):
            diff = (t[lo:lo + 2_048, d].double()[:, None] - cc[:, d][None]).float().double()   # fl(x - c)
            d2 = (d2 + diff * diff).float().double()                                           # one rounding: an FMA
        labels.append(d2.argmin(1).cpu().numpy())
    return np.concatenate(labels)


@pytest.mark.parametrize("n,dim,k,kind", [
    (9_000, 32, 512, "u8"),         # the tensor cores
    (4_097, 20, 1_030, "u8"),       # a last tile of six; one row past a chunk of 128
    (6_000, 132, 700, "far"),       # values past float16: the CUDA cores
    (5_000, 64, 3, "u8"),           # too few for the tensor cores
    (8_000, 16, 1_024, "ties"),     # rows repeated: many candidates with one distance
])
def test_train_entry_equals_plain_k_means(n, dim, k, kind):
    import paper_2307_10479_gb300 as deg
    x = synth.mixture_u8(n, synth.mixture_u8_centres(20, dim, 3), 25.0, 4)
    if kind == "far":
        x[::7] += 70_000.0
    if kind == "ties":
        x = np.repeat(x[:n // 100], 100, axis=0)
    idx = deg.Index.from_arrays(x, _ring(n))
    idx.upload()
    iters = 3
    sizes = idx.train_entry(k, iters)
    # the library numbers rows by its locality layout: read it back through the sampled pivots' labels
    np_ = min(4096, max(1, n // 256))
    pivots = np.arange(np_) * (n // np_)
    lab = _assign(x, x[pivots])
    order = np.argsort(lab, kind="stable")                      # internal order: by label, then id
    y = x[order]
    c = y[np.arange(k) * (n // k)].copy()
    for it in range(iters + 1):
        lab = _assign(y, c)
        if it == iters:
            break
        for j in range(k):
            m = lab == j
            if m.any():
                c[j] = y[m].sum(0, dtype=np.float32) / np.float32(m.sum())
    assert np.array_equal(sizes, np.bincount(lab, minlength=k))
