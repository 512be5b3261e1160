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


def _k_means(x, k, iters):
    """(sizes, learned points as caller ids) of plain k-means from the library's start, over its locality layout."""
    n = len(x)
    np_ = min(4096, max(1, n // 256))
    order = np.argsort(_assign(x, x[np.arange(np_) * (n // np_)]), kind="stable")
    y = x[order]
    c = y[np.arange(k) * (n // k)].copy()
    for it in range(iters + 1):
        lab = _assign(y, c)
        if it < iters:
            for j in np.unique(lab):
                m = lab == j
                c[j] = y[m].sum(0, dtype=np.float32) / np.float32(m.sum())
    return np.bincount(lab, minlength=k), order[_assign(c, y)]


@pytest.mark.parametrize("n,dim,k,step", [
    (20_000, 32, 512, 1),       # far from the origin: every row's candidates outgrow its list
    (20_000, 32, 512, 3),       # every third row only
    (150_000, 8, 1_000, 10),    # more than one chunk of 131,072 rows, some of them far
    (150_000, 12, 300, 200),    # and a few
])
def test_rows_whose_candidates_outgrow_their_list(n, dim, k, step):
    import paper_2307_10479_gb300 as deg
    x = synth.mixture_u8(n, synth.mixture_u8_centres(20, dim, 3), 25.0, 4)
    x[::step] += 3_000.0        # float16 holds the values; the rounding window spans all the centroids
    idx = deg.Index.from_arrays(x, _ring(n))
    idx.upload()
    sizes = idx.train_entry(k, 2)
    want, points = _k_means(x, k, 2)
    assert np.array_equal(sizes, want)
    assert np.array_equal(idx.pivots(learned=True), points)


def test_far_rows_cost_what_the_cuda_cores_cost():
    # the same rows times 100 lie outside float16 and go to the CUDA cores at once
    import time

    import paper_2307_10479_gb300 as deg
    x = synth.mixture(100_000, synth.mixture_centres(100, 64, 3), 0.3, 4) + np.float32(1_000.0)
    took = []
    for scale in (100.0, 1.0):
        idx = deg.Index.from_arrays(x * np.float32(scale), _ring(len(x)))
        idx.upload()
        idx.train_entry(512, 5)
        best = np.inf
        for _ in range(3):
            t = time.perf_counter()
            idx.train_entry(512, 5)
            best = min(best, time.perf_counter() - t)
        took.append(best)
    assert took[1] < 2 * took[0]
