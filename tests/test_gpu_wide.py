"""The block-per-query kernel of small batches against the warp-per-query kernel of large ones: the same
ids, distances, status and trace (hops, evaluations, peak of S) for the same queries, in every form
the small batches accept."""
import numpy as np
import pytest

from paper_2307_10479_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NQ = 2_000                       # above any small batch


def _circulant(n, degree, seed):
    """A permuted circulant graph: valid, and as good as random (long walks, large S)."""
    rng = np.random.default_rng(seed)
    p = rng.permutation(n).astype(np.int64)
    steps = rng.choice(np.arange(1, (n - 1) // 2), degree // 2, replace=False)
    steps = np.concatenate([steps, -steps])
    adj = np.empty((n, degree), np.int32)
    adj[p] = p[(np.arange(n)[:, None] + steps) % n]
    return adj


_made = {}


def _index(n, dim, degree, graph, precisions=("f32", "bf16", "fp8")):
    import paper_2307_10479_gb300 as deg
    key = (n, dim, degree, graph)
    if key not in _made:
        base = synth.mixture(n, synth.mixture_centres(40, dim, 7), 0.4, 1)
        if graph == "built":
            idx = deg.Index.build_device(base, degree, 2 * degree, 0.2, batch_div=64)
        else:
            idx = deg.Index.from_arrays(base, _circulant(n, degree, 3))
        idx.upload(precisions)
        if dim % 4 == 0:
            idx.train_entry(max(1, n // 256), 3)
        _made.clear()
        _made[key] = idx, torch.from_numpy(synth.mixture(NQ, synth.mixture_centres(40, dim, 7), 0.4, 2)).cuda()
    return _made[key]


def _compare(idx, q, sizes, **how):
    explore = how.get("explore", False)
    seeds = torch.from_numpy(synth.distinct_ids(idx.info()[0], NQ, 5)).cuda() if explore else how.pop("seeds", None)

    def run(sl):
        if explore:
            return idx.search(seeds=seeds[sl], with_status=True, with_trace=True, **how)
        s = None if seeds is None else seeds[sl]
        return idx.search(q[sl].contiguous(), seeds=s, with_status=True, with_trace=True, **how)

    want = run(slice(0, NQ))
    at = 0
    for size in sizes:
        got = run(slice(at, at + size))
        for g, w in zip(got, want):
            assert torch.equal(g.view(torch.int32), w[at:at + size].view(torch.int32)), (size, how)   # bits: NaN too
        at += size


@pytest.mark.parametrize("n,dim,degree,graph", [
    (6_000, 48, 16, "built"),
    (5_000, 100, 30, "built"),
    (3_000, 130, 8, "circulant"),     # not a multiple of any chunk; one more than 128
    (2_500, 24, 64, "circulant"),     # more than one word of neighbours
    (2_200, 520, 128, "circulant"),   # two chunks a lane, the largest degree
])
def test_small_batches_equal_large_ones(n, dim, degree, graph):
    idx, q = _index(n, dim, degree, graph)
    sizes = (1, 64, 65, 2, 150)
    for precision, rerank in (("f32", 0), ("bf16", 32), ("fp8", 32), ("fp8", -1)):
        for k, eps in ((1, 0.0), (10, 0.05), (32, 0.2)):
            if rerank > 0 and k > rerank:
                continue
            for entry in ("fixed", "pivot") + (("learned",) if dim % 4 == 0 else ()):
                _compare(idx, q, sizes, k=k, eps=eps, precision=precision, rerank=rerank, entry=entry)
    _compare(idx, q, sizes, k=100, eps=0.1, explore=True)
    _compare(idx, q, sizes, k=128, eps=0.0, explore=True, precision="bf16", rerank=128)
    _compare(idx, q, sizes, k=129, eps=0.0)                         # above what a block keeps
    for hops in (1, 7):
        _compare(idx, q, sizes, k=10, eps=0.3, max_hops=hops)


def test_every_vertex_is_checked():
    # a huge eps: S outgrows the front many times over and refills until the graph is exhausted
    idx, q = _index(4_000, 32, 12, "circulant")
    _compare(idx, q, (3, 70), k=20, eps=50.0)


def test_seeds_and_refused_queries():
    idx, q = _index(4_000, 32, 12, "circulant")
    seeds = torch.from_numpy(synth.distinct_ids(4_000, NQ, 9)).cuda()
    seeds[1], seeds[40], seeds[67] = -1, 4_000, 2**31 - 1
    _compare(idx, q, (2, 64, 80), k=5, eps=0.1, seeds=seeds)
    bad = q.clone()
    bad[0, 3], bad[5, 0], bad[66, 31] = float("nan"), float("inf"), -float("inf")
    for entry in ("pivot", "learned", "fixed"):
        _compare(idx, bad, (3, 60, 100), k=5, eps=0.1, entry=entry)


def test_equal_rows_order_by_id():
    import paper_2307_10479_gb300 as deg
    base = np.repeat(synth.uniform(400, 16, 1), 5, axis=0)          # every row five times
    idx = deg.Index.from_arrays(base, _circulant(2_000, 10, 4))
    idx.upload(("f32", "fp8"))
    q = torch.from_numpy(base[:NQ].copy()).cuda()                   # distance zero at several ids
    _compare(idx, q, (1, 64, 100), k=7, eps=0.2)
    _compare(idx, q, (1, 64, 100), k=1, eps=0.0)
    _compare(idx, q, (1, 64, 100), k=7, eps=0.1, precision="fp8", rerank=16)


POOL = 32_768                    # keys of S in device memory before a query moves to a second pass


def _two_clusters(far, near, degree, dim):
    """`far` vertices around the point 10 away and `near` ones around the origin, a circulant graph each, joined by
    one swapped pair of edges at a far vertex that is popped after 2,500 others: the walk fills S with far vertices,
    and those fall out of the radius once it has crossed."""
    rng = np.random.default_rng(1)
    x = (rng.random((far + near, dim)) - 0.5).astype(np.float32)
    x[:far] += np.float32(10 / np.sqrt(dim))
    adj = np.concatenate([_circulant(far, degree, 3), _circulant(near, degree, 4) + far]).astype(np.int32)
    a, b = int(np.argsort((x[:far] ** 2).sum(1))[2_500]), far
    a2, b2 = adj[a, 0], adj[b, 0]
    for u, old, new in ((a, a2, b), (b, b2, a), (a2, a, b2), (b2, b, a2)):
        adj[u, np.flatnonzero(adj[u] == old)[0]] = new
    return x, adj


@pytest.mark.parametrize("nq", [3, 64, 70])
@pytest.mark.parametrize("graph,k,eps,tier", [
    ("two clusters", 100, 0.6, 0),   # the pool fills, and has room again without the far vertices
    ("circulant", 20, 50.0, 1),      # the pool fills, and every key in it is still within the radius
])
def test_full_pools(graph, k, eps, tier, nq):
    # queue_cap keeps a batch on the warp-per-query kernel, here with the same pool of 32,768 keys
    import paper_2307_10479_gb300 as deg
    if graph not in _made:
        if graph == "circulant":
            x, adj = synth.uniform(50_000, 8, 1), _circulant(50_000, 32, 3)
        else:
            x, adj = _two_clusters(31_000, 60_000, 64, 8)
        _made.clear()
        _made[graph] = deg.Index.from_arrays(x, adj)
        _made[graph].upload()
    rng = np.random.default_rng(2)
    q = torch.from_numpy((rng.random((nq, 8)) * 1e-3).astype(np.float32)).cuda()
    seeds = torch.from_numpy(rng.integers(0, 31_000, nq).astype(np.int32)).cuda()
    how = dict(k=k, eps=eps, seeds=seeds, with_status=True, with_trace=True)
    want = _made[graph].search(q, queue_cap=POOL, **how)
    got = _made[graph].search(q, **how)
    for g, w in zip(got[:3], want[:3]):
        assert torch.equal(g.view(torch.int32), w.view(torch.int32))
    assert torch.equal(got[3][:, :2], want[3][:, :2])
    assert (want[3][:, 3] == tier).all() and torch.equal(got[3][:, 3], want[3][:, 3])
    assert (want[3][:, 2] > POOL).all() and (got[3][:, 2] > POOL).all()
    if tier:
        assert torch.equal(got[3][:, 2], want[3][:, 2])     # no key was dropped from either pool
