"""knn_exact's tensor-core filter in both 16-bit formats and over its list sizes: bit-identical to the
CUDA-core path (knn_exact_noalloc), whichever format the inputs lead to."""
import numpy as np
import pytest

from paper_2307_10479_gb300 import synth
from test_gpu_knn import _both

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _same(base, q, k):
    t_ids, t_d, s_ids, s_d = _both(base, q, k)
    assert np.array_equal(t_ids, s_ids)
    assert np.array_equal(t_d.view(np.uint32), s_d.view(np.uint32))


@pytest.mark.parametrize("scale,offset", [
    (1.0, 0.0),       # float16 copies
    (3e4, 0.0),       # values above 65504 among them: float16 cannot hold the rows
    (1e-7, 0.0),      # below float16's normal range: bfloat16 rounds better
    (1e-4, 0.0),      # straddles the edge of float16's normal range
    (0.3, 300.0),     # far from the origin: the rounding terms dominate the window
])
@pytest.mark.parametrize("n,dim,nq,k", [(20_000, 96, 150, 10), (3_001, 33, 65, 7)])
def test_formats_on_mixture_rows(scale, offset, n, dim, nq, k):
    c = synth.mixture_centres(50, dim, 7)
    base = synth.mixture(n, c, 0.3, 1) * np.float32(scale) + np.float32(offset)
    q = synth.mixture(nq, c, 0.3, 2) * np.float32(scale) + np.float32(offset)
    _same(base, q, k)


def test_one_query_outside_float16_moves_all_to_bfloat16():
    base = synth.uniform(9_000, 64, 1)
    q = synth.uniform(140, 64, 2)
    q[77, 5] = 1e6
    _same(base, q, 10)


def test_high_dimensional_mixture():
    # 60,000 x 960: with bfloat16 copies these queries overflowed their candidate lists
    c = synth.mixture_centres(30, 960, 7)
    _same(synth.mixture(60_000, c, 0.3, 1), synth.mixture(130, c, 0.3, 2), 10)


@pytest.mark.parametrize("n,dim,nq,k", [
    (1_024, 16, 9, 1),        # groups of 64 (16 of them), the block's last queries missing
    (1_023, 16, 8, 2),        # too few for groups of 64: 64 groups of 16
    (16_400, 20, 130, 32),    # 1,025 groups: one above what a warp selects among
    (65_536, 12, 20, 10),     # 1,024 groups of 64, every row sampled
    (65_537, 12, 129, 200),   # every second row sampled, 2,049 groups of 16
    (40_000, 48, 3, 256),     # lists longer than a warp scores at once
])
def test_sample_groups_and_list_sizes(n, dim, nq, k):
    _same(synth.uniform(n, dim, 31), synth.uniform(nq, dim, 32), k)


@pytest.mark.parametrize("n,dim,nq,k", [
    (1_300, 24, 5, 257),          # fewer groups than k, all rows in one list
    (8_192, 16, 3, 1_024),        # as many rows as the longest list holds
    (8_193, 16, 3, 1_024),        # one more: the CUDA-core path
    (16_384, 16, 20, 1_024),      # exactly k groups
    (70_000, 40, 130, 1_000),     # every second row sampled
    (300_000, 16, 3, 1_001),      # every fourth
])
def test_long_lists(n, dim, nq, k):
    _same(synth.uniform(n, dim, 33), synth.uniform(nq, dim, 34), k)


@pytest.mark.parametrize("k", [10, 300])
def test_undefined_and_infinite_rows_and_queries(k):
    base, q = synth.uniform(5_000, 32, 35), synth.uniform(12, 32, 36)
    base[17, 3], base[18, 0], base[4_000] = np.nan, np.inf, 1e30
    q[2, 1], q[3, 5] = np.nan, -np.inf
    t_ids, t_d, s_ids, s_d = _both(base, q, k)
    ok = [i for i in range(12) if i != 2]             # an undefined query has no defined order
    assert np.array_equal(t_ids[ok], s_ids[ok]) and np.array_equal(t_d[ok], s_d[ok])


@pytest.mark.parametrize("n,dim,nq,k", [
    (30_000, 64, 130, 10),        # a warp selects the threshold
    (30_000, 64, 9, 250),         # a block does
    (70_000, 20, 40, 600),        # every second row sampled
])
@pytest.mark.parametrize("offset", [10.0, 60.0, 1_000.0])
def test_queries_whose_candidates_outgrow_their_list(n, dim, nq, k, offset):
    # the window grows with the rows' distance from the origin: it takes some of the lists, most or all
    c = synth.mixture_centres(50, dim, 7)
    q = synth.mixture(nq, c, 0.3, 2)
    q[::3] *= np.float32(0.5)
    _same(synth.mixture(n, c, 0.3, 1) + np.float32(offset), q + np.float32(offset), k)


@pytest.mark.parametrize("k", [10, 300])
def test_far_rows_cost_little_more_than_the_cuda_cores(k):
    import paper_2307_10479_gb300 as deg
    from test_gpu_knn import _cuda_core
    c = synth.mixture_centres(50, 128, 7)
    base = torch.from_numpy(synth.mixture(100_000, c, 0.3, 1) + np.float32(1_000.0)).cuda()
    q = torch.from_numpy(synth.mixture(200, c, 0.3, 2) + np.float32(1_000.0)).cuda()
    took = []
    for f in (_cuda_core, deg.knn_exact):
        f(base, q, k)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(5):
            f(base, q, k)
        b.record()
        torch.cuda.synchronize()
        took.append(a.elapsed_time(b))
    assert took[1] < 2.5 * took[0]


@pytest.mark.parametrize("n,dim,nq,k", [
    (1_500, 53_000, 2, 300),      # above k = 256, and
    (1_100, 60_000, 3, 5),        # below: too wide for the re-rank's shared memory
    (1_100, 51_000, 3, 5),        # the widest that is not, nearly
])
def test_rows_of_many_columns(n, dim, nq, k):
    _same(synth.uniform(n, dim, 41), synth.uniform(nq, dim, 42), k)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33])      # up to 32 rows are scored outright
@pytest.mark.parametrize("dim", [3, 24, 130])
def test_nearest_of_very_few_rows(n, dim):
    import paper_2307_10479_gb300 as deg
    from test_gpu_knn import _cuda_core
    rows = synth.uniform(n, dim, 43)
    if n > 2:
        rows[n - 1] = rows[1]                          # a tie, to the lower index
    q = synth.uniform(77, dim, 44)
    q[5] = rows[n - 1]
    q[9, 0], q[70, dim - 1] = np.nan, np.inf
    r, qq = torch.from_numpy(rows).cuda(), torch.from_numpy(q).cuda()
    ids, d = deg.nearest_rows(r, qq)
    want, want_d = _cuda_core(r, qq, 1)
    ok = torch.tensor([i not in (9, 70) for i in range(77)], device="cuda")
    assert torch.equal(ids[ok], want[ok, 0]) and torch.equal(d[ok], want_d[ok, 0])
    assert (ids[~ok] == -1).all()                      # no finite distance: no row
