"""What a user of the library has it do, as measurable cases: batched and single searches, ground
truth, and the training of entry points and of the stop network.

The search cases run over graphs made here, on the GPU and in a few seconds, with the shape of a
search graph: every vertex linked to its nearest rows inside two partitions of the data, filled up
to the exact degree with random links. (The library's device builder leaves open which of two
concurrent insertions comes first, so two of its graphs differ.) A program keeps its index while
queries come and go, so an index is made once per size and kept; the queries come from the seed.
Rows are Gaussian mixtures: rounded to 0..255 ("u8"), as they are ("mix"), or scaled to unit length
("unit"). Sizes are those of the workloads in synth.py.
"""
import collections
import math

import numpy as np
import torch

import paper_2307_10479_gb300 as deg

U8 = {"data": "u8", "n": 1_000_000, "dim": 128, "degree": 30}

_KEPT = 3
_indexes = collections.OrderedDict()


def listed():
    return [
        # an interactive user: one query at a time against the full index, smallest latency wanted
        {"name": "one_query_fp8", "do": "search", **U8, "nq": 1, "k": 10, "eps": 0.015, "precision": "fp8", "rerank": 32, "entry": "learned"},
        # the same form as a service's or an offline job's batch: the benchmark's headline step
        {"name": "batch_fp8_learned", "do": "search", **U8, "nq": 10_000, "k": 10, "eps": 0.015, "precision": "fp8", "rerank": 32, "entry": "learned"},
        # the paper's own form: float32 rows, every query from the fixed entry vertex
        {"name": "batch_f32_fixed", "do": "search", **U8, "nq": 10_000, "k": 10, "eps": 0.08, "precision": "f32", "rerank": 0, "entry": "fixed"},
        # a web request's worth of queries in full precision, routed
        {"name": "batch64_f32_pivot", "do": "search", **U8, "nq": 64, "k": 10, "eps": 0.04, "precision": "f32", "rerank": 0, "entry": "pivot"},
        # unit vectors in 100 dimensions (no multiple of a 16-byte chunk), bfloat16 rows, an odd count
        {"name": "unit100_bf16", "do": "search", "data": "unit", "n": 200_000, "dim": 100, "degree": 30, "nq": 1_237, "k": 10, "eps": 0.02, "precision": "bf16", "rerank": 32, "entry": "pivot"},
        # browsing: the 100 nearest of a vertex the user looks at
        {"name": "explore_k100", "do": "explore", **U8, "nq": 2_000, "k": 100, "eps": 0.0, "precision": "f32", "rerank": 0, "entry": "fixed"},
        # the headline form from host buffers: copy in, search, copy out
        {"name": "host_fp8_learned", "do": "host", **U8, "nq": 10_000, "k": 10, "eps": 0.015, "precision": "fp8", "rerank": 32, "entry": "learned"},
        # ground truth of the benchmark: integer rows
        {"name": "truth_u8", "do": "knn", "data": "u8", "n": 1_000_000, "dim": 128, "nq": 10_000, "k": 10},
        # ground truth of float rows in many dimensions, where bfloat16 products are not exact
        {"name": "truth_mix960", "do": "knn", "data": "mix", "n": 1_000_000, "dim": 960, "nq": 1_000, "k": 10},
        # ground truth of the exploration protocol: recall@1000 and the vertex itself
        {"name": "truth_k1001", "do": "knn", "data": "u8", "n": 1_000_000, "dim": 128, "nq": 200, "k": 1_001},
        # preparing an index for routed searches: k-means entry points, one for 256 rows
        {"name": "train_entry", "do": "entry", "data": "u8", "n": 500_000, "dim": 128, "degree": 4, "k": 1_953, "iters": 10},
        # one minibatch of the early-stop network's training: loss, gradient, Adam step
        {"name": "stop_step", "do": "stop", "count": 8_192},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["search"] * 6 + ["explore", "host"] + ["knn"] * 3 + ["entry", "stop"])
    if do == "stop":
        return {"do": do, "count": _log(rng, 200, 65_536)}
    data = rng.choice(["u8", "u8", "mix", "unit"])
    if do == "knn":
        n, dim = _log(rng, 2_000, 1_000_000), _log(rng, 24, 960)
        nq = _log(rng, 1, max(2, min(10_000, 4 * 10**11 // (n * dim))))
        return {"do": do, "data": data, "n": n, "dim": dim, "nq": nq, "k": _log(rng, 1, rng.choice([100, 100, 1_024]))}
    if do == "entry":
        n = _log(rng, 20_000, 400_000)
        return {"do": do, "data": "u8", "n": n, "dim": 4 * _log(rng, 8, 64), "degree": 4, "k": _log(rng, n // 1_024, min(4_096, n // 128)), "iters": rng.randint(2, 10)}
    n, dim, degree = _log(rng, 10_000, 500_000), _log(rng, 24, 384), 2 * rng.randint(4, 20)
    case = {"do": do, "data": data, "n": n, "dim": dim, "degree": degree, "nq": _log(rng, 1, 10_000), "k": _log(rng, 1, 100)}
    case["precision"] = rng.choice(["f32", "bf16", "fp8"])
    case["rerank"] = 0 if case["precision"] == "f32" else max(32, 2 * case["k"])
    case["entry"] = "fixed" if do == "explore" else rng.choice(["fixed", "pivot", "learned" if dim % 4 == 0 else "pivot"])
    case["eps"] = round(rng.uniform(0.02, 0.08), 3) if case["entry"] == "fixed" and do != "explore" else round(rng.uniform(0.0, 0.03), 3)
    return case


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed & 0x7FFFFFFF)


def _rows(data, count, dim, seed):
    """`count` rows of the mixture (its centres are the same for every seed), float32 on the GPU."""
    g = _gen(seed)
    centres = {"u8": 1_000, "mix": 500, "unit": 1_000}[data]
    c = torch.rand((centres, dim), generator=_gen(7), device="cuda") * 255 if data == "u8" else torch.randn((centres, dim), generator=_gen(7), device="cuda")
    spread = {"u8": 20.0, "mix": 0.3, "unit": 0.5}[data]
    x = torch.empty((count, dim), device="cuda")
    for lo in range(0, count, 1 << 17):
        m = min(1 << 17, count - lo)
        at = torch.randint(centres, (m,), generator=g, device="cuda")
        x[lo:lo + m] = c[at] + torch.randn((m, dim), generator=g, device="cuda") * spread
    if data == "u8":
        x.round_().clamp_(0, 255)
    elif data == "unit":
        x /= x.norm(dim=1, keepdim=True)
    return x


def _near_pairs(x, want, seed, cell=512):
    """Pairs (u, v, d2) of near rows: rows sorted by the nearest of some sampled rows, cut into cells of
    `cell`, and the `want` nearest of every row inside its cell."""
    n, g = x.shape[0], _gen(seed)
    picks = x[torch.randperm(n, generator=g, device=x.device)[:max(1, n // cell)]]
    half = picks.square().sum(1) / 2
    label = torch.cat([(half - x[lo:lo + 65_536] @ picks.T).argmin(1) for lo in range(0, n, 65_536)])
    order = label.sort(stable=True).indices
    order = torch.cat([order, order[:-n % cell]]).view(-1, cell)
    out = []
    for lo in range(0, order.shape[0], 128):
        ids = order[lo:lo + 128]
        r = x[ids]
        s = r.square().sum(2)
        d2 = s.unsqueeze(2) + s.unsqueeze(1) - 2 * (r @ r.transpose(1, 2))
        d2.diagonal(dim1=1, dim2=2).fill_(float("inf"))
        d2, j = d2.sort(dim=2, stable=True)
        u = ids.unsqueeze(2).expand(-1, -1, want)
        v = ids.gather(1, j[:, :, :want].reshape(ids.shape[0], -1)).view_as(u)
        out.append((u.reshape(-1), v.reshape(-1), d2[:, :, :want].reshape(-1)))
    return [torch.cat(t) for t in zip(*out)]


def _graph(x, degree, seed=11):
    """Adjacency [n, degree] of a simple undirected regular graph over the rows."""
    n, dev, g = x.shape[0], x.device, _gen(seed)
    near = degree - max(2, degree // 8)
    u, v, d2 = (torch.cat(t) for t in zip(*[_near_pairs(x, near, seed + p) for p in (1, 2)]))
    ok = u != v
    u, v, d2 = u[ok], v[ok], d2[ok]
    key = torch.minimum(u, v) * n + torch.maximum(u, v)
    by = d2.sort(stable=True).indices
    key = key[by]
    key, at = key.sort(stable=True)                                # shortest first among equal pairs
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    at, key = at[first], key[first]
    key = key[at.sort(stable=True).indices]                        # distinct pairs, by length

    room = torch.full((n,), near, device=dev)
    kept = []
    for _ in range(8):                                             # greedily, many pairs at a time
        ends = torch.stack([key // n, key % n], 1).view(-1)
        s, i = ends.sort(stable=True)
        start = torch.zeros(n + 1, dtype=torch.long, device=dev)
        start[1:] = torch.bincount(s, minlength=n).cumsum(0)
        rank = torch.empty_like(i)
        rank[i] = torch.arange(len(i), device=dev) - start[s]
        take = (rank < room[ends]).view(-1, 2).all(1)
        kept.append(key[take])
        room -= torch.bincount(ends.view(-1, 2)[take].view(-1), minlength=n)
        key = key[~take]
        key = key[(room[key // n] > 0) & (room[key % n] > 0)]
        if not len(key):
            break
    edges = torch.cat(kept).sort().values

    def known(keys, among):
        i = torch.searchsorted(among, keys).clamp_(max=len(among) - 1)
        return among[i] == keys

    def pair(a, b):
        return torch.minimum(a, b) * n + torch.maximum(a, b)

    def once(keys):
        s, i = keys.sort(stable=True)
        f = torch.ones_like(s, dtype=torch.bool)
        f[1:] = s[1:] != s[:-1]
        out = torch.zeros_like(f)
        out[i] = f
        return out

    left = torch.repeat_interleave(torch.arange(n, device=dev), room + degree - near)
    for _ in range(12):                                            # random links between the free ends
        left = left[torch.randperm(len(left), generator=g, device=dev)]
        a, b = left.view(-1, 2).T
        k = pair(a, b)
        good = (a != b) & once(k) & ~known(k, edges)
        edges = torch.cat([edges, k[good]]).sort().values
        left = left.view(-1, 2)[~good].reshape(-1)
        if not len(left):
            break
    while len(left):                                               # the last ones: a-x and b-y for an edge x-y
        left = left[torch.randperm(len(left), generator=g, device=dev)]
        a, b = left.view(-1, 2).T
        i = torch.randint(len(edges), (len(a),), generator=g, device=dev)
        p, q = edges[i] // n, edges[i] % n
        k1, k2 = pair(a, p), pair(b, q)
        good = once(i) & (a != p) & (b != q) & (k1 != k2) & ~known(k1, edges) & ~known(k2, edges)
        both = once(torch.cat([k1, k2])).view(2, -1)
        good &= both[0] & both[1]
        drop = torch.zeros(len(edges), dtype=torch.bool, device=dev)
        drop[i[good]] = True
        edges = torch.cat([edges[~drop], k1[good], k2[good]]).sort().values
        left = left.view(-1, 2)[~good].reshape(-1)
    u, v = edges // n, edges % n
    src, i = torch.cat([u, v]).sort(stable=True)
    return torch.cat([v, u])[i].view(n, degree).int()


def _index(case):
    """The index of a case's size: rows of a fixed seed, the graph, the copies and entry points it needs."""
    key = tuple(case[f] for f in ("data", "n", "dim", "degree"))
    idx = _indexes.pop(key, None)
    if idx is None:
        while len(_indexes) >= _KEPT:
            _indexes.popitem(last=False)
        x = _rows(case["data"], case["n"], case["dim"], 1)
        idx = deg.Index.from_arrays(x.cpu().numpy(), _graph(x, case["degree"]).cpu().numpy())
        del x
        torch.cuda.empty_cache()
        idx.upload(("f32", "bf16", "fp8"))
        if case["dim"] % 4 == 0:
            idx.train_entry(max(1, min(4_096, case["n"] // 256)), 10)
    _indexes[key] = idx
    return idx


def _stop_inputs(case, seed):
    """Features in their ranges with labels that depend on them, weights, and Adam's moments after a while."""
    g, count = _gen(2 * seed + 102), case["count"]
    x = torch.rand((count, deg.STOP_FEATURES), generator=g, device="cuda") * 2
    y = (x[:, 6] - x[:, 7] + torch.randn(count, generator=g, device="cuda") > 0.5).int()
    w = torch.from_numpy(deg.mlp_init(seed)).cuda()
    m = torch.randn(w.shape, generator=g, device="cuda") * 1e-3
    return x, y, w, m, m.square() + torch.rand(w.shape, generator=g, device="cuda") * 1e-5 + 1e-6


def prepare(case, seed):
    s = dict(case)
    if case["do"] == "stop":
        s["x"], s["y"], s["w"], s["m"], s["v"] = _stop_inputs(case, seed)
        return s
    if case["do"] == "knn":
        s["base"] = _rows(case["data"], case["n"], case["dim"], 2 * seed + 101)
        s["queries"] = _rows(case["data"], case["nq"], case["dim"], 2 * seed + 102)
        return s
    if case["do"] == "entry":
        # the graph plays no part in the training: a ring with chords
        i = np.arange(case["n"], dtype=np.int32)[:, None]
        ring = (i + np.array([-2, -1, 1, 2], np.int32)) % case["n"]
        s["index"] = deg.Index.from_arrays(_rows(case["data"], case["n"], case["dim"], 2 * seed + 101).cpu().numpy(), ring.astype(np.int32))
        s["index"].upload()
        return s
    s["index"] = _index(case)
    if case["do"] == "explore":
        s["vertices"] = torch.randperm(case["n"], generator=_gen(2 * seed + 102), device="cuda")[:case["nq"]].int()
        return s
    q = _rows(case["data"], case["nq"], case["dim"], 2 * seed + 102)
    if case["do"] == "host":
        s["queries"] = q.cpu().pin_memory()
        s["ids"] = torch.empty((case["nq"], case["k"]), dtype=torch.int32).pin_memory()
        s["dists"] = torch.empty((case["nq"], case["k"]), dtype=torch.float32).pin_memory()
    else:
        s["queries"] = q
    return s


def run(s):
    do = s["do"]
    if do == "stop":
        loss, grad = deg.mlp_loss_grad(s["w"], s["x"], s["y"])
        deg.mlp_adam(s["w"], s["m"], s["v"], grad, 100, 2e-3)
        return loss, grad, s["w"], s["m"], s["v"]
    if do == "knn":
        return deg.knn_exact(s["base"], s["queries"], s["k"])
    if do == "entry":
        sizes = s["index"].train_entry(s["k"], s["iters"])
        return sizes, s["index"].pivots(learned=True)
    how = {"k": s["k"], "eps": s["eps"], "precision": s["precision"], "rerank": s["rerank"]}
    if do == "explore":
        return s["index"].search(seeds=s["vertices"], explore=True, **how)
    if do == "host":
        return s["index"].search_host(s["queries"].numpy(), entry=s["entry"], out=(s["ids"].numpy(), s["dists"].numpy()), **how)
    return s["index"].search(s["queries"], entry=s["entry"], **how)


def work(case):
    if case["do"] == "stop":
        params = deg.STOP_PARAMS
        return {"bytes": 4.0 * (13 * case["count"] + 8 * params), "flops": 6.0 * case["count"] * params}
    n, dim, k = case["n"], case["dim"], case["k"]
    if case["do"] == "knn":
        return {"bytes": 4 * dim * (n + case["nq"]) + 8 * k * case["nq"], "flops": 2.0 * case["nq"] * n * dim}
    if case["do"] == "entry":
        return {"bytes": 4.0 * n * dim * (case["iters"] + 1), "flops": 2.0 * n * dim * k * (case["iters"] + 1) + 2.0 * n * dim * k}
    # a walk reads an adjacency row for every expanded vertex and a stored row for every new one
    hops, new = _walk(case)
    row = {"f32": 4 * dim, "bf16": 2 * dim, "fp8": dim + 4}[case["precision"]]
    again = 0 if case["precision"] == "f32" else 4 * dim * max(case["rerank"], k)
    per = 4 * dim + 8 * k + hops * (4 * case["degree"] + new * row) + again
    return {"bytes": float(case["nq"] * per), "flops": 2.0 * case["nq"] * dim * hops * new}


def _walk(case):
    """About how many vertices a query of the case expands, and how many new rows each shows."""
    kept = max(case["k"], case["rerank"])
    far = 100 if case["entry"] == "fixed" and case["do"] != "explore" else 0
    return (kept + 10) * (1 + 25 * case["eps"]) + far, 0.45 * case["degree"]


def _exact_stop(case, seed):
    x, y, w, m, v = _stop_inputs(case, seed)
    w = w.double().requires_grad_()
    w1, b1, w2, b2, w3, b3 = w.split([64 * 12, 64, 64 * 64, 64, 2 * 64, 2])
    h = torch.relu(torch.relu(x.double() @ w1.view(64, 12).T + b1) @ w2.view(64, 64).T + b2)
    loss = torch.nn.functional.cross_entropy(h @ w3.view(2, 64).T + b3, y.long())
    grad, = torch.autograd.grad(loss, w)
    m, v = 0.9 * m.double() + 0.1 * grad, 0.999 * v.double() + 0.001 * grad.square()
    step = 2e-3 * (m / (1 - 0.9**100)) / ((v / (1 - 0.999**100)).sqrt() + 1e-8)
    return loss.detach().view(1), grad, w.detach() - step, m, v


def exact(case, seed):
    if case["do"] == "stop":
        return _exact_stop(case, seed)
    if case["do"] != "knn" or case["n"] * case["nq"] * case["dim"] > 1.5e12:
        return None
    s = prepare(case, seed)
    x, q, k = s["base"].double(), s["queries"].double(), case["k"]
    half, out = x.square().sum(1) / 2, []
    step = max(1, min(case["nq"], 2 * 10**9 // case["n"] // 8))
    for lo in range(0, case["nq"], step):
        at = (half - q[lo:lo + step] @ x.T).topk(min(case["n"], k + 8), largest=False, sorted=False).indices
        d = torch.stack([(x[i] - v).square().sum(1).sqrt() for i, v in zip(at, q[lo:lo + step])])
        out.append(d.sort(dim=1).values[:, :k])
    return None, torch.cat(out)
