"""The work a user of this library has it do, as cases that can be timed and checked.

Every case goes through the public entry points of
``paper_1304_4327_gb300.dtree``: build the trees, search, give the trees back,
as a program with new points does; ``serve`` keeps its reference tree from
call to call, as a program that answers queries against one data set does.
Sizes and distributions are the library's own workloads (``inputs.py``,
``bench.py``), at full size or at a share of it.  Points are drawn on the GPU.

Sets come back in a canonical order: range results with each row's indices
ascending, in buffers of a size known beforehand (the rest holds -1 and 0), and
spanning-tree edges by their endpoints (what code that goes on to a sparse
matrix does), since their order follows the tree's layout.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1304_4327_gb300 import dtree

_TRAIN_HIDDEN = 256  # width of the proposal network's hidden layers


def listed():
    return [
        # one small data set, all neighbours of its own points (k-means seeding,
        # local outlier factor on a few thousand rows): launches and latency
        {"name": "knn_small", "op": "knn", "data": "uniform", "m": 10_000, "n": 0, "d": 3, "k": 5,
         "precision": "fp32", "leaf": 20, "block": 0, "cap": 0},
        # a service: the reference tree stays, a ragged batch of new queries
        # arrives and is answered on its own
        {"name": "knn_serve", "op": "serve", "data": "gmm", "m": 1_000_000, "n": 4_097, "d": 16, "k": 10,
         "precision": "bf16", "leaf": 32, "block": 0, "cap": 0},
        # the 16-dimensional mixture at full size, tensor-core tiles
        {"name": "knn_gmm16", "op": "knn", "data": "gmm", "m": 4_000_000, "n": 1_000_000, "d": 16, "k": 10,
         "precision": "bf16", "leaf": 32, "block": 256, "cap": 0},
        # low intrinsic dimension at full size: float32 tiles (the BF16 band is
        # wider than such data's neighbour gaps)
        {"name": "knn_latent8", "op": "knn", "data": "latent", "m": 10_000_000, "n": 1_000_000, "d": 8, "k": 10,
         "precision": "fp32", "leaf": 32, "block": 0, "cap": 0},
        # the high-dimensional workload (embeddings): long lists, hardly any
        # pruning; an eighth of the headline's pairs or so
        {"name": "knn_powerlaw64", "op": "knn", "data": "powerlaw", "m": 500_000, "n": 500_000, "d": 64, "k": 50,
         "precision": "bf16", "leaf": 32, "block": 512, "cap": 16},
        # one data set against itself at TF32, ragged size and odd dimension
        {"name": "knn_mono_tf32", "op": "knn", "data": "powerlaw", "m": 131_071, "n": 0, "d": 27, "k": 20,
         "precision": "tf32", "leaf": 32, "block": 0, "cap": 0},
        # many uneven problems in one call (per-class or per-patch searches)
        {"name": "knn_batch", "op": "batch", "problems": 24, "n_min": 1_000, "n_max": 200_000,
         "precision": "bf16", "leaf": 32, "block": 256},
        # k-furthest neighbours (diversity sampling, diameters) on the mixture
        {"name": "kfn_gmm16", "op": "kfn", "data": "gmm", "m": 1_000_000, "n": 200_000, "d": 16, "k": 10, "leaf": 32},
        # all neighbours within a radius (density estimates, DBSCAN)
        {"name": "range_gmm16", "op": "range", "data": "gmm", "m": 1_000_000, "n": 200_000, "d": 16, "leaf": 32,
         "lo": 0.0, "hi": 2.5, "room": 12},
        # the Euclidean minimum spanning tree: point clouds in space, and
        # single-linkage clustering of a mixture
        {"name": "emst_uniform3", "op": "emst", "data": "uniform", "m": 1_000_000, "d": 3, "leaf": 32},
        {"name": "emst_gmm16", "op": "emst", "data": "gmm", "m": 60_000, "d": 16, "leaf": 32},
        # one training step's loss and gradients of the leaf proposal
        {"name": "proposal_grad", "op": "grad", "n": 2_048, "d": 8, "classes": 8_192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _within(m, d, r):
    """Points of the mixture within r of one of its points, on average (d even; other components are out of reach)."""
    x = r * r / 4
    return m / 32 * (1 - math.exp(-x) * sum(x ** i / math.factorial(i) for i in range(d // 2)))


def draw(rng):
    kind = rng.choice(["knn", "knn", "knn", "serve", "batch", "kfn", "range", "emst", "grad"])
    leaf = rng.choice([16, 20, 32, 32, 64])
    if kind in ("knn", "serve"):
        data = rng.choice(["uniform", "gmm", "latent", "powerlaw"])
        d = {"uniform": rng.choice([2, 3, 4]), "gmm": rng.choice([10, 16, 20, 24]),
             "latent": rng.randint(4, 12), "powerlaw": rng.randint(24, 64)}[data]
        fp32 = data in ("uniform", "latent")
        m = _log_int(rng, 3_000, 4_000_000 if fp32 else 1_000_000)
        n = 0 if kind == "knn" and rng.random() < 0.3 else _log_int(rng, 500, 8_000 if kind == "serve" else 500_000)
        if n == 0:
            m = min(m, 400_000)
        if data == "powerlaw":  # hardly any pruning: all pairs, no more than the listed case's
            m, n = min(m, 400_000), min(n, 400_000)
        return {"op": kind, "data": data, "m": m, "n": n, "d": d, "k": rng.choice([1, 5, 10, 10, 20, 50]),
                "precision": "fp32" if fp32 else rng.choice(["bf16", "bf16", "tf32"]), "leaf": leaf,
                "block": rng.choice([0, 0, 256, 512]), "cap": rng.choice([0, 0, 16])}
    if kind == "batch":
        lo = _log_int(rng, 500, 2_000)
        return {"op": "batch", "problems": rng.randint(6, 30), "n_min": lo, "n_max": _log_int(rng, 20_000, 200_000),
                "precision": rng.choice(["bf16", "fp32"]), "leaf": leaf, "block": rng.choice([0, 256, 512])}
    if kind == "kfn":
        data = rng.choice(["gmm", "gmm", "uniform"])
        d = rng.choice([10, 16, 20]) if data == "gmm" else rng.choice([2, 3, 8])
        mono = rng.random() < 0.4
        return {"op": "kfn", "data": data, "m": _log_int(rng, 5_000, 40_000 if mono else 1_000_000),
                "n": 0 if mono else _log_int(rng, 2_000, 100_000), "d": d, "k": rng.choice([1, 5, 10, 30]), "leaf": leaf}
    if kind == "range":
        if rng.random() < 0.5:
            m, d = _log_int(rng, 10_000, 1_000_000), 16
            hi, lo = rng.uniform(2.0, 2.7), rng.choice([0.0, 0.0, 1.5])
            data, found = "gmm", _within(m, d, hi)
        else:
            m, d = _log_int(rng, 10_000, 2_000_000), rng.choice([2, 3, 5])
            ball = math.pi ** (d / 2) / math.gamma(d / 2 + 1)
            found = rng.uniform(8, 60)  # points within the radius
            hi = (found / (m * ball)) ** (1 / d)
            lo, data = rng.choice([0.0, 0.0, 0.5]) * hi, "uniform"
        return {"op": "range", "data": data, "m": m, "n": _log_int(rng, 2_000, 200_000), "d": d, "leaf": leaf,
                "lo": lo, "hi": hi, "room": math.ceil(1.3 * found) + 3}
    if kind == "emst":
        if rng.random() < 0.5:
            return {"op": "emst", "data": "uniform", "m": _log_int(rng, 3_000, 800_000), "d": rng.choice([2, 3, 4]),
                    "leaf": leaf}
        return {"op": "emst", "data": "gmm", "m": _log_int(rng, 3_000, 50_000), "d": rng.choice([8, 16]), "leaf": leaf}
    return {"op": "grad", "n": rng.randint(300, 4_096), "d": rng.randint(3, 64), "classes": _log_int(rng, 100, 10_000)}


# ---- inputs ---------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _points(data, n, d, g, shared):
    """n points of a distribution; ``shared`` holds what references and queries have in common."""
    if data == "uniform":
        return torch.rand(n, d, generator=g, device="cuda")
    if data == "gmm":  # 32 isotropic components, centres U[-10, 10]^d, sigma 1
        if "c" not in shared:
            shared["c"] = torch.rand(32, d, generator=g, device="cuda") * 20 - 10
        comp = torch.randint(0, 32, (n,), generator=g, device="cuda")
        return torch.randn(n, d, generator=g, device="cuda") + shared["c"][comp]
    if data == "latent":  # 3 latent uniforms mapped to d dimensions, plus N(0, 0.01^2)
        if "a" not in shared:
            shared["a"] = torch.randn(d, 3, generator=g, device="cuda")
        z = torch.rand(n, 3, generator=g, device="cuda")
        return z @ shared["a"].T + 0.01 * torch.randn(n, d, generator=g, device="cuda")
    # powerlaw: Gaussian, eigenvalue i ~ i^-1.5, a random rotation
    if "m" not in shared:
        q, r = torch.linalg.qr(torch.randn(d, d, generator=g, device="cuda", dtype=torch.float64).cpu())
        q = (q * torch.sign(torch.diagonal(r))[None, :]).cuda()
        scale = torch.arange(1, d + 1, device="cuda", dtype=torch.float64) ** -0.75
        shared["m"] = (q * scale[None, :]).float()
    return torch.randn(n, d, generator=g, device="cuda") @ shared["m"].T


def _shapes(case):
    """The problems of a batch: sizes log-normal around 14,142, d in {3, 8, 32}, k in {1, 10}."""
    rng = random.Random(case["problems"] * 1_000_003 + case["n_max"])
    out = []
    for _ in range(case["problems"]):
        n = int(round(math.exp(rng.gauss(math.log(14_142), 1.32))))
        out.append((max(case["n_min"], min(case["n_max"], n)), rng.choice([3, 8, 32]), rng.choice([1, 10]),
                    rng.choice(["uniform", "gaussian"])))
    return out


def _inputs(case, seed):
    g = _gen(seed)
    if case["op"] == "batch":
        return [torch.rand(n, d, generator=g, device="cuda") if kind == "uniform" else
                torch.randn(n, d, generator=g, device="cuda") for n, d, _, kind in _shapes(case)]
    if case["op"] == "grad":
        n, d, c, h = case["n"], case["d"], case["classes"], _TRAIN_HIDDEN
        shapes = [(h, d), (h,), (h, h), (h,), (c, h), (c,)]
        params = [torch.randn(s, generator=g, device="cuda") * (s[-1] ** -0.5 if len(s) == 2 else 0.1) for s in shapes]
        x = torch.randn(n, d, generator=g, device="cuda")
        t = torch.zeros(n, c, device="cuda")  # each example's neighbours fall into a few cells
        cells = torch.randint(0, c, (n, 8), generator=g, device="cuda")
        t.scatter_add_(1, cells, torch.full((n, 8), 0.125, device="cuda"))
        return params, x, t
    shared = {}
    ref = _points(case["data"], case["m"], case["d"], g, shared)
    query = _points(case["data"], case["n"], case["d"], g, shared) if case.get("n") else None
    return ref, query


def prepare(case, seed):
    state = {"case": case, "in": _inputs(case, seed)}
    if case["op"] == "serve":
        state["tree"] = dtree.dtree_build(state["in"][0], case["leaf"])
    return state


# ---- one pass -------------------------------------------------------------

def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "knn":
        ref, query = state["in"]
        return dtree.knn(ref, query, case["k"], leaf_size=case["leaf"], precision=case["precision"],
                         query_block=case["block"], cap_leaves=case["cap"])
    if op == "serve":
        tq = dtree.dtree_build(state["in"][1], case["leaf"])
        try:
            return dtree.dtree_knn(tq, state["tree"], case["k"], precision=case["precision"],
                                   query_block=case["block"], cap_leaves=case["cap"])
        finally:
            tq.free()
    if op == "batch":
        trees = [dtree.dtree_build(p, case["leaf"]) for p in state["in"]]
        try:
            return dtree.dtree_knn_batch([(None, t, k, case["block"]) for t, (_, _, k, _) in zip(trees, _shapes(case))],
                                         precision=case["precision"])
        finally:
            for t in trees:
                t.free()
    if op == "grad":
        return dtree.dtree_mlp_loss_grad(*state["in"])
    ref, query = state["in"] if op != "emst" else (state["in"][0], None)
    tr = dtree.dtree_build(ref, case["leaf"])
    tq = None if query is None else dtree.dtree_build(query, case["leaf"])
    try:
        if op == "kfn":
            return dtree.dtree_kfn(tq, tr, case["k"])
        if op == "range":
            return _by_row(*dtree.dtree_range(tq, tr, case["lo"], case["hi"]), case)
        edges, dist = dtree.dtree_emst(tr)
        order = torch.argsort(edges[:, 0] * case["m"] + edges[:, 1])
        return edges[order], dist[order]
    finally:
        tr.free()
        if tq is not None:
            tq.free()


def _by_row(offsets, idx, dist, case):
    """Range results with each row's indices ascending (canonical CSR), in buffers of room x n."""
    rows = torch.repeat_interleave(torch.arange(case["n"], device=idx.device), offsets.diff(), output_size=idx.numel())
    order = torch.argsort(rows * case["m"] + idx)
    return offsets, *_room(idx[order], dist[order], case)


def _room(idx, dist, case):
    size = case["room"] * case["n"]
    out_idx = torch.full((size,), -1, dtype=idx.dtype, device=idx.device)
    out_dist = torch.zeros(size, dtype=dist.dtype, device=idx.device)
    out_idx[:idx.numel()] = idx
    out_dist[:idx.numel()] = dist
    return out_idx, out_dist


def work(case):
    """Inputs read and outputs written once; of the distances only the returned ones."""
    op = case["op"]
    if op == "grad":
        n, d, c, h = case["n"], case["d"], case["classes"], _TRAIN_HIDDEN
        weights = h * d + h * h + c * h
        return {"bytes": 4 * (2 * weights + n * (d + c)), "flops": 6 * n * weights}
    if op == "batch":
        s = _shapes(case)
        return {"bytes": sum(4 * n * d + 12 * n * k for n, d, k, _ in s), "flops": sum(3 * d * n * k for n, d, k, _ in s)}
    m, d = case["m"], case["d"]
    if op == "emst":
        return {"bytes": 4 * m * d + 20 * (m - 1), "flops": 3 * d * m}
    n = case["n"] or m
    k = case.get("k", case.get("room"))
    read = 4 * d * n if op == "serve" or not case["n"] else 4 * d * (m + n)
    return {"bytes": read + 12 * n * k, "flops": 3 * d * n * k}


# ---- the same in 64 bits --------------------------------------------------

def _filter(q, r):
    """Rough squared distances in float32 (the sign and order are settled in float64 afterwards)."""
    if r.shape[1] <= 12:
        acc = torch.zeros(q.shape[0], r.shape[0], device=q.device)
        for j in range(r.shape[1]):
            t = q[:, j, None] - r[None, :, j]
            acc.addcmul_(t, t)
        return acc
    return torch.addmm((q * q).sum(1, keepdim=True) + (r * r).sum(1)[None, :], q, r.T, alpha=-2)


def _brute_knn(ref, query, k, furthest=False):
    mono = query is None
    query = ref if mono else query
    shift = ref.mean(0)
    r32, q32 = ref - shift, query - shift
    take = min(k + 40, ref.shape[0] - (1 if mono else 0))
    step = max(1, min(2_000_000_000 // (4 * ref.shape[0]), 16_384))
    idx, dist = [], []
    for a in range(0, query.shape[0], step):
        d2 = _filter(q32[a:a + step], r32)
        if mono:
            i = torch.arange(d2.shape[0], device=d2.device)
            d2[i, i + a] = -math.inf if furthest else math.inf
        cand = d2.topk(take, dim=1, largest=furthest, sorted=False).indices.sort(1).values
        del d2
        e = (query[a:a + step, None, :].double() - ref[cand].double()).square_().sum(2)
        e, o = e.sort(dim=1, descending=furthest, stable=True)  # ties: the lower index first
        idx.append(cand.gather(1, o[:, :k]))
        dist.append(e[:, :k].sqrt())
    return torch.cat(idx), torch.cat(dist)


def _brute_range(ref, query, case):
    lo, hi = case["lo"], case["hi"]
    shift = ref.mean(0)
    step = max(1, min(1_000_000_000 // (4 * ref.shape[0]), 16_384))
    tol = 1e-5 * float((ref - shift).square().sum(1).max()) if ref.shape[1] > 12 else 0.0
    counts, idx, dist = [], [], []
    for a in range(0, query.shape[0], step):
        row, col = torch.nonzero(_filter(query[a:a + step] - shift, ref - shift) <= hi * hi * 1.001 + tol, as_tuple=True)
        e = (query[a + row].double() - ref[col].double()).square_().sum(1).sqrt_()
        keep = (e >= lo) & (e <= hi)
        counts.append(torch.bincount(row[keep], minlength=min(step, query.shape[0] - a)))
        idx.append(col[keep])
        dist.append(e[keep])
    offsets = torch.cat([torch.zeros(1, dtype=torch.int64, device=ref.device), torch.cat(counts).cumsum(0)])
    return offsets, *_room(torch.cat(idx), torch.cat(dist), case)


def _prim(points):
    p = points.double()
    n = p.shape[0]
    best = torch.full((n,), math.inf, dtype=torch.float64, device=p.device)
    near = torch.zeros(n, dtype=torch.int64, device=p.device)
    done = torch.zeros(n, dtype=torch.bool, device=p.device)
    ends = torch.zeros(n, 2, dtype=torch.int64, device=p.device)
    d2 = torch.zeros(n, dtype=torch.float64, device=p.device)
    cur = torch.zeros(1, dtype=torch.int64, device=p.device)
    inf = torch.full((), math.inf, dtype=torch.float64, device=p.device)
    for t in range(1, n):
        done.index_fill_(0, cur, True)
        e = (p - p[cur]).square_().sum(1)
        closer = e < best
        best = torch.where(closer, e, best)
        near = torch.where(closer, cur, near)
        v, cur = torch.where(done, inf, best).min(0, keepdim=True)
        d2[t:t + 1] = v
        ends[t, :1] = near[cur]
        ends[t, 1:] = cur
    ends, d2 = ends[1:].sort(1).values, d2[1:]
    order = torch.argsort(ends[:, 0] * n + ends[:, 1])
    return ends[order], d2[order].sqrt()


def exact(case, seed):
    op = case["op"]
    x = _inputs(case, seed)
    if op == "grad":
        params, inp, t = x
        p = [w.double().requires_grad_() for w in params]
        h = torch.relu(inp.double() @ p[0].T + p[1])
        h = torch.relu(h @ p[2].T + p[3])
        loss = -(t.double() * torch.log_softmax(h @ p[4].T + p[5], 1)).sum(1).mean()
        return loss.item(), list(torch.autograd.grad(loss, p))
    if op == "batch":
        if sum(n * n for n, _, _, _ in _shapes(case)) > 2e11:
            return None
        return [_brute_knn(p, None, k) for p, (_, _, k, _) in zip(x, _shapes(case))]
    if op == "emst":
        return _prim(x[0]) if case["m"] <= 60_000 else None
    ref, query = x
    if case["m"] * (case["n"] or case["m"]) > 2.6e11:
        return None
    if op == "range":
        return _brute_range(ref, query, case)
    return _brute_knn(ref, query, case["k"], furthest=op == "kfn")
