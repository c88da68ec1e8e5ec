"""Range search by the block search (d > 8, a billion pairs or more) against
the one-warp-per-query walk, which takes the same queries in smaller calls and
is checked by the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


def clusters(n, d, seed):
    g = np.random.default_rng(seed)
    c = np.random.default_rng(d).uniform(-10, 10, size=(12, d))
    return g.normal(size=(n, d)) + c[g.integers(0, 12, n)]


def canonical(off, idx, dist, m):
    rows = torch.repeat_interleave(torch.arange(off.numel() - 1, device=idx.device), off.diff())
    order = torch.argsort(rows * m + idx)
    return idx[order], dist[order]


def compare(R, Q, lo, hi, leaf=32):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    R, Q = cuda(R), cuda(Q)
    m = R.shape[0]
    assert m * Q.shape[0] >= 10 ** 9
    tr, tq = dtree.dtree_build(R, leaf), dtree.dtree_build(Q, leaf)
    counts, ids, ds = [], [], []
    try:
        off, idx, dist = dtree.dtree_range(tq, tr, lo, hi)
        again = dtree.dtree_range(tq, tr, lo, hi)
        assert all(torch.equal(x, y) for x, y in zip((off, idx, dist), again))  # the same order every call
        step = min(9_000, 10 ** 9 // m - 1)
        for a in range(0, Q.shape[0], step):
            t = dtree.dtree_build(Q[a:a + step], leaf)
            o, i, d = dtree.dtree_range(t, tr, lo, hi)
            t.free()
            i, d = canonical(o, i, d, m)
            counts.append(o.diff())
            ids.append(i)
            ds.append(d)
    finally:
        tr.free()
        tq.free()
    assert torch.equal(off.diff(), torch.cat(counts))
    idx, dist = canonical(off, idx, dist, m)
    assert torch.equal(idx, torch.cat(ids)) and torch.equal(dist, torch.cat(ds))
    return int(off[-1])


@pytest.mark.parametrize("d", [9, 16, 17, 33, 64])
@pytest.mark.parametrize("lo,hi", [(0.0, 0.62), (0.55, 0.75)])
def test_clusters(d, lo, hi):
    s = (2 * d) ** 0.5  # the typical distance within a cluster
    assert compare(clusters(30_011, d, 1), clusters(33_333, d, 2), lo * s, hi * s) > 0


@pytest.mark.parametrize("nq,leaf", [(20_001, 20), (81_003, 64), (40_000, 5)])
def test_sizes(nq, leaf):
    compare(clusters(50_001, 12, 3), clusters(nq, 12, 4), 0.0, 2.2, leaf)


def test_both_ends_hit_exactly():
    # integer points: many distances on both ends
    g = np.random.default_rng(5)
    R, Q = g.integers(0, 4, size=(40_000, 10)), g.integers(0, 4, size=(25_001, 10))
    assert compare(R, Q, 1.0, 2.0) > 0


@pytest.mark.parametrize("lo,hi", [(0.0, 1e-3), (60.0, 1e4), (1e3, 2e3), (3.0, 3.0)])
def test_extremes(lo, hi):
    # (a radius far below the extents stays with the walk)
    compare(clusters(40_000, 16, 6) * 1.0, clusters(25_001, 16, 7), lo, hi)


def test_monochromatic():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    P = cuda(clusters(32_003, 16, 9))
    t, t2 = dtree.dtree_build(P, 32), dtree.dtree_build(P, 16)
    try:
        off, idx, dist = dtree.dtree_range(None, t, 0.0, 2.5)
        o2, i2, d2 = dtree.dtree_range(t2, t, 0.0, 2.5)  # the same points as other queries: each finds itself too
    finally:
        t.free()
        t2.free()
    assert torch.equal(off.diff() + 1, o2.diff())
    i2, d2 = canonical(o2, i2, d2, P.shape[0])
    rows = torch.repeat_interleave(torch.arange(P.shape[0], device="cuda"), o2.diff())
    keep = i2 != rows
    idx, dist = canonical(off, idx, dist, P.shape[0])
    assert torch.equal(idx, i2[keep]) and torch.equal(dist, d2[keep])
