"""k-furthest neighbours by the block search (d > 8, a billion pairs or more)
against the one-warp-per-query search, which takes the same queries in smaller
calls and is checked by the oracle."""
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


def lattice(n, d, seed):  # equal distances everywhere
    return np.random.default_rng(seed).integers(0, 3, size=(n, d))


def compare(R, Q, k, leaf=32):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    R, Q = cuda(R), cuda(Q)
    assert R.shape[0] * Q.shape[0] >= 10 ** 9
    tr, tq = dtree.dtree_build(R, leaf), dtree.dtree_build(Q, leaf)
    parts = []
    try:
        idx, dist = dtree.dtree_kfn(tq, tr, k)
        step = min(4_000, 10 ** 9 // R.shape[0] - 1)
        for a in range(0, Q.shape[0], step):
            t = dtree.dtree_build(Q[a:a + step], leaf)
            parts.append(dtree.dtree_kfn(t, tr, k))
            t.free()
    finally:
        tr.free()
        tq.free()
    assert torch.equal(idx, torch.cat([p[0] for p in parts]))
    assert torch.equal(dist, torch.cat([p[1] for p in parts]))


@pytest.mark.parametrize("d", [9, 16, 17, 33, 64])
@pytest.mark.parametrize("k", [1, 10, 18, 63])
def test_clusters(d, k):
    compare(clusters(30_011, d, 1), clusters(33_333, d, 2), k)


@pytest.mark.parametrize("nq,leaf", [(20_000, 20), (81_003, 64), (160_001, 5)])  # chunks alone and in pairs
def test_sizes(nq, leaf):
    compare(clusters(50_001, 12, 3), clusters(nq, 12, 4), 10, leaf)


@pytest.mark.parametrize("k", [1, 10])
def test_ties(k):
    compare(lattice(40_000, 10, 5), lattice(25_001, 10, 6), k)


@pytest.mark.parametrize("scale,shift", [(1.0, 1000.0), (1e-11, 0.0), (1e12, 0.0), (1e-15, 0.0), (1e22, 0.0), (0.0, 3.0)])
def test_ranges(scale, shift):
    # (the last three extents are outside the block search's range)
    compare(clusters(30_000, 16, 7) * scale + shift, clusters(33_400, 16, 8) * scale + shift, 5)


@pytest.mark.parametrize("k", [1, 30])
def test_monochromatic(k):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    P = cuda(clusters(32_003, 16, 9))
    t = dtree.dtree_build(P, 32)
    try:
        idx, dist = dtree.dtree_kfn(None, t, k)
        # against the same points as queries of their own: no point is its own
        # furthest neighbour here, so the lists agree
        tq = dtree.dtree_build(P[:5_000], 32)
        i2, d2 = dtree.dtree_kfn(tq, t, k)
        tq.free()
    finally:
        t.free()
    assert torch.equal(idx[:5_000], i2) and torch.equal(dist[:5_000], d2)
