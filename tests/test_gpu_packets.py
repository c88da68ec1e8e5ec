"""The spanning tree's walks by packets of points, at the sizes where a packet
can go wrong: node counts around 32, leaves of more than one packet,
and coordinates whose float32 squares underflow or overflow."""
import numpy as np
import pytest
import torch

from oracle import emst as oemst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


def cloud(n, d, scale, seed):
    return (np.random.default_rng(seed).normal(size=(n, d)) * scale).astype(np.float32)


CASES = [(31, 3, 32, 1.0), (33, 3, 32, 1.0), (65, 16, 64, 1.0), (700, 2, 300, 1.0), (1023, 8, 33, 1.0),
         (500, 64, 100, 1.0), (400, 3, 32, 1e-21), (400, 16, 8, 1e-25), (300, 4, 40, 3e19), (513, 5, 16, 1e30)]


@pytest.mark.parametrize("n,d,leaf,scale", CASES)
def test_emst_packets(dt, n, d, leaf, scale):
    P = cloud(n, d, scale, n + d)
    t = dt.dtree_build(cuda(P), leaf)
    try:
        e, dist = dt.dtree_emst(t)
    finally:
        t.free()
    te, td2 = oemst.canonical(*oemst.emst_kruskal(P))
    ge, gd = oemst.canonical(e.cpu().numpy(), dist.cpu().numpy())
    assert np.array_equal(ge, te)
    assert np.array_equal(gd, np.sqrt(td2).astype(np.float32))


@pytest.mark.parametrize("n", [20_000, 40_000, 80_000])  # four, two and one lanes per point on 152 SMs
def test_emst_packet_sizes(dt, n):
    # in the plane the tree is a subgraph of the Delaunay triangulation
    sp = pytest.importorskip("scipy.spatial")
    sparse = pytest.importorskip("scipy.sparse")
    P = np.random.default_rng(n).random((n, 2)).astype(np.float32)
    t = dt.dtree_build(cuda(P), 32)
    try:
        e, dist = dt.dtree_emst(t)
    finally:
        t.free()
    X = P.astype(np.float64)
    s = sp.Delaunay(X).simplices
    pairs = np.unique(np.sort(np.concatenate([s[:, [0, 1]], s[:, [1, 2]], s[:, [0, 2]]]), axis=1), axis=0)
    w = np.sqrt(((X[pairs[:, 0]] - X[pairs[:, 1]]) ** 2).sum(axis=1))
    tree = sparse.csgraph.minimum_spanning_tree(sparse.coo_matrix((w, (pairs[:, 0], pairs[:, 1])), shape=(n, n))).tocoo()
    want = np.sort(np.stack([tree.row, tree.col], axis=1), axis=1)
    want = want[np.lexsort((want[:, 1], want[:, 0]))]
    got = e.cpu().numpy()
    order = np.lexsort((got[:, 1], got[:, 0]))
    assert np.array_equal(got[order], want)
    ends = X[want]
    assert np.array_equal(dist.cpu().numpy()[order], np.sqrt(((ends[:, 0] - ends[:, 1]) ** 2).sum(axis=1)).astype(np.float32))
