"""The block search of k-furthest neighbours and range searches: that it is what
runs at the sizes its tests are made for, and on query blocks of several chunks
of 128 (query leaves of more points), whole, odd and in pairs."""
import numpy as np
import pytest
import torch

from oracle import kfn as okfn
from oracle import rangesearch as orange
from test_gpu_kfn_routes import mixture
from test_gpu_kfn_tiles import clusters, cuda, lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def furthest(dt, R, Q, k, leaf, qleaf):
    """Tiles for the whole call, a walk for the same queries in small ones."""
    tr, tq = dt.dtree_build(R, leaf), dt.dtree_build(Q, qleaf)
    idx, dist, st = dt.dtree_kfn(tq, tr, k, with_stats=True)
    assert st["query_blocks"] > 0
    for a in range(0, Q.shape[0], 4_000):
        t = dt.dtree_build(Q[a:a + 4_000], qleaf)
        i, d, s = dt.dtree_kfn(t, tr, k, with_stats=True)
        t.free()
        assert s["query_blocks"] == 0
        assert torch.equal(i, idx[a:a + 4_000]) and torch.equal(d, dist[a:a + 4_000])
    tr.free()
    tq.free()
    return st["query_blocks"]


def within(dt, R, Q, lo, hi, leaf, qleaf):
    m = R.shape[0]
    tr, tq = dt.dtree_build(R, leaf), dt.dtree_build(Q, qleaf)
    off, idx, dist, st = dt.dtree_range(tq, tr, lo, hi, with_stats=True)
    assert st["query_blocks"] > 0
    for a in range(0, Q.shape[0], 9_000):
        t = dt.dtree_build(Q[a:a + 9_000], qleaf)
        o, i, d, s = dt.dtree_range(t, tr, lo, hi, with_stats=True)
        t.free()
        assert s["query_blocks"] == 0
        n0, n1 = int(off[a]), int(off[min(a + 9_000, Q.shape[0])])
        assert torch.equal(o, off[a:a + 9_001] - n0)
        rows = torch.repeat_interleave(torch.arange(o.numel() - 1, device="cuda"), o.diff())
        p, p2 = torch.argsort(rows * m + i), torch.argsort(rows * m + idx[n0:n1])
        assert torch.equal(i[p], idx[n0:n1][p2]) and torch.equal(d[p], dist[n0:n1][p2])
    tr.free()
    tq.free()
    return st["query_blocks"]


# 100,001 queries: 391 a block in 256 blocks (four chunks), 782 in 128 (seven), 196 in
# 512 (two); paired, as the pairs fill the GPU.  20,001: 625 in 32 (five), not paired
@pytest.mark.parametrize("nq,qleaf", [(100_001, 400), (100_001, 1_000), (100_001, 200), (20_001, 700)])
@pytest.mark.parametrize("d,k", [(16, 10), (33, 18), (64, 40)])
def test_furthest_neighbours_in_chunks(dt, nq, qleaf, d, k):
    furthest(dt, mixture(50_001, d, 1), mixture(nq, d, 2), k, 32, qleaf)


@pytest.mark.parametrize("nq,qleaf", [(100_001, 400), (100_001, 1_000), (20_001, 700)])
@pytest.mark.parametrize("d,lo,hi", [(16, 0.0, 2.4), (33, 5.0, 5.6), (64, 0.0, 8.5)])
def test_range_in_chunks(dt, nq, qleaf, d, lo, hi):
    within(dt, mixture(50_001, d, 1), mixture(nq, d, 2), lo, hi, 32, qleaf)


@pytest.mark.parametrize("d", [9, 16, 17, 33, 64])
@pytest.mark.parametrize("k", [1, 10, 18, 50])
def test_furthest_neighbours_of_clusters(dt, d, k):
    furthest(dt, cuda(clusters(30_011, d, 1)), cuda(clusters(33_333, d, 2)), k, 32, 32)


@pytest.mark.parametrize("nq,leaf", [(20_000, 20), (81_003, 64)])
def test_furthest_neighbours_of_clusters_by_size(dt, nq, leaf):
    furthest(dt, cuda(clusters(50_001, 12, 3)), cuda(clusters(nq, 12, 4)), 10, leaf, leaf)


def test_furthest_neighbours_tied(dt):
    furthest(dt, cuda(lattice(40_000, 16, 5)), cuda(lattice(25_001, 16, 6)), 1, 32, 32)


@pytest.mark.parametrize("d", [16, 17, 33, 64])
def test_range_of_clusters(dt, d):
    s = (2 * d) ** 0.5
    within(dt, cuda(clusters(30_011, d, 1)), cuda(clusters(33_333, d, 2)), 0.0, 0.5 * s, 32, 32)
    within(dt, cuda(clusters(30_011, d, 1)), cuda(clusters(33_333, d, 2)), 0.45 * s, 0.5 * s, 32, 32)


def test_range_ends_hit_exactly(dt):
    # integer points: many squared distances of exactly 4 and 9
    g = torch.Generator(device="cuda").manual_seed(5)
    R = torch.randint(0, 4, (40_000, 16), generator=g, device="cuda").float()
    Q = torch.randint(0, 4, (25_001, 16), generator=g, device="cuda").float()
    within(dt, R, Q, 2.0, 3.0, 32, 32)


@pytest.mark.parametrize("d,k,qleaf", [(16, 10, 32), (33, 1, 400), (64, 50, 32)])
def test_sampled_queries_against_the_oracle(dt, d, k, qleaf):
    R, Q = mixture(60_001, d, 3), mixture(100_001 if qleaf > 128 else 20_001, d, 4)
    pick = torch.arange(0, Q.shape[0], 1_571)
    rows, sample = R.cpu().numpy(), Q[pick.cuda()].cpu().numpy()
    tr, tq = dt.dtree_build(R, 32), dt.dtree_build(Q, qleaf)
    idx, dist, st = dt.dtree_kfn(tq, tr, k, with_stats=True)
    assert st["query_blocks"] > 0
    ti, td2 = okfn.kfn_brute(rows, sample, k)
    assert np.array_equal(idx[pick.cuda()].cpu().numpy(), ti)
    assert np.array_equal(dist[pick.cuda()].cpu().numpy(), np.sqrt(td2).astype(np.float32))
    lo, hi = 0.4 * (2 * d) ** 0.5, 0.5 * (2 * d) ** 0.5
    off, idx, dist, st = dt.dtree_range(tq, tr, lo, hi, with_stats=True)
    assert st["query_blocks"] > 0
    to, ti, td = orange.range_brute(rows, sample, lo, hi)
    off, idx, dist = off.cpu().numpy(), idx.cpu().numpy(), dist.cpu().numpy()
    for n, q in enumerate(pick.tolist()):
        i, e = idx[off[q]:off[q + 1]], dist[off[q]:off[q + 1]]
        order = np.argsort(i)
        assert np.array_equal(i[order], ti[to[n]:to[n + 1]])
        assert np.array_equal(e[order], td[to[n]:to[n + 1]].astype(np.float32))
    tr.free()
    tq.free()
