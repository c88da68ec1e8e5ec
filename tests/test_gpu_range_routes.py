"""Which range searches go to the block search and which to a walk per query: the
walks keep those of few leaves and those of many results, where they are
faster.  Results are the same either way."""
import pytest
import torch

from test_gpu_kfn_routes import latent, mixture

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def ordered(off, idx, dist, m):
    rows = torch.repeat_interleave(torch.arange(off.numel() - 1, device=idx.device), off.diff())
    order = torch.argsort(rows * m + idx)
    return idx[order], dist[order]


def search(dt, R, Q, lo, hi, leaf=32):
    m = R.shape[0]
    assert m * Q.shape[0] >= 10 ** 9
    tr, tq = dt.dtree_build(R, leaf), dt.dtree_build(Q, leaf)
    off, idx, dist, st = dt.dtree_range(tq, tr, lo, hi, with_stats=True)
    t = dt.dtree_build(Q[:2_000], leaf)
    o, i, d = dt.dtree_range(t, tr, lo, hi)
    for x in (tr, tq, t):
        x.free()
    assert torch.equal(o, off[:2_001])
    n = int(o[-1])
    i, d = ordered(o, i, d, m)
    i2, d2 = ordered(o, idx[:n], dist[:n], m)
    assert torch.equal(i, i2) and torch.equal(d, d2)
    return st["query_blocks"] > 0


@pytest.mark.parametrize("d", [10, 16, 32, 64])
@pytest.mark.parametrize("dims,hi", [(2, 0.1), (3, 0.2), (4, 0.5)])
def test_low_intrinsic_dimension_walks(dt, d, dims, hi):
    s = (d / 16) ** 0.5  # (the maps' spread)
    assert not search(dt, latent(100_000, d, dims, 1), latent(20_000, d, dims, 2), 0.0, hi * s)


def test_many_points_within_the_range_walk(dt):
    R, Q = torch.randn(50_000, 16, device="cuda"), torch.randn(20_001, 16, device="cuda")
    assert not search(dt, R, Q, 0.0, 3.8)
    assert not search(dt, R, Q, 9.5, 20.0)  # few results, but nearly all points are nearer than 20


@pytest.mark.parametrize("d,hi", [(16, 2.0), (16, 2.7), (24, 4.0), (64, 8.0)])
@pytest.mark.parametrize("leaf", [16, 32, 700])
def test_the_mixture_goes_to_the_tiles(dt, d, hi, leaf):
    assert search(dt, mixture(100_000, d, 1), mixture(20_001, d, 2), 0.0, hi, leaf)
    assert search(dt, mixture(100_000, d, 1), mixture(20_001, d, 2), 0.75 * hi, hi, leaf)
