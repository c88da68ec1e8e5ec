"""k-furthest neighbours where the block search's candidate bands overflow: such
queries are searched again with float32 keys, and only those whose float32 band
overflows too in float64."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def search(dt, R, Q, k):
    """One call, and the same queries in calls too small for the block search."""
    assert R.shape[0] * Q.shape[0] >= 10 ** 9
    tr, tq = dt.dtree_build(R, 32), dt.dtree_build(Q, 32)
    idx, dist, st = dt.dtree_kfn(tq, tr, k, with_stats=True)
    for a in range(0, Q.shape[0], 4_000):
        t = dt.dtree_build(Q[a:a + 4_000], 32)
        i, d, s = dt.dtree_kfn(t, tr, k, with_stats=True)
        t.free()
        assert s["query_blocks"] == 0  # walks
        assert torch.equal(i, idx[a:a + 4_000]) and torch.equal(d, dist[a:a + 4_000])
    tr.free()
    tq.free()
    return st


@pytest.mark.parametrize("k", [1, 10, 40])
def test_queries_at_the_centre_of_a_sphere(dt, k):
    g = torch.Generator(device="cuda").manual_seed(k)
    R = torch.randn(40_001, 16, generator=g, device="cuda")
    R /= R.norm(dim=1, keepdim=True)
    Q = torch.randn(30_000, 16, generator=g, device="cuda") * 0.5
    Q[::100] *= 2e-4  # 300 queries whose squared distances differ by 2e-4 or so
    st = search(dt, R, Q, k)
    assert st["query_blocks"] > 0  # tiles
    # far more points than a list holds lie within a tile's band (some 1e-4 of
    # the extents squared), a few within float32's (6e-6)
    assert 200 <= st["fallback_queries"] <= 600
    assert st["fallback64_queries"] <= 30


def test_lists_too_short_for_the_band(dt):
    g = torch.Generator(device="cuda").manual_seed(63)
    R = torch.randn(50_000, 16, generator=g, device="cuda")
    Q = torch.randn(20_001, 16, generator=g, device="cuda")
    assert search(dt, R, Q, 50)["query_blocks"] > 0
    assert search(dt, R, Q, 51)["query_blocks"] == 0
    assert search(dt, R, Q, 63)["query_blocks"] == 0
