"""k-furthest and range searches whose block search gives up: a diagnostic makes
its bounded waits run out, and the call must still return the result, from the
walks that served it before there were tiles."""
import pytest
import torch

from test_gpu_kfn_routes import mixture

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def with_stall(dt, f):
    dt.dtree_debug_tc_stall(True)
    try:
        return f()
    finally:
        dt.dtree_debug_tc_stall(False)


def test_furthest_neighbours(dt):
    tr, tq = dt.dtree_build(mixture(60_000, 16, 1)), dt.dtree_build(mixture(17_000, 16, 2))
    idx, dist, st = dt.dtree_kfn(tq, tr, 10, with_stats=True)
    assert st["query_blocks"] > 0  # (tiles, when nothing stalls)
    i, d, s = with_stall(dt, lambda: dt.dtree_kfn(tq, tr, 10, with_stats=True))
    assert s["query_blocks"] == 0
    assert torch.equal(i, idx) and torch.equal(d, dist)
    i, d = dt.dtree_kfn(tq, tr, 10)
    assert torch.equal(i, idx) and torch.equal(d, dist)


def test_range(dt):
    tr, tq = dt.dtree_build(mixture(100_000, 16, 1)), dt.dtree_build(mixture(20_001, 16, 2))

    def search():
        off, idx, dist, st = dt.dtree_range(tq, tr, 0.0, 2.5, with_stats=True)
        rows = torch.repeat_interleave(torch.arange(off.numel() - 1, device="cuda"), off.diff())
        order = torch.argsort(rows * tr.n + idx)
        return st["query_blocks"], off, idx[order], dist[order]

    blocks, *want = search()
    assert blocks > 0
    blocks, *got = with_stall(dt, search)
    assert blocks == 0 and all(torch.equal(x, y) for x, y in zip(got, want))
