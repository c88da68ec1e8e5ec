"""The spanning tree where several lanes serve a point (eight, four and two on 152
SMs) and many warps lower the same components' bounds meanwhile: against Prim's
algorithm in float64, in every one of several calls."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def prim(points):
    p = points.double()
    n = p.shape[0]
    best = torch.full((n,), float("inf"), dtype=torch.float64, device="cuda")
    near = torch.zeros(n, dtype=torch.int64, device="cuda")
    out = torch.zeros(n, dtype=torch.bool, device="cuda")
    ends = torch.zeros(n, 2, dtype=torch.int64, device="cuda")
    cur = torch.zeros(1, dtype=torch.int64, device="cuda")
    inf = torch.full((), float("inf"), dtype=torch.float64, device="cuda")
    for t in range(1, n):
        out.index_fill_(0, cur, True)
        e = (p - p[cur]).square_().sum(1)
        closer = e < best
        best = torch.where(closer, e, best)
        near = torch.where(closer, cur, near)
        cur = torch.where(out, inf, best).argmin(0, keepdim=True)
        ends[t, :1] = near[cur]
        ends[t, 1:] = cur
    return ends[1:].sort(1).values


@pytest.mark.parametrize("n", [12_001, 24_001, 40_001])
def test_clusters(n):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = torch.Generator(device="cuda").manual_seed(n)
    c = torch.rand(8, 16, generator=g, device="cuda") * 20 - 10
    P = torch.randn(n, 16, generator=g, device="cuda") + c[torch.randint(0, 8, (n,), generator=g, device="cuda")]
    want = prim(P)
    want = want[torch.argsort(want[:, 0] * n + want[:, 1])]
    t = dtree.dtree_build(P, 32)
    try:
        for _ in range(5):
            e, _ = dtree.dtree_emst(t)
            assert torch.equal(e[torch.argsort(e[:, 0] * n + e[:, 1])], want)
    finally:
        t.free()
