"""Which k-furthest problems go to the block search and which to a walk per query:
the walks keep points of low intrinsic dimension and bands wider than a list,
where they are faster.  Results are the same either way."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def latent(n, d, dims, seed):
    a = torch.randn(d, dims, generator=torch.Generator(device="cuda").manual_seed(dims), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(n, dims, generator=g, device="cuda") @ a.T + 0.01 * torch.randn(n, d, generator=g, device="cuda")


def mixture(n, d, seed):
    c = torch.rand(32, d, generator=torch.Generator(device="cuda").manual_seed(d), device="cuda") * 20 - 10
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, d, generator=g, device="cuda") + c[torch.randint(0, 32, (n,), generator=g, device="cuda")]


def sphere(n, d, seed):
    x = torch.randn(n, d, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
    return x / x.norm(dim=1, keepdim=True)


def repeated(n, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    base = torch.randint(0, 4, (50, d), generator=torch.Generator(device="cuda").manual_seed(0), device="cuda").float()
    return base[torch.randint(0, 50, (n,), generator=g, device="cuda")].contiguous()


def search(dt, R, Q, k, leaf=32):
    assert R.shape[0] * Q.shape[0] >= 10 ** 9
    tr, tq = dt.dtree_build(R, leaf), dt.dtree_build(Q, leaf)
    idx, dist, st = dt.dtree_kfn(tq, tr, k, with_stats=True)
    t = dt.dtree_build(Q[:2_000], leaf)
    i, d = dt.dtree_kfn(t, tr, k)
    for x in (tr, tq, t):
        x.free()
    assert torch.equal(i, idx[:2_000]) and torch.equal(d, dist[:2_000])
    return st["query_blocks"] > 0


@pytest.mark.parametrize("d", [10, 16, 32, 64])
@pytest.mark.parametrize("dims,k", [(2, 10), (3, 1), (3, 50), (4, 10)])
def test_low_intrinsic_dimension_walks(dt, d, dims, k):
    assert not search(dt, latent(100_000, d, dims, 1), latent(20_000, d, dims, 2), k)


@pytest.mark.parametrize("d,k", [(10, 1), (16, 10), (24, 18), (64, 10)])
@pytest.mark.parametrize("leaf", [12, 32, 700])
def test_the_mixture_goes_to_the_tiles(dt, d, k, leaf):
    assert search(dt, mixture(60_000, d, 1), mixture(17_000, d, 2), k, leaf)


def test_wide_bands_walk(dt):
    assert not search(dt, sphere(50_000, 16, 1), torch.randn(20_001, 16, device="cuda") * 1e-3, 10)
    assert not search(dt, repeated(60_000, 16, 1), repeated(20_000, 16, 2), 10)


def test_points_are_counted_not_leaves(dt):
    # 32 leaves of some 900 points each
    assert search(dt, mixture(30_000, 10, 5), mixture(40_000, 10, 6), 10, 1_000)
    assert not search(dt, latent(30_000, 10, 3, 5), latent(40_000, 10, 3, 6), 10, 1_000)


@pytest.mark.parametrize("nq,m", [(4_096, 250_000), (1_000_000, 1_010)])
def test_few_queries_and_few_references(dt, nq, m):
    # (1,010 points in 64 leaves: every leaf is scored)
    assert search(dt, mixture(m, 16, 3), mixture(nq, 16, 4), 5, 16)
