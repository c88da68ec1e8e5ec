"""k-furthest and range searches leave nothing in their trees: a second call makes
the same allocations as the first, and a kNN search after them the same as on a
fresh tree."""
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


def allocations(dt, f):
    n = dt._lib.dtree_alloc_count()
    st = f()[-1]
    return dt._lib.dtree_alloc_count() - n, st


@pytest.mark.parametrize("call", ["kfn", "range"])
def test_a_second_call_allocates_as_the_first(dt, call):
    R, Q = mixture(100_000, 16, 1), mixture(20_001, 16, 2)
    tr, tq = dt.dtree_build(R), dt.dtree_build(Q)
    search = {"kfn": lambda: dt.dtree_kfn(tq, tr, 10, with_stats=True),
              "range": lambda: dt.dtree_range(tq, tr, 0.0, 2.5, with_stats=True)}[call]
    first, st = allocations(dt, search)
    assert st["query_blocks"] > 0  # tiles: operand rows were made
    assert allocations(dt, search)[0] == first
    # the rows a kNN search keeps are its own
    fresh = dt.dtree_build(R)
    knn = lambda t: allocations(dt, lambda: dt.dtree_knn(tq, t, 10, precision="bf16", with_stats=True))[0]
    assert knn(tr) == knn(fresh)
    # and serve the later calls of either kind
    assert allocations(dt, search)[0] < first
