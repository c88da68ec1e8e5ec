"""Tensor-core work items of two chunks of 128 queries: blocks of 129 to 256
queries (and 512), enough of them that the pairs are taken, every list length
that allows it; equal to the float32 search, which the oracle checks."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


@pytest.mark.parametrize("nq,block", [(80_001, 256), (65_537, 256), (129 * 512, 200), (160_003, 512)])
@pytest.mark.parametrize("d,k,precision", [(3, 1, "bf16"), (16, 10, "bf16"), (27, 18, "tf32"), (64, 10, "bf16"), (64, 18, "tf32")])
def test_wide(nq, block, d, k, precision):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(nq + d)
    R, Q = cuda(g.normal(size=(2_531, d))), cuda(g.normal(size=(nq, d)))
    want = dtree.knn(R, Q, k)
    got = dtree.knn(R, Q, k, precision=precision, query_block=block)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_wide_batch():
    # problems of one chunk a block beside problems of two
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(5)
    P = [cuda(g.normal(size=(n, 8))) for n in (90_000, 127, 20_011, 255, 1)]
    P[-1] = cuda(g.normal(size=(40, 8)))
    T = [dtree.dtree_build(p, 32) for p in P]
    try:
        for prec in ("bf16", "tf32"):
            got = dtree.dtree_knn_batch([(None, t, 10, 256) for t in T], precision=prec)
            for t, (i, d) in zip(T, got):
                wi, wd = dtree.dtree_knn(None, t, 10)
                assert torch.equal(i, wi) and torch.equal(d, wd)
    finally:
        for t in T:
            t.free()
