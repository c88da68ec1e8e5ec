"""Tensor-core work items split over several CTAs: few queries against many
points, so that items are fewer than SMs and have from one to many windows of
candidates; equal to the float32 search."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


@pytest.mark.parametrize("nq,m,d", [(1, 40_000, 16), (129, 9_000, 16), (1_000, 300_000, 16), (4_097, 120_000, 64),
                                    (700, 100_000, 30), (5_000, 8_000, 3)])
@pytest.mark.parametrize("k,precision", [(1, "bf16"), (10, "bf16"), (18, "tf32"), (50, "bf16")])
def test_slices(nq, m, d, k, precision):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(nq + d)
    R, Q = cuda(g.normal(size=(m, d))), cuda(g.normal(size=(nq, d)))
    want = dtree.knn(R, Q, k)
    got = dtree.knn(R, Q, k, precision=precision)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_ties_across_slices():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(3)
    R, Q = cuda(g.integers(0, 3, size=(60_000, 8))), cuda(g.integers(0, 3, size=(900, 8)))
    want = dtree.knn(R, Q, 10)
    got = dtree.knn(R, Q, 10, precision="bf16")
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
