"""The float32 tile at the edges of its 32-point steps: reference counts
around a step and a stage, leaves of 1 to 33 points, lists of every length."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,leaf", [(31, 40), (32, 40), (33, 40), (65, 64), (513, 33), (1025, 5)])
@pytest.mark.parametrize("d", [2, 8, 16, 27, 64])
@pytest.mark.parametrize("k", [1, 7, 15, 23, 30])
def test_tile_steps(m, leaf, d, k):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(m * 64 + d)
    R = g.normal(size=(m, d)).astype(np.float32)
    Q = g.normal(size=(130, d)).astype(np.float32)
    i, dist = dtree.knn(torch.from_numpy(R).cuda(), torch.from_numpy(Q).cuda(), k, leaf_size=leaf)
    ti, td = oracle.knn_brute(R, Q, k)
    assert np.array_equal(i.cpu().numpy(), ti)
    assert np.array_equal(dist.cpu().numpy(), np.sqrt(td).astype(np.float32))
