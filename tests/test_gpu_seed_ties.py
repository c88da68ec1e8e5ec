"""Tie groups that lie wholly in a block's seed subtree: more points at the
k-th distance than the seed's list once held, the lowest indices among them
placed anywhere in the tree's order."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "bf16", "tf32"])
@pytest.mark.parametrize("copies,k", [(18, 10), (20, 5), (22, 3), (30, 15)])
def test_duplicates_inside_the_seed(precision, copies, k):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(copies)
    centres = (g.normal(size=(300, 6)) * 50).astype(np.float32)
    R = np.repeat(centres, copies, axis=0)[g.permutation(300 * copies)]
    Q = centres + np.float32(0.25)
    i, d = dtree.knn(torch.from_numpy(R).cuda(), torch.from_numpy(Q).cuda(), k, precision=precision)
    ti, td = oracle.knn_brute(R, Q, k)
    assert np.array_equal(i.cpu().numpy(), ti)
    assert np.array_equal(d.cpu().numpy(), np.sqrt(td).astype(np.float32))
