"""Range search's segment offsets: the prefix sums' block edges (4096 counts
to a block) against the oracle's counts."""
import numpy as np
import pytest
import torch

from oracle import rangesearch as orange

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [1, 4095, 4096, 4097, 9001])
def test_offsets(nq):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(nq)
    R, Q = g.random((60, 2)).astype(np.float32), g.random((nq, 2)).astype(np.float32)
    tr, tq = dtree.dtree_build(torch.from_numpy(R).cuda(), 8), dtree.dtree_build(torch.from_numpy(Q).cuda(), 32)
    try:
        off, idx, _ = dtree.dtree_range(tq, tr, 0.1, 0.4)
    finally:
        tr.free()
        tq.free()
    to, ti, _ = orange.range_brute(R, Q, 0.1, 0.4)
    assert np.array_equal(off.cpu().numpy(), to)
    assert idx.numel() == len(ti)
