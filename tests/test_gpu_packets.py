"""Searches that walk the tree by packets of 32 points, at the sizes where a
packet can go wrong: node counts around 32, leaves of more than one packet,
and coordinates whose float32 squares underflow or overflow."""
import numpy as np
import pytest
import torch

from oracle import emst as oemst

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()


def cloud(n, d, scale, seed):
    return (np.random.default_rng(seed).normal(size=(n, d)) * scale).astype(np.float32)


CASES = [(31, 3, 32, 1.0), (33, 3, 32, 1.0), (65, 16, 64, 1.0), (700, 2, 300, 1.0), (1023, 8, 33, 1.0),
         (500, 64, 100, 1.0), (400, 3, 32, 1e-21), (400, 16, 8, 1e-25), (300, 4, 40, 3e19), (513, 5, 16, 1e30)]


@pytest.mark.parametrize("n,d,leaf,scale", CASES)
def test_emst_packets(dt, n, d, leaf, scale):
    P = cloud(n, d, scale, n + d)
    t = dt.dtree_build(cuda(P), leaf)
    try:
        e, dist = dt.dtree_emst(t)
    finally:
        t.free()
    te, td2 = oemst.canonical(*oemst.emst_kruskal(P))
    ge, gd = oemst.canonical(e.cpu().numpy(), dist.cpu().numpy())
    assert np.array_equal(ge, te)
    assert np.array_equal(gd, np.sqrt(td2).astype(np.float32))
