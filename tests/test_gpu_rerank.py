"""The tensor-core tile's re-rank in pairs of float32: distances that differ
in their last float32 bits, ties, zeros, and sums below and above the range in
which the pairs are trusted, against the float64 oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def near_ties(m, d, seed):
    # shells of points around a few centres: equal distances but for rounding
    g = np.random.default_rng(seed)
    c = g.normal(size=(6, d))
    u = g.normal(size=(m, d))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    return (c[g.integers(0, 6, m)] + u * (1 + 1e-7 * g.integers(0, 3, (m, 1)))).astype(np.float32), c.astype(np.float32)


@pytest.mark.parametrize("d", [3, 16, 33, 64])
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e9])
@pytest.mark.parametrize("precision", ["bf16", "tf32"])
@pytest.mark.parametrize("k", [1, 10, 49])
def test_rerank(d, scale, precision, k):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    R, C = near_ties(1500, d, d)
    g = np.random.default_rng(d + 1)
    Q = np.concatenate([C, R[:100], R[100:200] + np.float32(2 ** -12), g.normal(size=(100, d)).astype(np.float32)])
    R, Q = (R * np.float32(scale)).astype(np.float32), (Q * np.float32(scale)).astype(np.float32)
    i, dist = dtree.knn(torch.from_numpy(R).cuda(), torch.from_numpy(Q).cuda(), k, precision=precision)
    ti, td = oracle.knn_brute(R, Q, k)
    assert np.array_equal(i.cpu().numpy(), ti)
    assert np.array_equal(dist.cpu().numpy(), np.sqrt(td).astype(np.float32))
