"""The tree at the sizes where the build's passes change: subtrees around a
power of two, one and several chunks per node, leaves of 1 to 1024 points.
Every node's box is tight and every split is the median of its widest
dimension."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf", [(2, 1), (63, 2), (64, 5), (65, 32), (129, 1), (1023, 16), (2048, 32), (2049, 20),
                                    (4097, 3), (8193, 1024), (20_011, 32), (262_145, 64)])
@pytest.mark.parametrize("d", [1, 3, 8, 16, 31, 64])
def test_splits_and_boxes(n, leaf, d):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    g = np.random.default_rng(n + d)
    P = g.normal(size=(n, d)).astype(np.float32)
    P[g.random(n) < 0.2, 0] = 0.5  # ties on a coordinate
    t = dtree.dtree_build(torch.from_numpy(P).cuda(), leaf)
    try:
        e = {k: v.cpu().numpy() for k, v in dtree.dtree_export(t).items()}
        leaves = t.leaves
    finally:
        t.free()
    assert np.array_equal(np.sort(e["perm"]), np.arange(n))
    X = P[e["perm"]]
    step = max(1, (2 * leaves - 1) // 500)  # a sample of the nodes, the top ones among them
    for i in sorted(set(range(0, min(63, 2 * leaves - 1))) | set(range(0, 2 * leaves - 1, step))):
        b, c = e["begin"][i], e["count"][i]
        pts = X[b:b + c]
        assert np.array_equal(e["box"][i, 0], pts.min(axis=0)) and np.array_equal(e["box"][i, 1], pts.max(axis=0))
        far = np.sqrt(((pts.astype(np.float64) - 0.5 * (e["box"][i, 0].astype(np.float64) + e["box"][i, 1])) ** 2).sum(1)).max()
        assert e["lambda"][i] >= far * (1 - 1e-6)
        if i < leaves - 1:
            left, right = 2 * i + 1, 2 * i + 2
            assert e["begin"][left] == b and e["count"][left] == c // 2
            assert e["begin"][right] == b + c // 2 and e["count"][right] == c - c // 2
            ext = e["box"][i, 1] - e["box"][i, 0]
            dim = int(np.argmax(ext))
            assert pts[:c // 2, dim].max() <= pts[c // 2:, dim].min()
