"""Loss and gradients of the proposal network where the products are sliced
along K: class and row counts around 8 and 128, and many chunks of K."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,C", [(1, 5, 1), (7, 2, 9), (127, 64, 127), (129, 16, 2055), (2049, 8, 130), (1500, 8, 3001)])
def test_sliced_products(n, d, C):
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    p = omlp.init(d, C, seed=n + C, scale=0.7)
    g = np.random.default_rng(n)
    X = g.normal(size=(n, d))
    T = g.random(size=(n, C)) * (g.random(size=(n, C)) < 0.05)
    T[:, 0] += 1e-3
    T /= T.sum(axis=1, keepdims=True)
    L, G = omlp.loss_grad(p, X, T)
    params = [torch.from_numpy(p[k].astype(np.float32)).cuda() for k in omlp.NAMES]
    Lg, grads = dtree.dtree_mlp_loss_grad(params, torch.from_numpy(X.astype(np.float32)).cuda(),
                                          torch.from_numpy(T.astype(np.float32)).cuda())
    # FP16 operands (2^-11 each) through three layers, float32 sums; a gradient
    # that is zero to rounding is held to the layer's scale
    assert abs(Lg - L) <= 5e-3 * max(abs(L), 1e-2)
    for name, gg in zip(omlp.NAMES, grads):
        err = np.linalg.norm(gg.cpu().numpy() - G[name]) / max(np.linalg.norm(G[name]), 1e-4)
        assert err < 3e-2, (name, err)
