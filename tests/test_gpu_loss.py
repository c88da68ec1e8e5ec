"""The proposal network's loss: the mean over the rows, the same in every call
and not worse for their number."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dt():
    from paper_1304_4327_gb300 import build
    build.build()
    from paper_1304_4327_gb300 import dtree
    return dtree


def network(d, C, scale, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shapes = [(256, d), (256,), (256, 256), (256,), (C, 256), (C,)]
    return [torch.randn(s, generator=g, device="cuda") * scale for s in shapes], g


@pytest.mark.parametrize("n", [1, 255, 257, 4_095, 4_096])
@pytest.mark.parametrize("C", [2, 39, 47, 840])
def test_equal_rows(dt, n, C):
    # a network of zeros: every logit is zero, so every row's loss is log C, and
    # so is their mean.  logf is within an ulp; two more for the products and
    # the final rounding
    params, _ = network(3, C, 0.0, 1)
    T = torch.zeros(n, C, device="cuda")
    T[torch.arange(n), torch.arange(n) % C] = 1.0
    loss, _ = dt.dtree_mlp_loss_grad(params, torch.ones(n, 3, device="cuda"), T)
    assert abs(loss - math.log(C)) <= 3 * np.spacing(np.float32(math.log(C)))


def test_the_same_in_every_call(dt):
    params, g = network(8, 1_000, 0.05, 2)
    X = torch.randn(4_096, 8, generator=g, device="cuda")
    T = torch.softmax(4 * torch.randn(4_096, 1_000, generator=g, device="cuda"), 1)
    losses = {dt.dtree_mlp_loss_grad(params, X, T)[0] for _ in range(20)}
    assert len(losses) == 1
