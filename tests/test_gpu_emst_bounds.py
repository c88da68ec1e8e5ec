"""The spanning tree's bounds kept from round to round, where a float32 key
overflows although the squared length does not."""
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


def key(q, r):
    """The float32 key: fused multiply-adds in double, rounded once each."""
    s = np.float32(0)
    for a, b in zip(q, r):
        t = float(np.float32(a) - np.float32(b))
        with np.errstate(over="ignore"):
            s = np.float32(np.longdouble(t) * np.longdouble(t) + np.longdouble(float(s)))
    return s


def test_lengths_just_below_the_largest_float(dt):
    # Q-Y, Q-W and P-W have squared lengths just below the largest float, in this
    # order, and float32 keys that round to infinity.  Q and P are one component
    # after the first round and join Y's in the second (by Q-Y); in the third,
    # P's bound is finite (its answer, W, still leaves the component) and Q must
    # still be searched, whose edge to W is the shortest.
    Q = (0.0, 0.0, 0.0)
    P = (0.0, 0.0, -499999993495552.0)
    Y = (1.3441075551259329e+19, 1.2634073598890344e+19, 3862042645626880.0)
    W = (-1.31011505364161e+19, 1.298623068059258e+19, 3201935700131840.0)
    pts = np.array([Q, P, Y, (Y[0] * 1.01, Y[1], Y[2]), W, (W[0] * 1.01, W[1], W[2]),
                    (W[0] * 1.1, W[1], W[2]), (W[0] * 1.11, W[1], W[2])], dtype=np.float32)

    def d2(a, b):
        return float(((pts[a].astype(np.float64) - pts[b].astype(np.float64)) ** 2).sum())

    assert d2(0, 2) < d2(0, 4) < d2(1, 4) < min(d2(1, 2), float(np.finfo(np.float32).max))
    for a in (0, 1):
        for b in range(2, 8):
            assert np.isinf(key(pts[a], pts[b]))
    t = dt.dtree_build(torch.from_numpy(pts).cuda(), 32)
    try:
        e, dist = dt.dtree_emst(t)
    finally:
        t.free()
    te, td2 = oemst.canonical(*oemst.emst_kruskal(pts))
    ge, gd = oemst.canonical(e.cpu().numpy(), dist.cpu().numpy())
    assert np.array_equal(ge, te)
    assert np.array_equal(gd, np.sqrt(td2).astype(np.float32))
