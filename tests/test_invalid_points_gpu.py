"""Correspondences that are not finite: what they leave untouched stays
finite.  A point p that is NaN takes no part in the maxima of the warm start's
network (its layer-1 outputs are zero), so it has no part in the gradient; a
3-point sample with an infinite target point has no rotation and an infinite
translation."""
import numpy as np
import pytest

import oracle as O
import oracle.warmstart as W
import synthgen as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bt():
    from paper_2108_00516_gb300 import build as lbuild
    lbuild.build()
    from paper_2108_00516_gb300 import bt as _bt
    _bt.load()
    return _bt


def _set(rng, n, bad):
    """A set and its training pair of poses, and its features without the rows
    `bad`, whose p is NaN (their q counts towards the centre)."""
    p = (rng.normal(size=(n, 3)) * [0.04, 0.04, 0.03] + [0.0, 0.0, 0.45]).astype(np.float32)
    M = O.se3_exp(np.concatenate([0.02 * rng.normal(size=3), 0.1 * rng.normal(size=3)]))
    q = (p @ M[:3, :3].T + M[:3, 3] + rng.normal(scale=0.001, size=(n, 3))).astype(np.float32)
    M0 = O.se3_exp(np.concatenate([0.01 * rng.normal(size=3), 0.08 * rng.normal(size=3)])) @ M
    x, c = W.features(p, q, M0)
    p[bad] = np.nan
    return p, q, M0, M, np.delete(x, bad, axis=0), c


def _lead(P, x):
    """Smallest relative lead of a positive channel maximum over the runner-up."""
    L = W.unpack(P)
    h1 = W.bf16(np.maximum(x @ W.bf16(L["W1"]).T + L["b1"], 0))
    s = np.sort(np.maximum(h1 @ W.bf16(L["W2"]).T + L["b2"], 0), axis=0)
    pos = s[-1] > 0
    return np.min((s[-1] - s[-2])[pos] / s[-1][pos])


@pytest.mark.parametrize("n,bad", [(5, [0]), (130, [0, 64, 128])])
def test_nan_point_has_no_part_in_the_gradient(bt, n, bad):
    # layer-2 biases below zero: a row of zero layer-1 outputs, which the NaN
    # point's is, holds no positive maximum; some channels have none at all
    rng = np.random.default_rng(11)
    P = (S.warmstart_init(1) + rng.normal(scale=0.01, size=W.N_PARAMS)).astype(np.float32)
    offs = np.cumsum([0] + [int(np.prod(s)) for _, s in W.LAYERS])
    b2 = slice(offs[3], offs[4])
    P[b2] = -np.abs(P[b2]) - np.linspace(0.01, 3.0, offs[4] - offs[3], dtype=np.float32)
    # channel maxima that lead by far more than FP32 rounding, so that both
    # sides route the gradient to the same rows
    sets = []
    while len(sets) < 2:
        s = _set(rng, n, bad)
        if _lead(P, s[4]) > 2e-5:
            sets.append(s)
    ws = bt.WarmStart(P)
    for p, q, M0, M, _, _ in sets:
        ws.add_set(p, q, np.eye(4), M0, np.eye(4), M)
    loss, g = ws.gradient([0, 1])
    ws.close()
    lo, go = W.loss_and_grad(P.astype(np.float64), [s[4] for s in sets], [W.label(s[2], s[3], s[5]) for s in sets])
    assert any((W.forward(P, s[4])[1]["g"] == 0).any() for s in sets)
    # the bounds of the gradient's parity test
    assert abs(loss - lo) <= 1e-4 * lo
    for k, (name, _) in enumerate(W.LAYERS):
        a, b = g[offs[k]:offs[k + 1]].astype(np.float64), go[offs[k]:offs[k + 1]]
        assert np.isfinite(a).all(), name
        assert np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b), name


@pytest.mark.parametrize("value", [np.inf, -np.inf])
def test_infinite_target_point(bt, value):
    p = np.array([[0, 0, 0.5], [0.1, 0, 0.5], [0, 0.1, 0.5]], np.float32)
    q = p.copy()
    q[1, 0] = value
    M, count = bt.ransac(p, q, hypotheses=16, seed=1, inlier_dist=0.01, refine=False)
    assert count == 0 and np.array_equal(M[:3, :3], np.eye(3))
    # the centroid's first component is infinite, the others as they are
    assert M[0, 3] == value and np.abs(M[1:3, 3]).max() <= 4 * 2.0**-53
