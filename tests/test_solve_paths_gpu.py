"""The two ways of the dense solve (bt_ldlt.h) at the sizes where either
changes form: the FP32 inverse with corrections on both sides of each of its
shapes (up to 12, 30, 60, 96, 120 and 138 unknowns), and the FP64
factorisation, which takes the systems that the inverse declines.

A chain of frames, each held by the correspondence set with the one before it
and nothing else.  Where the points of the sets lie close to a line that is
oblique to the object's axes, the rotations about it are weakly held and no
scaling of the unknowns helps: the smallest pivot of the scaled system is
below 2^-10, which the inverse leaves to the factorisation."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

OBLIQUE = O.se3_exp(np.array([0, 0, 0, 0.7, -0.4, 1.1]))[:3, :3]
DECLINED = 2.0**-10


@pytest.fixture(scope="module")
def bt():
    from paper_2108_00516_gb300 import build as lbuild
    lbuild.build()
    from paper_2108_00516_gb300 import bt as _bt
    _bt.load()
    return _bt


def _chain(bt, seed, n_frames, spread):
    """A graph of n_frames views: points with the given spread about a line."""
    rng = np.random.default_rng(seed)
    blank = (np.zeros((8, 8), np.float32), np.zeros((8, 8, 3), np.float32), np.zeros((8, 8), np.uint8))
    T = [O.se3_exp(np.concatenate([[0, 0, 0.5], 0.1 * rng.normal(size=3)])) for _ in range(n_frames)]
    pg = bt.PoseGraph(dict(huber_sparse=1.0))
    ids = []
    for k in range(n_frames):
        sets = []
        if k:
            x = (0.05 * rng.normal(size=(40, 3)) * [1.0, spread, spread]) @ OBLIQUE.T
            at = [(x @ T[f][:3, :3].T + T[f][:3, 3]).astype(np.float32) for f in (k, k - 1)]
            sets = [(ids[-1], at[0] + np.float32(1e-4) * rng.normal(size=(40, 3)).astype(np.float32), at[1])]
        ids.append(pg.add_frame(*blank, (10.0, 10.0, 4.0, 4.0, 8, 8), T[k], k == 0, sets))
    return pg, T


def _smallest_pivot(H):
    """Of the system scaled as the library scales it: rows and columns by powers
    of two, the diagonal in [1, 4)."""
    s = np.exp2(-(np.floor(np.log2(np.diag(H))).astype(int) >> 1))
    A = H * s[:, None] * s[None, :]
    least = np.inf
    for k in range(len(A)):
        least = min(least, A[k, k])
        A[k + 1:, k + 1:] -= np.outer(A[k + 1:, k], A[k, k + 1:]) / A[k, k]
    return least


def _step_error(pg, T):
    """Relative error of one step in the scaled unknowns against the exported
    system solved in extended precision, its condition number, the smallest
    pivot, and what the update, its logarithm here and the poses themselves
    allow for (1e-13)."""
    H, b, _ = pg.debug_normal_equations()
    P, _ = pg.solve(1)
    x = np.linalg.solve(H, -b)
    for _ in range(3):
        r = -b.astype(np.longdouble) - H.astype(np.longdouble) @ x.astype(np.longdouble)
        x = x + np.linalg.solve(H, r.astype(np.float64))
    dx = np.concatenate([O.se3_log(np.linalg.solve(T[k], P[k])) for k in range(1, len(T))])
    d = 1.0 / np.sqrt(np.diag(H))
    norm = np.linalg.norm(x / d)
    return (np.linalg.norm((dx - x) / d) / norm, np.linalg.cond(H * d[:, None] * d[None, :]), _smallest_pivot(H),
            1e-13 * np.linalg.norm(1.0 / d) / norm)


@pytest.mark.parametrize("n_frames", [2, 3, 4, 6, 7, 11, 12, 14, 17, 18, 21, 22, 23, 24])
def test_inverse(bt, n_frames):
    pg, T = _chain(bt, 40 + n_frames, n_frames, 1.0)
    err, cond, pivot, floor = _step_error(pg, T)
    pg.close()
    assert pivot > DECLINED
    # corrections from a residual whose n products of double-float numbers are
    # good to 3 x 2^-44 each
    assert err <= 3 * 6 * (n_frames - 1) * cond * 2.0**-44 + floor, (err, cond)


@pytest.mark.parametrize("n_frames", [2, 3, 6, 7, 11, 12, 17, 18, 21, 22, 24])
def test_factorisation_of_declined_systems(bt, n_frames):
    """H = sum of d_k l_k l_k^T: a reciprocal of the pivot d_k that is off by
    1e-12 changes H by as much of that term, and so all of them by at most
    1e-12 |H|; the rest of the factorisation and the substitutions are FP64, 3 n
    products of 2^-53 each.  Both are amplified by the condition."""
    for seed in range(12):
        pg, T = _chain(bt, 1000 * seed + n_frames, n_frames, 1e-3)
        err, cond, pivot, floor = _step_error(pg, T)
        # the later iterations of a solve go straight to the factorisation:
        # three iterations at once, or one by one
        pg.set_poses(np.stack(T))
        many, rep = pg.solve(3)
        pg.set_poses(np.stack(T))
        costs = []
        for _ in range(3):
            single, rep1 = pg.solve(1)
            costs.append(rep1["cost_init"])
        pg.close()
        assert pivot < DECLINED and cond > 1e4, (seed, pivot, cond)
        assert err <= (3 * 6 * (n_frames - 1) * 2.0**-53 + 1e-12) * cond + floor, (seed, err, cond)
        assert np.array_equal(many, single) and list(rep["cost_per_iter"][:3]) == costs, seed
