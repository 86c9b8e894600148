"""The solve of the normal equations (double-float LDL^T, bt_ldlt.h) at the
sizes where its panels and row blocks change: one node (a single panel),
up to 32 rows (one warp a panel), 33 and more, and the largest system."""
import numpy as np
import pytest

import oracle as O
import synthgen as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_frames", [2, 3, 5, 6, 10, 11, 19, 24])
def test_step_solves_the_exported_system(n_frames):
    from paper_2108_00516_gb300 import build as lbuild
    lbuild.build()
    from paper_2108_00516_gb300 import bt
    g = S.random_graph(1300 + n_frames, n_frames, S.TINY_CAMERA, 60, 0.2)
    pg = bt.graph_from_synth(g)
    H, b, _ = pg.debug_normal_equations()
    n = 6 * (n_frames - 1)
    assert H.shape == (n, n)
    P, _ = pg.solve(1)
    pg.close()
    x = np.linalg.solve(H, -b)
    for _ in range(2):                                   # refined in extended precision
        r = -b.astype(np.longdouble) - H.astype(np.longdouble) @ x.astype(np.longdouble)
        x = x + np.linalg.solve(H, r.astype(np.float64))
    dx = np.concatenate([O.se3_log(np.linalg.solve(g.pose_init[k], P[k])) for k in range(1, n_frames)])
    # backward error of the factorisation and both substitutions: 3 n products
    # of 2^-44 each against the scaled system, amplified by its condition; the
    # update, its logarithm here and the poses themselves: 1e-13
    d = 1.0 / np.sqrt(np.diag(H))
    cond = np.linalg.cond(H * d[:, None] * d[None, :])
    err = np.linalg.norm((dx - x) / d) / np.linalg.norm(x / d)
    floor = 1e-13 * np.linalg.norm(1.0 / d) / np.linalg.norm(x / d)
    assert err <= 3 * n * cond * 2.0 ** -44 + floor, (err, cond)


@pytest.mark.parametrize("spread,n_frames", [(1.0, 4), (1e-1, 4), (1e-2, 4), (1e-2, 11), (1e-3, 18)])
def test_weakly_held_node(spread, n_frames):
    """One node is held only by points close to a line, down to systems whose
    smallest pivot the FP32 inverse does not take: the step still solves the
    exported system, to the same bound."""
    from paper_2108_00516_gb300 import build as lbuild
    lbuild.build()
    from paper_2108_00516_gb300 import bt
    rng = np.random.default_rng(int(1e4 * spread) + n_frames)
    blank = (np.zeros((8, 8), np.float32), np.zeros((8, 8, 3), np.float32), np.zeros((8, 8), np.uint8))
    T = [O.se3_exp(np.concatenate([[0, 0, 0.5], 0.1 * rng.normal(size=3)])) for _ in range(n_frames)]
    with bt.PoseGraph(dict(huber_sparse=1.0)) as pg:
        ids = []
        for k in range(n_frames):
            sets = []
            if k:
                x = 0.05 * rng.normal(size=(40, 3))
                if k == n_frames - 1:
                    x[:, 1:] *= spread
                at = [(x @ T[f][:3, :3].T + T[f][:3, 3]).astype(np.float32) for f in (k, k - 1)]
                sets = [(ids[-1], at[0] + np.float32(1e-4) * rng.normal(size=(40, 3)).astype(np.float32), at[1])]
            ids.append(pg.add_frame(*blank, (10.0, 10.0, 4.0, 4.0, 8, 8), T[k], k == 0, sets))
        H, b, _ = pg.debug_normal_equations()
        P, _ = pg.solve(1)
    n = 6 * (n_frames - 1)
    x = np.linalg.solve(H, -b)
    for _ in range(2):
        r = -b.astype(np.longdouble) - H.astype(np.longdouble) @ x.astype(np.longdouble)
        x = x + np.linalg.solve(H, r.astype(np.float64))
    dx = np.concatenate([O.se3_log(np.linalg.solve(T[k], P[k])) for k in range(1, n_frames)])
    d = 1.0 / np.sqrt(np.diag(H))
    cond = np.linalg.cond(H * d[:, None] * d[None, :])
    err = np.linalg.norm((dx - x) / d) / np.linalg.norm(x / d)
    floor = 1e-13 * np.linalg.norm(1.0 / d) / np.linalg.norm(x / d)
    assert err <= 3 * n * cond * 2.0 ** -44 + floor, (err, cond)
