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
