"""The closed-form fit of 3-point samples (bt_ransac with exactly three
points) against the SVD form, from well-shaped triangles to slivers, where the
largest eigenvalue of the quaternion matrix comes close to the next one."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bt():
    from paper_2108_00516_gb300 import build as lbuild
    lbuild.build()
    from paper_2108_00516_gb300 import bt as _bt
    _bt.load()
    return _bt


def _svd_fit(p, q):
    pc, qc = p.mean(0), q.mean(0)
    U, s, Vt = np.linalg.svd((p - pc).T @ (q - qc))
    d = np.sign(np.linalg.det(Vt.T @ U.T))
    R = Vt.T @ np.diag([1.0, 1.0, d]) @ U.T
    return R, qc - R @ pc, s


@pytest.mark.parametrize("scale", [1e-4, 1.0, 1e4])
@pytest.mark.parametrize("height", [1.0, 1e-1, 1e-2, 1e-3, 1e-4])
def test_three_point_fit_matches_svd(bt, height, scale):
    """Triangles of base 1 and the given height, the second one noisy and
    turned by up to half a turn.  The rotation is determined to about u times
    the largest over the second singular value of the cross-covariance (u =
    2^-53; 64 roundings allowed on each side)."""
    rng = np.random.default_rng(int(1e6 * height))
    for _ in range(24):
        w = rng.normal(size=3)
        w *= rng.uniform(0, np.pi) / np.linalg.norm(w)
        T = O.se3_exp(np.concatenate([rng.normal(size=3), w]))
        p = np.array([[0, 0, 0], [1, 0, 0], [rng.uniform(0.2, 0.8), height, 0]]) + 0.1 * height * rng.normal(size=(3, 3))
        p = ((p @ O.se3_exp(np.concatenate([np.zeros(3), rng.normal(size=3)]))[:3, :3].T) * scale).astype(np.float32)
        q = (p @ T[:3, :3].T + scale * (T[:3, 3] + 0.1 * height * rng.normal(size=(3, 3)))).astype(np.float32)
        M, count = bt.ransac(p, q, hypotheses=16, seed=1, inlier_dist=100.0 * scale, refine=False)
        assert count == 3
        R, t, s = _svd_fit(p.astype(np.float64), q.astype(np.float64))
        tol = 128 * 2.0**-53 * s[0] / s[1]
        assert np.abs(M[:3, :3] - R).max() <= tol, (height, scale, np.abs(M[:3, :3] - R).max(), tol)
        assert np.abs(M[:3, 3] - t).max() <= 4 * tol * scale
        assert np.abs(M[:3, :3] @ M[:3, :3].T - np.eye(3)).max() <= 64 * 2.0**-53


def test_coincident_target_points(bt):
    """No rotation to recover (zero cross-covariance): the identity, as before."""
    p = np.array([[0, 0, 0.5], [0.1, 0, 0.5], [0, 0.1, 0.5]], np.float32)
    q = np.tile(np.float32([0.1, 0.2, 0.5]), (3, 1))
    M, count = bt.ransac(p, q, hypotheses=16, seed=1, inlier_dist=10.0, refine=False)
    assert count == 3 and np.array_equal(M[:3, :3], np.eye(3))
