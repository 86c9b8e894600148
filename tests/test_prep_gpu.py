"""Frame preparation (target map, compacted source list) at image sizes around
its blocks of 1024 pixels and past the largest grid of its second kernel: the
dense energy of two stored frames equals that of the raw frames
(bt_pair_dense_energy_noalloc, which prepares nothing)."""
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


def _frame(rng, w, h, share):
    depth = (0.5 + 0.002 * rng.normal(size=(h, w))).astype(np.float32)
    depth[rng.random((h, w)) < 0.05] = 0.0
    depth[rng.random((h, w)) < 0.02] = np.nan
    n = rng.normal(size=(h, w, 3)) * 0.2 + [0, 0, -1]
    n = (n / np.linalg.norm(n, axis=-1, keepdims=True)).astype(np.float32)
    n[rng.random((h, w)) < 0.05] = np.nan
    mask = (rng.random((h, w)) < share).astype(np.uint8) * 3
    return depth, n, mask


@pytest.mark.parametrize("w,h,share", [(1, 1, 1.0), (31, 33, 0.7), (32, 32, 1.0), (1025, 1, 0.5), (317, 243, 0.3),
                                       (640, 480, 0.0), (640, 480, 0.9), (1400, 1000, 0.6)])
def test_stored_frames_hold_the_raw_pixels(bt, w, h, share):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(w * 7 + h)
    K = (float(w), float(w), w / 2.0, h / 2.0, w, h)
    frames = [_frame(rng, w, h, share) for _ in range(2)]
    T = [np.eye(4), O.se3_exp(np.array([0.004, -0.003, 0.002, 0.01, -0.02, 0.015]))]
    with bt.PoseGraph() as g:
        for k in range(2):
            g.add_frame(*frames[k], K, T[k], k == 0)
        e = g.eval_cost()
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    dev = [[torch.from_numpy(x).cuda() for x in f] for f in frames]
    bt.pair_dense_energy_noalloc(*dev[0], K, T[0], *dev[1], K, T[1], out)
    torch.cuda.synchronize()
    assert e["dense_inliers"] == int(out[1])
    # sums of the same non-negative terms, grouped differently: FP32 within a
    # lane or tile, at most 64 + 8 additions deep
    assert abs(e["dense"] - float(out[0])) <= 72 * 2.0**-24 * float(out[0])
