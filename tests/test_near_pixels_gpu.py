"""16-bit target maps hold the depth as an offset from the frame's mean depth:
a valid pixel much nearer than that mean can come back as a depth that is not
positive, and is then no target (as in the FP32 map, whose depths are all
positive).  Pixels a few millimetres from the camera in a frame whose mean is
a metre away, seen by a frame that holds those pixels at full resolution."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, H = 40, 30
K = (30.0, 30.0, W / 2.0, H / 2.0, W, H)


@pytest.fixture(scope="module")
def bt():
    from paper_2108_00516_gb300 import build as lbuild
    lbuild.build()
    from paper_2108_00516_gb300 import bt as _bt
    _bt.load()
    return _bt


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_depths_that_decode_to_nothing_are_no_targets(bt, storage):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    normals = np.tile(np.float32([0, 0, -1]), (H, W, 1))
    mask = np.ones((H, W), np.uint8)
    near = rng.random((H, W)) < 0.2
    far_frame = np.where(near, np.exp(rng.uniform(np.log(5e-5), np.log(5e-3), (H, W))), 1.2).astype(np.float32)
    near_frame = np.full((H, W), 0.005, np.float32)
    zref = np.float32(far_frame.astype(np.float64).mean())
    if storage == "fp32":
        decoded = far_frame
    else:
        to = torch.float16 if storage == "fp16" else torch.bfloat16
        decoded = zref + torch.from_numpy(far_frame - zref).to(to).float().numpy()
    lost = near & (decoded <= 0)
    assert lost.any() == (storage != "fp32") and (near & (decoded > 0)).any()
    config = bt.config_default()
    config.precision = {"fp32": bt.BT_FP32, "fp16": bt.BT_FP16, "bf16": bt.BT_BF16}[storage]
    with bt.PoseGraph(config) as g:
        g.add_frame(near_frame, normals, mask, K, np.eye(4), True)
        g.add_frame(far_frame, normals, mask, K, np.eye(4), False)
        out = g.debug_associate(0, 1).reshape(H, W)
        energy = g.eval_cost()
        reverse = int((g.debug_associate(1, 0) >= 0).sum())
    # one camera, so that a source pixel looks up its own place; the targets
    # are all within the distance gate of 2 cm (both lie within 6 mm of the
    # camera, at most 0.7 of their depth off the axis), the far pixels outside it
    own = np.arange(W * H).reshape(H, W)
    assert np.array_equal(out, np.where(near & (decoded > 0), own, -1))
    assert energy["dense_inliers"] == int((out >= 0).sum()) + reverse
