"""What a program that tracks objects with this library has it do, as timed cases.

A case is a dict of plain values; `kind` names the call:

  solve   PoseGraph.set_poses + PoseGraph.solve on frames already stored
  track   one frame of an online tracker from host memory: add_frame with its
          correspondence sets, set_active, set_poses, solve, remove_frame
  build   a new PoseGraph from device-resident frames and sets, its energy, and its end
  batch   Batch.solve over many graphs of mixed size
  warm    Batch.solve_warm: learned warm start and a few iterations
  predict the warm-start network on many correspondence sets
  train   loss and gradient of the warm-start network over a minibatch
  ransac  PoseGraph.ransac_init
  pair    pair_dense_energy_noalloc on two raw device frames

Scenes follow the recipe of the repository's generator (box and ellipsoid,
1 mm depth noise, central-difference normals on smoothed depth, steps of up
to 10 degrees and 2 cm between views, correspondences with outliers, starts
5 degrees / 1 cm off), drawn here on the GPU so that a state is quick to make.

Poses leave `run` as float32, as a tracker hands them to its renderer or
controller: below that they hold the rounding of the single-precision
residual pass.  Energies are the Python floats of the reports.
"""
import math
from pathlib import Path

import numpy as np
import torch

import paper_2108_00516_gb300 as package
from paper_2108_00516_gb300 import bt

STORAGE = {"fp32": bt.BT_FP32, "bf16": bt.BT_BF16, "fp16": bt.BT_FP16}
MAX_DIST, MAX_DEG, HUBER = 0.02, 45.0, 0.005     # the default configuration
GRADS, FEATURES = (128, 256, 128), 6             # widths of the warm-start network


def listed():
    return [
        # the smallest graph in use (4 views, 160x120): launches and the one-block solve count
        dict(name="solve_tiny", kind="solve", n=4, width=160, height=120, cover=0.2, sets=200, iters=7, storage="fp32"),
        # the paper's graph: 9 keyframes and the current VGA frame, 10 iterations
        dict(name="solve_paper", kind="solve", n=10, width=640, height=480, cover=0.22, sets=500, iters=10,
             storage="fp32"),
        # one iteration at odd sizes with the maps stored in 16 bits
        dict(name="step_odd_fp16", kind="solve", n=7, width=317, height=243, cover=0.3, sets=333, iters=1,
             storage="fp16"),
        # one iteration of the largest graph of the batched workload: 20 close VGA views, 800 matches a pair
        dict(name="step_large", kind="solve", n=20, width=640, height=480, cover=0.38, sets=800, iters=1,
             storage="fp32"),
        # an online tracker's frame, from host buffers to poses
        dict(name="track_frame", kind="track", n=10, width=640, height=480, cover=0.22, sets=500, iters=10,
             storage="fp32"),
        # a graph made from frames that another GPU stage produced
        dict(name="build_graph", kind="build", n=6, width=640, height=480, cover=0.25, sets=500, iters=0,
             storage="fp32"),
        # offline refinement of many tracks: 64 graphs of 3..20 views, QVGA and VGA
        dict(name="batch_mixed", kind="batch", n=64, width=640, height=480, cover=0.225, sets=450, iters=10,
             storage="fp32"),
        # the same with the learned warm start, which needs 2 iterations
        dict(name="batch_warm", kind="warm", n=32, width=640, height=480, cover=0.225, sets=450, iters=2,
             storage="fp32"),
        # network inference over the sets of a batch of graphs
        dict(name="predict_sets", kind="predict", n=2048, width=0, height=0, cover=0.0, sets=450, iters=0,
             storage="fp32"),
        # a training minibatch (train_step runs these passes and then one elementwise Adam kernel)
        dict(name="train_batch", kind="train", n=256, width=0, height=0, cover=0.0, sets=450, iters=0,
             storage="fp32"),
        # coarse initialisation of a paper-sized graph
        dict(name="ransac_graph", kind="ransac", n=10, width=160, height=120, cover=0.2, sets=500, iters=256,
             storage="fp32"),
        # dense energy of two VGA frames inside another framework's memory budget
        dict(name="pair_energy", kind="pair", n=2, width=640, height=480, cover=0.25, sets=0, iters=0,
             storage="fp32"),
    ]


def _between(rng, lo, hi):
    """A whole number in lo..hi, spread over the logarithm of the range."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["track", "track", "build", "batch", "batch", "warm", "predict", "train",
                                       "ransac", "pair"])
    storage = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16"])
    width = _between(rng, 96, 640)
    case = dict(kind=kind, n=_between(rng, 2, 20), width=width, height=max(72, int(width * rng.uniform(0.65, 0.85))),
                cover=round(rng.uniform(0.05, 0.4), 3), sets=_between(rng, 100, 800), iters=rng.randint(1, 3),
                storage=storage)
    if kind == "track":
        case["n"] = rng.randint(3, 12)
    elif kind == "build":
        case.update(n=rng.randint(2, 10), iters=0)
    elif kind in ("batch", "warm"):
        case.update(n=_between(rng, 4, 40), iters=2 if kind == "warm" else rng.randint(1, 4))
    elif kind in ("predict", "train"):
        case.update(n=_between(rng, 16, 3000) if kind == "predict" else _between(rng, 8, 400), width=0, height=0,
                    cover=0.0, iters=0, storage="fp32")
    elif kind == "ransac":
        case.update(n=rng.randint(3, 16), width=160, height=120, cover=0.2, iters=_between(rng, 64, 1024),
                    storage="fp32")
    elif kind == "pair":
        case.update(n=2, sets=0, iters=0, storage="fp32")
    return case


# ------------------------------------------------------------------ scenes

def _unit(rng):
    v = rng.normal(size=3)
    return v / np.linalg.norm(v)


def _rotation(axis, angle):
    x, y, z = axis
    K = np.array([[0, -z, y], [z, 0, -x], [-y, x, 0]])
    return np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * (K @ K)


def _pose(R, t):
    T = np.eye(4)
    T[:3, :3], T[:3, 3] = R, t
    return T


class Scene:
    """n views of one object: poses, intrinsics, depth / normals / mask (CUDA)
    and the correspondence sets of every pair i < j, (n_pairs, sets, 3) each."""

    def __init__(self, n, width, height, cover, sets, outliers, seed, key):
        self.n, self.width, self.height = n, width, height
        rng = np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed), int(key)])))
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(rng.integers(1 << 62)))
        f = 600.0 * width / 640.0 if width >= 240 else 140.0 * width / 160.0
        self.intrinsics = (f, f, width / 2.0, height / 2.0, width, height)
        box, axes, offset = rng.uniform(0.03, 0.08, 3), rng.uniform(0.02, 0.06, 3), rng.uniform(-0.04, 0.04, 3)
        self.object = [torch.tensor(x, device="cuda", dtype=torch.float32) for x in (box, axes, offset)]
        R = _rotation(_unit(rng), rng.uniform(0, math.pi))
        dist = self._distance(R, cover)
        home = np.array([0.0, 0.0, dist])
        poses = [_pose(R, home)]
        for _ in range(1, n):
            R, t = poses[-1][:3, :3], poses[-1][:3, 3]
            step = rng.uniform(0, 0.02) * _unit(rng)
            t = t + step if np.linalg.norm(t + step - home) <= 0.03 else t - step
            poses.append(_pose(_rotation(_unit(rng), math.radians(rng.uniform(0, 10))) @ R, t))
        self.true = np.stack(poses)
        self.start = self.true.copy()
        for k in range(1, n):
            dR = _rotation(_unit(rng), math.radians(5.0))
            self.start[k] = _pose(dR @ self.true[k, :3, :3], self.true[k, :3, 3] + 0.01 * _unit(rng))
        clean = self._cast(self.true, width, height, self.intrinsics)
        hit = torch.isfinite(clean)
        noise = 0.001 * torch.randn(clean.shape, generator=gen, device="cuda")
        self.depth = torch.where(hit, (clean + noise).clamp_min(1e-3), torch.zeros_like(clean))
        self.mask = hit.to(torch.uint8)
        self.normals = self._normals(max(1, width // 160))
        self.pairs = [(i, j) for i in range(n) for j in range(i + 1, n)]
        self.pts_i = self.pts_j = None
        if sets > 0:
            self._matches(clean, hit, sets, outliers, gen)

    def _cast(self, poses, W, H, K):
        """Depth of the object along every pixel's ray (inf where it misses)."""
        fx, fy, cx, cy = K[:4]
        v, u = torch.meshgrid(torch.arange(H, device="cuda", dtype=torch.float32),
                              torch.arange(W, device="cuda", dtype=torch.float32), indexing="ij")
        rays = torch.stack([(u - cx) / fx, (v - cy) / fy, torch.ones_like(u)], -1)
        T = torch.tensor(np.asarray(poses), device="cuda", dtype=torch.float32)
        d = torch.einsum("hwc,ncd->nhwd", rays, T[:, :3, :3])
        o = -torch.einsum("nc,ncd->nd", T[:, :3, 3], T[:, :3, :3])[:, None, None, :]
        box, axes, offset = self.object
        inv = 1.0 / torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
        a, b = (-box - o) * inv, (box - o) * inv
        near, far = torch.minimum(a, b).amax(-1), torch.maximum(a, b).amin(-1)
        inf = torch.full_like(near, math.inf)
        best = torch.where((far >= near) & (near > 0), near, inf)
        d2, o2 = d / axes, (o - offset) / axes
        qa, qb, qc = (d2 * d2).sum(-1), 2 * (d2 * o2).sum(-1), (o2 * o2).sum(-1) - 1
        disc = qb * qb - 4 * qa * qc
        s = torch.where(disc >= 0, (-qb - disc.clamp_min(0).sqrt()) / (2 * qa), inf)
        return torch.minimum(best, torch.where(s > 0, s, inf))

    def _distance(self, R, cover):
        """The distance at which the object covers about `cover` of the image."""
        ds = np.linspace(0.2, 1.6, 48)
        f = self.intrinsics[0] * 80.0 / self.width
        h = max(1, round(80 * self.height / self.width))
        seen = torch.isfinite(self._cast(np.stack([_pose(R, [0, 0, d]) for d in ds]), 80, h, (f, f, 40.0, h / 2.0)))
        share = seen.float().mean((1, 2)).tolist()
        return float(ds[min(range(len(ds)), key=lambda k: abs(share[k] - cover))])

    def _normals(self, k):
        """Central differences over +-k pixels of the smoothed, back-projected depth."""
        valid = self.mask.float()[:, None]
        z = self.depth[:, None]
        if k > 1:
            pool = torch.nn.functional.avg_pool2d
            den = pool(valid, 2 * k - 1, 1, k - 1)
            z = torch.where(valid > 0, pool(z, 2 * k - 1, 1, k - 1) / den.clamp_min(1e-9), torch.zeros_like(z))
        z = z[:, 0]
        P = self._backproject(z)
        ok = valid[:, 0] > 0
        out = torch.full(P.shape, math.nan, device="cuda")
        du = P[:, k:-k, 2 * k:] - P[:, k:-k, :-2 * k]
        dv = P[:, 2 * k:, k:-k] - P[:, :-2 * k, k:-k]
        m = torch.linalg.cross(dv, du)
        good = (ok[:, k:-k, k:-k] & ok[:, k:-k, 2 * k:] & ok[:, k:-k, :-2 * k] & ok[:, 2 * k:, k:-k]
                & ok[:, :-2 * k, k:-k])
        length = m.norm(dim=-1, keepdim=True)
        good &= length[..., 0] > 0
        m = m / length.clamp_min(1e-30)
        m = torch.where(((m * P[:, k:-k, k:-k]).sum(-1) > 0)[..., None], -m, m)
        out[:, k:-k, k:-k] = torch.where(good[..., None], m, torch.full_like(m, math.nan))
        return out.contiguous()

    def _backproject(self, z):
        fx, fy, cx, cy, W, H = self.intrinsics
        v, u = torch.meshgrid(torch.arange(H, device="cuda", dtype=z.dtype),
                              torch.arange(W, device="cuda", dtype=z.dtype), indexing="ij")
        return torch.stack([(u - cx) * z / fx, (v - cy) * z / fy, z], -1)

    def _matches(self, clean, hit, count, outliers, gen):
        """For every pair, `count` noisy surface points that both views see
        (repeated where fewer than that do), a share of them outliers."""
        fx, fy, cx, cy, W, H = self.intrinsics
        n, P = self.n, len(self.pairs)
        i = torch.tensor([p[0] for p in self.pairs], device="cuda")
        j = torch.tensor([p[1] for p in self.pairs], device="cuda")
        surface = self._backproject(torch.where(hit, clean, torch.zeros_like(clean))).reshape(n, -1, 3)
        flat = hit.reshape(n, -1)
        order = torch.argsort(flat.to(torch.int8), dim=1, descending=True, stable=True)     # masked pixels first
        masked = flat.sum(1).clamp_min(1)
        tries = 4 * count

        def points(node):
            r = torch.rand(P, tries, generator=gen, device="cuda")
            k = (r * masked[node][:, None]).long().clamp_max(H * W - 1)
            pix = torch.gather(order[node], 1, torch.minimum(k, masked[node][:, None] - 1))
            return torch.gather(surface[node], 1, pix[..., None].expand(-1, -1, 3))

        M = np.stack([self.true[q] @ np.linalg.inv(self.true[p]) for p, q in self.pairs])
        M = torch.tensor(M, device="cuda", dtype=torch.float32)
        pi = points(i)
        pj = pi @ M[:, :3, :3].transpose(1, 2) + M[:, None, :3, 3]
        u, v = (pj[..., 0] / pj[..., 2] * fx + cx).round().long(), (pj[..., 1] / pj[..., 2] * fy + cy).round().long()
        inside = (u >= 0) & (u < W) & (v >= 0) & (v < H)
        at = torch.where(inside, v * W + u, torch.zeros_like(u))
        seen = torch.gather(clean.reshape(n, -1)[j], 1, at)
        visible = inside & ((seen - pj[..., 2]).abs() < 0.005)
        first = torch.argsort(visible.to(torch.int8), dim=1, descending=True, stable=True)
        number = visible.sum(1).clamp_min(1)
        pick = torch.gather(first, 1, torch.arange(count, device="cuda")[None, :] % number[:, None])[..., None]
        pi, pj = torch.gather(pi, 1, pick.expand(-1, -1, 3)), torch.gather(pj, 1, pick.expand(-1, -1, 3))
        bad = torch.rand(P, count, generator=gen, device="cuda") < outliers
        pj = torch.where(bad[..., None], points(j)[:, :count], pj)
        self.pts_i = pi + 0.001 * torch.randn(pi.shape, generator=gen, device="cuda")
        self.pts_j = pj + 0.001 * torch.randn(pj.shape, generator=gen, device="cuda")

    def sets_of(self, k, ids):
        """The sets between frame k and the frames before it, as add_frame takes them."""
        if self.pts_i is None:
            return []
        return [(ids[i], self.pts_j[p], self.pts_i[p]) for p, (i, j) in enumerate(self.pairs) if j == k]

    def fill(self, graph, upto=None):
        ids = []
        for k in range(self.n if upto is None else upto):
            ids.append(graph.add_frame(self.depth[k], self.normals[k], self.mask[k], self.intrinsics, self.start[k],
                                       k == 0, self.sets_of(k, ids)))
        return ids


def _scene(case, seed, key=0):
    return Scene(case["n"], case["width"], case["height"], case["cover"], case["sets"], 0.2, seed, key)


def _scenes(case, seed):
    """The graphs of a batch: 3..20 views, full or half size, their own cover, sets and outliers."""
    rng = np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed), 99])))
    sizes = np.random.Generator(np.random.PCG64(4000))     # a batch's mix of sizes belongs to the case
    out = []
    for k in range(case["n"]):
        views, half = int(sizes.integers(3, 21)), bool(sizes.random() < 0.5)
        w, h = (case["width"] // 2, case["height"] // 2) if half else (case["width"], case["height"])
        cover, sets = case["cover"] * sizes.uniform(0.4, 1.6), int(case["sets"] * sizes.uniform(0.3, 1.7))
        out.append(Scene(views, w, h, cover, max(1, sets), float(rng.uniform(0.1, 0.3)), seed, k + 1))
    return out


def _weights():
    return np.load(Path(package.__file__).parent / "weights" / "warmstart.npz")["params"].astype(np.float32)


def _set_counts(case):
    """Points of each correspondence set: a fifth to twice the case's figure, ragged."""
    rng = np.random.Generator(np.random.PCG64(6000))
    return [max(1, int(case["sets"] * x)) for x in rng.uniform(0.2, 1.8, case["n"])]


def _point_sets(case, seed):
    """Many sets p, q with q close to M p, their poses as they start and as a solve left them (CUDA points)."""
    rng = np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed), 7])))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(rng.integers(1 << 62)))
    out = []
    for n in _set_counts(case):
        Ti = _pose(_rotation(_unit(rng), rng.uniform(0, math.pi)), [0, 0, rng.uniform(0.35, 0.6)])
        Tj = _pose(_rotation(_unit(rng), math.radians(rng.uniform(0, 20))) @ Ti[:3, :3],
                   Ti[:3, 3] + rng.uniform(0, 0.02) * _unit(rng))
        S = _pose(_rotation(_unit(rng), math.radians(5.0)) @ Tj[:3, :3], Tj[:3, 3] + 0.01 * _unit(rng))
        x = (torch.rand(n, 3, generator=gen, device="cuda") - 0.5) * 0.12
        noise = 0.001 * torch.randn(2, n, 3, generator=gen, device="cuda")
        bad = torch.rand(n, 1, generator=gen, device="cuda") < 0.2
        y = torch.where(bad, x.flip(0), x)
        A, B = (torch.tensor(T, device="cuda", dtype=torch.float32) for T in (Ti, Tj))
        out.append((x @ A[:3, :3].T + A[:3, 3] + noise[0], y @ B[:3, :3].T + B[:3, 3] + noise[1], Ti, S, Ti, Tj))
    return out


# ------------------------------------------------------------------ states

def _graph(case):
    return bt.PoseGraph(dict(precision=STORAGE[case["storage"]]), stream=torch.cuda.current_stream())


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind in ("solve", "ransac"):
        scene = _scene(case, seed)
        state["graph"] = _graph(case)
        scene.fill(state["graph"])
        state["start"] = scene.start
        torch.cuda.synchronize()
    elif kind == "track":
        scene = _scene(case, seed)
        n = case["n"]
        state["graph"] = _graph(case)
        state["ids"] = scene.fill(state["graph"], n - 1)
        state["start"] = scene.start

        def pinned(x):
            return x.contiguous().cpu().pin_memory().numpy()

        state["frame"] = [pinned(x[n - 1]) for x in (scene.depth, scene.normals, scene.mask)]
        state["intrinsics"] = scene.intrinsics
        state["sets"] = [(i, pinned(a), pinned(b)) for i, a, b in scene.sets_of(n - 1, state["ids"])]
        torch.cuda.synchronize()
    elif kind == "build":
        state["scene"] = _scene(case, seed)
    elif kind in ("batch", "warm"):
        scenes = _scenes(case, seed)
        state["graphs"] = [_graph(case) for _ in scenes]
        state["starts"] = [s.start for s in scenes]
        state["batch"] = bt.Batch(stream=None)
        for s, g in zip(scenes, state["graphs"]):
            s.fill(g)
            state["batch"].add(g)
        if kind == "warm":
            state["network"] = bt.WarmStart(_weights())
        torch.cuda.synchronize()
    elif kind in ("predict", "train"):
        state["network"] = bt.WarmStart(_weights())
        sets = _point_sets(case, seed)
        torch.cuda.synchronize()
        for p, q, *poses in sets:
            state["network"].add_set(p, q, *poses)
        state["ids"] = np.arange(case["n"], dtype=np.int32)
    else:
        state["scene"] = _scene(case, seed)
        state["out"] = torch.zeros(2, dtype=torch.float64, device="cuda")
    return state


def _answer(poses, report):
    return dict(poses=poses.astype(np.float32), cost_init=report["cost_init"], cost_final=report["cost_final"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        state["graph"].set_poses(state["start"])
        return _answer(*state["graph"].solve(case["iters"]))
    if kind == "track":
        g = state["graph"]
        new = g.add_frame(*state["frame"], state["intrinsics"], state["start"][-1], False, state["sets"])
        g.set_active(state["ids"] + [new])
        g.set_poses(state["start"])
        answer = _answer(*g.solve(case["iters"]))
        g.remove_frame(new)
        return answer
    if kind == "build":
        with _graph(case) as g:
            state["scene"].fill(g)
            return g.eval_cost()
    if kind in ("batch", "warm"):
        for g, start in zip(state["graphs"], state["starts"]):
            g.set_poses(start)
        if kind == "batch":
            reports = state["batch"].solve(case["iters"])
        else:
            reports = state["batch"].solve_warm(state["network"], case["iters"], 10)
        poses = np.concatenate([g.get_poses() for g in state["graphs"]]).astype(np.float32)
        return dict(poses=poses, cost_init=np.float32([r["cost_init"] for r in reports]),
                    cost_final=np.float32([r["cost_final"] for r in reports]))
    if kind == "predict":
        return state["network"].predict(state["ids"])
    if kind == "train":
        loss, gradient = state["network"].gradient(state["ids"])
        return dict(loss=loss, gradient=gradient)
    if kind == "ransac":
        g = state["graph"]
        g.set_poses(state["start"])
        g.ransac_init(case["iters"], seed=1)
        return g.get_poses()
    s = state["scene"]
    bt.pair_dense_energy_noalloc(s.depth[0], s.normals[0], s.mask[0], s.intrinsics, s.start[0], s.depth[1],
                                 s.normals[1], s.mask[1], s.intrinsics, s.start[1], state["out"],
                                 stream=torch.cuda.current_stream())
    return state["out"]


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Bytes: every input read once (of the maps, the object's pixels), every
    output written once.  Flops: about 120 for a pixel pair of a Gauss-Newton
    pass, 50 for one of an energy pass, 80 for a correspondence."""
    kind = case["kind"]
    if kind in ("predict", "train"):
        points = sum(_set_counts(case))
        params = sum(a * b for a, b in zip((FEATURES,) + GRADS, GRADS + (FEATURES,)))
        layers = 2 * points * (FEATURES * GRADS[0] + GRADS[0] * GRADS[1]) + 2 * case["n"] * GRADS[1] * GRADS[2]
        back = 4 * case["n"] * params if kind == "train" else 0
        return {"bytes": 24 * points + 2 * params + (4 * params if kind == "train" else 24 * case["n"]),
                "flops": layers + back}
    if kind == "ransac":
        sets = case["n"] - 1
        return {"bytes": sets * (24 * case["sets"] + 96), "flops": sets * case["iters"] * (26 * case["sets"] + 2000)}
    if kind in ("batch", "warm"):
        sizes = np.random.Generator(np.random.PCG64(4000))
        graphs = []
        for _ in range(case["n"]):
            views, half = int(sizes.integers(3, 21)), bool(sizes.random() < 0.5)
            pixels = case["width"] * case["height"] // (4 if half else 1)
            graphs.append((views, pixels * case["cover"] * sizes.uniform(0.4, 1.6),
                           int(case["sets"] * sizes.uniform(0.3, 1.7))))
    else:
        graphs = [(case["n"], case["width"] * case["height"] * case["cover"], case["sets"])]
    full = case["iters"]
    energy = 1
    per_pixel = 17 if case["storage"] == "fp32" or kind in ("track", "build", "pair") else 8
    total = {"bytes": 0.0, "flops": 0.0}
    for views, pixels, sets in graphs:
        pairs = views * (views - 1)
        total["bytes"] += views * pixels * per_pixel + pairs // 2 * sets * 24 + views * 256
        total["flops"] += (120 * full + 50 * energy) * pairs * pixels + 80 * (full + energy) * pairs // 2 * sets
        total["flops"] += full * 2 * (6 * (views - 1)) ** 3 / 6
    if kind == "warm":
        points = sum(v * (v - 1) // 2 * s for v, _, s in graphs)
        total["flops"] += 2 * points * (FEATURES * GRADS[0] + GRADS[0] * GRADS[1])
    return total


# ------------------------------------------------------------------ the same in 64 bits

def _adjoint(T):
    A = torch.zeros(6, 6, dtype=torch.float64, device="cuda")
    R, t = T[:3, :3], T[:3, 3]
    A[:3, :3] = A[3:, 3:] = R
    A[:3, 3:] = _skew(t) @ R
    return A


def _skew(w):
    o = torch.zeros((), dtype=torch.float64, device="cuda")
    return torch.stack([o, -w[2], w[1], w[2], o, -w[0], -w[1], w[0], o]).reshape(3, 3)


def _huber(r):
    return torch.where(r <= HUBER, 0.5 * r * r, HUBER * (r - 0.5 * HUBER)), HUBER / r.clamp_min(HUBER)


class Exact:
    """The pose graph of a scene in 64 bits: energy and one Gauss-Newton step."""

    def __init__(self, scene):
        self.s = scene
        ok = (scene.mask > 0) & (scene.depth > 0) & torch.isfinite(scene.normals).all(-1)
        self.ok = ok.reshape(scene.n, -1)
        self.z = scene.depth.double().reshape(scene.n, -1)
        self.normal = scene.normals.double().reshape(scene.n, -1, 3)
        self.P = scene._backproject(scene.depth.double()).reshape(scene.n, -1, 3)

    def system(self, T, full):
        """(E_dense, E_sparse, accepted, H, g) for right perturbations of every node."""
        s = self.s
        fx, fy, cx, cy, W, Hh = s.intrinsics
        H = torch.zeros(s.n, s.n, 6, 6, dtype=torch.float64, device="cuda")
        g = torch.zeros(s.n, 6, dtype=torch.float64, device="cuda")
        dense, sparse, accepted = 0.0, 0.0, 0
        points = [(self.P[k][self.ok[k]], self.normal[k][self.ok[k]]) for k in range(s.n)]
        for i in range(s.n):
            for j in range(s.n):
                if i == j:
                    continue
                M = T[j] @ torch.linalg.inv(T[i])
                p, n = points[i]
                q, n = p @ M[:3, :3].T + M[:3, 3], n @ M[:3, :3].T
                u = torch.floor(q[:, 0] / q[:, 2] * fx + cx + 0.5).long()
                v = torch.floor(q[:, 1] / q[:, 2] * fy + cy + 0.5).long()
                keep = (q[:, 2] > 0) & (u >= 0) & (u < W) & (v >= 0) & (v < Hh)
                at = torch.where(keep, v * W + u, torch.zeros_like(u))
                t = self.P[j][at]
                keep &= self.ok[j][at] & ((t - q).norm(dim=1) <= MAX_DIST)
                keep &= (n * torch.nan_to_num(self.normal[j][at])).sum(1) >= math.cos(math.radians(MAX_DEG))
                t, q, n = t[keep], q[keep], n[keep]
                r = (n * (t - q)).sum(1)
                rho, w = _huber(r.abs())
                dense = dense + rho.sum()
                accepted += int(keep.sum())
                if full:
                    J = torch.cat([n, torch.linalg.cross(t, n)], 1) @ _adjoint(T[j])
                    K, b = (J * w[:, None]).T @ J, (J * (w * r)[:, None]).sum(0)
                    H[i, i] += K
                    H[j, j] += K
                    H[i, j] -= K
                    H[j, i] -= K
                    g[i] += b
                    g[j] -= b
        for p, (i, j) in enumerate(s.pairs):
            if s.pts_i is None:
                break
            Ti, Tj = torch.linalg.inv(T[i]), torch.linalg.inv(T[j])
            a = s.pts_i[p].double() @ Ti[:3, :3].T + Ti[:3, 3]
            b = s.pts_j[p].double() @ Tj[:3, :3].T + Tj[:3, 3]
            e = a - b
            rho, w = _huber(e.norm(dim=1))
            sparse = sparse + 2 * rho.sum()
            if full:
                eye = torch.eye(3, dtype=torch.float64, device="cuda").expand(len(a), 3, 3)
                zero = torch.zeros_like(a[:, 0])

                def S(x):
                    X = torch.stack([zero, -x[:, 2], x[:, 1], x[:, 2], zero, -x[:, 0], -x[:, 1], x[:, 0], zero], 1)
                    return torch.cat([eye, -X.reshape(-1, 3, 3)], 2)

                Ja, Jb = -S(a), S(b)
                for r_, J1 in ((i, Ja), (j, Jb)):
                    g[r_] += 2 * torch.einsum("kra,k,kr->a", J1, w, e)
                    for c_, J2 in ((i, Ja), (j, Jb)):
                        H[r_, c_] += 2 * torch.einsum("kra,k,krb->ab", J1, w, J2)
        return dense, sparse, accepted, H, g

    def step(self, T):
        dense, sparse, _, H, g = self.system(T, True)
        n = self.s.n
        A = H.permute(0, 2, 1, 3).reshape(6 * n, 6 * n)[6:, 6:]
        d = torch.linalg.solve(A, -g.reshape(-1)[6:]).reshape(n - 1, 6)
        out = T.clone()
        for k in range(1, n):
            X = torch.zeros(4, 4, dtype=torch.float64, device="cuda")
            X[:3, :3], X[:3, 3] = _skew(d[k - 1, 3:]), d[k - 1, :3]
            out[k] = T[k] @ torch.linalg.matrix_exp(X)
        return out, dense + sparse


def _network(case, seed):
    """The warm-start network on every set of a case: (outputs, labels, weights)."""
    params = torch.tensor(_weights(), device="cuda")
    shapes = [(128, 6), (128,), (256, 128), (256,), (128, 256), (128,), (6, 128), (6,)]
    w, at = [], 0
    for shape in shapes:
        x = params[at:at + math.prod(shape)].reshape(shape)
        at += x.numel()
        w.append((x.bfloat16() if len(shape) == 2 else x).double().requires_grad_())
    outputs, labels = [], []
    for p, q, Ti, Tj, Li, Lj in _point_sets(case, seed):
        M0 = Tj @ np.linalg.inv(Ti)
        p, q = p.double(), q.double()
        c = q.mean(0)
        M = torch.tensor(M0, device="cuda")
        y = p @ M[:3, :3].T + M[:3, 3]
        h = torch.relu(torch.cat([(y - c) * 10.0, (q - y) * 100.0], 1) @ w[0].T + w[1])
        h = h + (h.float().bfloat16().double() - h).detach()
        top = torch.relu(h @ w[2].T + w[3]).max(0).values
        outputs.append(torch.relu(w[4] @ top + w[5]) @ w[6].T + w[7])
        D = Lj @ np.linalg.inv(Li) @ np.linalg.inv(M0)
        angle = math.acos(min(1.0, max(-1.0, (np.trace(D[:3, :3]) - 1) / 2)))
        k = 0.5 + angle * angle / 12 if angle < 1e-4 else 0.5 * angle / math.sin(angle)
        omega = k * np.array([D[2, 1] - D[1, 2], D[0, 2] - D[2, 0], D[1, 0] - D[0, 1]])
        cc = c.cpu().numpy()
        shift = D[:3, :3] @ cc + D[:3, 3] - cc
        labels.append(torch.tensor(np.concatenate([omega / 0.1, shift / 0.01]), device="cuda"))
    return torch.stack(outputs), torch.stack(labels), w


def _ransac(case, scene):
    """Coarse poses: of the drawn 3-point fits of each set (0, j), the one with the most inliers."""
    U, mask = 0x9E3779B97F4A7C15, (1 << 64) - 1

    def mix(c):
        z = (1 + (c + 1) * U) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)

    n, count = case["sets"], case["iters"]
    picks = []
    for h in range(count):
        got = []
        for c in range(16):
            k = mix(16 * h + c) % n
            if len(got) < 3 and k not in got:
                got.append(k)
        picks.append(got if len(got) == 3 else [0, 0, 0])
    picks = np.array(picks)
    out = scene.start.copy()
    limit = np.float32(0.005 * 0.005)
    for j in range(1, scene.n):
        at = scene.pairs.index((0, j))
        p32, q32 = scene.pts_i[at].cpu().numpy(), scene.pts_j[at].cpu().numpy()
        p, q = p32.astype(np.float64)[picks], q32.astype(np.float64)[picks]
        pc, qc = p.mean(1), q.mean(1)
        U_, _, Vt = np.linalg.svd(np.einsum("hka,hkb->hab", p - pc[:, None], q - qc[:, None]))
        flip = np.ones((count, 3))
        flip[:, 2] = np.linalg.det(np.einsum("hba,hcb->hac", Vt, U_))
        R = np.einsum("hba,hb,hcb->hac", Vt, flip, U_)
        t = qc - np.einsum("hab,hb->ha", R, pc)
        R4, t4 = R.astype(np.float32), t.astype(np.float32)
        e2 = np.zeros((count, n), np.float32)
        for r in range(3):
            u = (R4[:, r, 0, None] * p32[:, 0] + R4[:, r, 1, None] * p32[:, 1]) + R4[:, r, 2, None] * p32[:, 2]
            d = (u + t4[:, r, None]) - q32[:, r]
            e2 = d * d if r == 0 else e2 + d * d
        inliers = (e2 < limit).sum(1)
        a, b = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
        area, size = np.linalg.norm(np.cross(a, b), axis=1), (a * a).sum(1) + (b * b).sum(1)
        inliers[~(area > 1e-12 * np.maximum(size, 1e-30))] = -1
        k = int(np.argmax(inliers))
        out[j] = _pose(R[k], t[k]) @ scene.start[0]
    return out


def exact(case, seed):
    """None where one call makes several Gauss-Newton iterations: each decides
    the association anew at poses that carry the rounding of the one before,
    so the end of such a path has no value of its own in 64 bits."""
    kind = case["kind"]
    if kind == "solve" and case["iters"] == 1:
        scene = _scene(case, seed)
        e = Exact(scene)
        T, before = e.step(torch.tensor(scene.start, device="cuda"))
        dense, sparse, _, _, _ = e.system(T, False)
        return dict(poses=T, cost_init=float(before), cost_final=float(dense + sparse))
    if kind in ("build", "pair"):
        scene = _scene(case, seed)
        e = Exact(scene)
        dense, sparse, accepted, _, _ = e.system(torch.tensor(scene.start, device="cuda"), False)
        if kind == "pair":
            return torch.tensor([float(dense), float(accepted)], dtype=torch.float64)
        return dict(total=float(dense + sparse), dense=float(dense), sparse=float(sparse), dense_inliers=None)
    if kind == "predict":
        return _network(case, seed)[0].detach()
    if kind == "train":
        y, label, w = _network(case, seed)
        loss = 0.5 * ((y - label) ** 2).sum(1).mean()
        loss.backward()
        return dict(loss=float(loss), gradient=torch.cat([x.grad.reshape(-1) for x in w]))
    if kind == "ransac":
        return _ransac(case, _scene(case, seed))
    return None
