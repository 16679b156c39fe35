"""Performance cases: the work a program has this framework do, through its public entry points.

Each agent of a collaborative reconstruction keeps a voxel map and a relocalisation forest.  Live
frames are fused into the map and train the forest; synthetic views of one agent's map are
relocalised against another's, one at a time or in batches; the joined maps are rendered
together; the learned regressor is the forest's alternative.  The cases below are those calls.

Maps (the voxel scene, the forest trained on its trajectory's frames) are what a program keeps for
as long as it runs: each is built once per process.  Frames, query poses, sensor noise, RANSAC
seeds, network weights and optimiser moments are drawn from the seed of each preparation.

Camera frames come from the analytic box worlds of the framework's own input generator, rendered
here in closed form, so that no kernel under measurement makes its own input.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import presets, synth

DEPTH_MAX = 12.0
ORIGIN = presets.LEARNED.extra["origin"]


def listed():
    return [
        # One synthetic RGB-D view of a small room, the size a phone client streams: a call of a few
        # tens of microseconds, where launches and latency count.
        dict(name="view_room", kind="view", map="room", width=320, height=240),
        # The renders of one online training step of the regressor: sixteen noisy house views.
        dict(name="views_house", kind="views", map="house", n=16, width=640, height=480, noise=True),
        # A live camera frame relocalised against the house by its three stages: forest, preemptive
        # RANSAC with the paper-sized parameters, verification.
        dict(name="frame_house", kind="frame", map="house", width=640, height=480, hyps=1024, pixels=64),
        # One attempt in the room: what a server does for a lone request.
        dict(name="attempt_room", kind="attempt", map="room", n=1, width=320, height=240, hyps=64, pixels=500,
             noise=False),
        # The headline batch: 256 noisy house attempts in one prepared run.
        dict(name="batch_house", kind="batch", map="house", n=256, width=640, height=480, hyps=1024, pixels=64,
             noise=True),
        # Ordered pairs of fragments, mixed view sizes and hypothesis counts, one-shot call.
        dict(name="batch_fragments", kind="pairs", n=24, max_width=640, pixels=64),
        # A room's forest trained from its first ten frames, leaves clustered and read back.
        dict(name="forest_training", kind="training", map="room", n=10, width=320, height=240, stride=1, capacity=64),
        # One online training step of the regressor: sixteen views, forward, backward and Adam.
        dict(name="regressor_step", kind="reg_step", n=16, width=640, height=480),
        # The regressor's forward pass over a batch of views.
        dict(name="regressor_forward", kind="reg_forward", n=64, width=640, height=480),
        # The joined map: four fragments in one view, with colour and owners.
        dict(name="render_global", kind="global", n=4, width=640, height=480),
        # Mapping: each live frame is fused into the growing room, which is rendered for the client.
        dict(name="mapping_room", kind="mapping", n=8, width=640, height=480, colour=True),
        # An odd-sized view of the house, not a multiple of any tile, without noise.
        dict(name="view_odd", kind="view", map="house", width=517, height=389),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "views", "frame", "attempt", "batch", "pairs", "training", "reg_step", "reg_forward",
                       "global", "mapping"])
    width = _log_int(rng, 160, 640)
    height = max(96, min(480, width * 3 // 4 + rng.randint(-9, 9)))
    size8 = dict(width=max(64, width // 8 * 8), height=max(64, height // 8 * 8))
    if kind == "view":
        return dict(kind=kind, map=rng.choice(["room", "house"]), width=width, height=height)
    if kind == "views":
        return dict(kind=kind, map=rng.choice(["room", "house"]), n=_log_int(rng, 2, 16), width=width, height=height,
                    noise=rng.random() < 0.5)
    if kind == "frame":
        return dict(kind=kind, map=rng.choice(["room", "house"]), width=width, height=height,
                    hyps=_log_int(rng, 32, 1024), pixels=_log_int(rng, 48, 500))
    if kind == "attempt":
        return dict(kind=kind, map="room", n=_log_int(rng, 1, 12), width=width, height=height,
                    hyps=_log_int(rng, 32, 512), pixels=_log_int(rng, 48, 500), noise=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, map="house", n=_log_int(rng, 12, 200), width=width, height=height,
                    hyps=_log_int(rng, 200, 1024), pixels=_log_int(rng, 48, 128), noise=rng.random() < 0.8)
    if kind == "pairs":
        return dict(kind=kind, n=rng.randint(6, 48), max_width=rng.choice([480, 640]), pixels=_log_int(rng, 48, 128))
    if kind == "training":
        return dict(kind=kind, map="room", n=rng.randint(2, 10), width=width, height=height, stride=rng.randint(1, 4),
                    capacity=_log_int(rng, 16, 96))
    if kind == "reg_step":
        return dict(kind=kind, n=_log_int(rng, 1, 16), **size8)
    if kind == "reg_forward":
        return dict(kind=kind, n=_log_int(rng, 1, 64), **size8)
    if kind == "global":
        return dict(kind=kind, n=rng.randint(2, 4), width=width, height=height)
    return dict(kind=kind, n=rng.randint(2, 8), width=width, height=height, colour=rng.random() < 0.7)


# ------------------------------------------------------------------------------------------------
# Camera frames of the analytic worlds
# ------------------------------------------------------------------------------------------------
def _frames(world, intr, poses, seed, noise=True):
    """RGB-D frames of a box world, camera-to-world poses [n, 4, 4]: depth in mm (int16 bits) [n, H, W]
    with noise 1.5 mm z^2, and colour (uint8) [n, H, W, 4] of the nearest surface's texture."""
    dev = "cuda"
    n, H, W = len(poses), intr.height, intr.width
    T = torch.as_tensor(np.stack(poses), dtype=torch.float64, device=dev)
    v, u = torch.meshgrid(torch.arange(H, device=dev, dtype=torch.float64),
                          torch.arange(W, device=dev, dtype=torch.float64), indexing="ij")
    ray = torch.stack([(u - intr.cx) / intr.fx, (v - intr.cy) / intr.fy, torch.ones_like(u)], -1)
    d = torch.einsum("nij,hwj->nihw", T[:, :3, :3], ray).float()
    C = T[:, :3, 3].float()[:, :, None, None]
    inv = 1.0 / torch.where(d.abs() < 1e-9, torch.full_like(d, 1e-9), d)
    best = torch.full((n, H, W), 1e9, device=dev)
    who = torch.zeros((n, H, W), dtype=torch.int64, device=dev)
    comps = np.asarray(world.comps)
    for i, c in enumerate(comps):
        lo = torch.as_tensor(c[1:4], device=dev).float().view(1, 3, 1, 1)
        hi = torch.as_tensor(c[4:7], device=dev).float().view(1, 3, 1, 1)
        t1, t2 = (lo - C) * inv, (hi - C) * inv
        near, far = torch.minimum(t1, t2).amax(1), torch.maximum(t1, t2).amin(1)
        t = far if c[0] == 0 else torch.where((far >= near) & (near > 0), near, torch.full_like(near, 1e9))
        closer = t < best
        best = torch.where(closer, t, best)
        who[closer] = i
    tex = torch.as_tensor(comps[:, 7:13], device=dev).float()[who]
    p = C.movedim(1, -1) + best[..., None] * d.movedim(1, -1)
    x, y, z = p.unbind(-1)
    w = 2 * math.pi
    shade = 0.55 + 0.25 * torch.sin(w * tex[..., 3] * (x + 0.37 * z)) * torch.sin(w * tex[..., 4] * (y - 0.21 * z)) \
        + 0.2 * torch.sin(w * tex[..., 5] * (x + y + z))
    rgba = torch.full((n, H, W, 4), 255, dtype=torch.uint8, device=dev)
    rgba[..., :3] = ((tex[..., :3] * shade[..., None]).clamp(0, 1) * 255 + 0.5).to(torch.uint8)
    mm = best * 1000
    if noise:
        g = torch.Generator(device=dev).manual_seed(int(seed))
        mm = mm + 1.5 * best * best * torch.randn(best.shape, generator=g, device=dev)
    hit = (best > intr.depth_min) & (best < intr.depth_max)
    depth = torch.where(hit, (mm + 0.5).floor().clamp(1, 32767), torch.zeros_like(mm)).to(torch.int16)
    rgba[~hit] = 0
    return depth.contiguous(), rgba.contiguous()


def _noise(n, H, W, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7)
    return torch.randn((n, H, W), generator=g, device="cuda")


# ------------------------------------------------------------------------------------------------
# Maps: voxel scene and trained forest
# ------------------------------------------------------------------------------------------------
def _train(forest, world, to_scene, poses, sizes, stride, capacity):
    B.forest_train_begin(forest, B.train_params(capacity=capacity, stride=stride, seed=7))
    for k in range(0, len(poses), 16):
        some = poses[k:k + 16]
        for W, H in sizes:
            intr = synth.Intrinsics.for_size(W, H, DEPTH_MAX)
            depth, rgba = _frames(world, intr, some, 100 + k)
            for i, P in enumerate(some):
                B.forest_train_frame(forest, intr, to_scene @ P, depth[i], rgba[i])
    B.forest_train_finish(forest)


@functools.lru_cache(maxsize=None)
def _world(name):
    return synth.room_world(1) if name == "room" else synth.house_world(2)


@functools.lru_cache(maxsize=None)
def _scene(name):
    p = presets.TINY if name == "room" else presets.HOUSE
    return B.Scene(synth.sample_scene(_world(name)), p.log2_buckets)


@functools.lru_cache(maxsize=None)
def _poses(name):
    p = presets.TINY if name == "room" else presets.HOUSE
    return synth.training_poses(_world(name), p.train_per_room, seed=11)


@functools.lru_cache(maxsize=None)
def _forest(name):
    p = presets.TINY if name == "room" else presets.HOUSE
    nodes = synth.random_forest_nodes(p.trees, p.depth, seed=5, depth_tau=100, colour_tau=32)
    forest = B.Forest(nodes, max_modes=p.max_modes)
    _train(forest, _world(name), np.eye(4), _poses(name), p.sizes, 2 if name == "room" else 4, min(256, p.reservoir))
    return forest


@functools.lru_cache(maxsize=None)
def _fragments():
    """Four fragments of the house, one or two rooms each, in frames of their own."""
    p, world = presets.FRAGMENTS, _world("house")
    frags = synth.house_fragments(world, 4, seed=3, max_rooms=2)
    synth.fragment_trajectories(world, frags, 8)
    for k, f in enumerate(frags):
        f["scene"] = B.Scene(synth.sample_scene(world, scene_to_world=f["scene_to_world"], crop=f["crop"]),
                             p.log2_buckets)
        f["forest"] = B.Forest(synth.random_forest_nodes(p.trees, p.depth, seed=60 + k, depth_tau=100, colour_tau=32),
                               max_modes=p.max_modes)
        _train(f["forest"], world, np.linalg.inv(f["scene_to_world"]), f["train_w"], p.sizes, 4, 128)
    return frags


def _intr(case):
    return synth.Intrinsics.for_size(case["width"], case["height"], DEPTH_MAX)


def _images(n, H, W):
    return (torch.zeros((n, H, W), dtype=torch.int16, device="cuda"),
            torch.zeros((n, H, W, 4), dtype=torch.uint8, device="cuda"))


# ------------------------------------------------------------------------------------------------
# Regressor inputs
# ------------------------------------------------------------------------------------------------
_LAYERS = [(4, 64, 2), (64, 64, 2), (64, 64, 2)] + [(64, 64, 1)] * 4 + [(64, 4, 1)]


def _network(seed):
    """Weights as after a stretch of training (He-scaled layers, small biases) and Adam's moments."""
    rng = np.random.default_rng([int(seed), 3])
    p = []
    for k, (cin, cout, _) in enumerate(_LAYERS):
        bound = math.sqrt(6.0 / (9 * cin)) * (0.1 if k == len(_LAYERS) - 1 else 1.0)
        p += [rng.uniform(-bound, bound, 9 * cin * cout), rng.uniform(-0.02, 0.02, cout)]
    p = np.concatenate(p).astype(np.float32)
    return dict(params=p, m=(1e-3 * rng.standard_normal(p.size)).astype(np.float32),
                v=(1e-6 * rng.uniform(0.5, 4.0, p.size)).astype(np.float32), step=400)


def _views(case, seed):
    world = _world("house")
    poses = synth.query_poses(world, _poses("house"), case["n"], seed=int(seed))
    parts = [_frames(world, _intr(case), poses[k:k + 16], int(seed) + k) for k in range(0, case["n"], 16)]
    return poses, torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])


# ------------------------------------------------------------------------------------------------
# Preparation
# ------------------------------------------------------------------------------------------------
def _attempts(case, seed):
    """Attempts of a batch against one map: query poses near its trajectory, noise, RANSAC seeds."""
    world, scene, forest, intr = _world(case["map"]), _scene(case["map"]), _forest(case["map"]), _intr(case)
    poses = synth.query_poses(world, _poses(case["map"]), case["n"], seed=int(seed))
    noise = _noise(case["n"], case["height"], case["width"], seed) if case["noise"] else None
    return noise, [dict(scene_b=scene, scene_a=scene, forest_a=forest, intr=intr, pose_b=P,
                        noise=None if noise is None else noise[k], seed=(int(seed) << 20) + k)
                   for k, P in enumerate(poses)]


def _pairs(case, seed):
    """Attempts over ordered pairs of fragments: a view of b's trajectory against a's map."""
    frags, world = _fragments(), _world("house")
    rng = np.random.default_rng([int(seed), 5])
    sizes = [s for s in presets.FRAGMENTS.sizes if s[0] <= case["max_width"]]
    both = [(a, b) for a in range(len(frags)) for b in range(len(frags)) if a != b]
    keep, items = [], []
    for k in range(case["n"]):
        a, b = (frags[i] for i in both[k % len(both)])
        W, H = sizes[rng.integers(len(sizes))]
        P = synth.query_poses(world, b["train_w"], 1, seed=int(rng.integers(1 << 30)))[0]
        keep.append(_noise(1, H, W, int(rng.integers(1 << 30)))[0])
        items.append(dict(scene_b=b["scene"], scene_a=a["scene"], forest_a=a["forest"],
                          intr=synth.Intrinsics.for_size(W, H, DEPTH_MAX),
                          pose_b=synth.world_to_scene_pose(P, b["scene_to_world"]), noise=keep[-1],
                          n_hyps=int(rng.integers(256, 1025)), seed=int(rng.integers(1 << 40))))
    return keep, items


def prepare(case, seed):
    kind, s = case["kind"], SimpleNamespace(case=case)
    if kind == "view":
        s.scene, s.intr = _scene(case["map"]), _intr(case)
        s.pose = synth.query_poses(_world(case["map"]), _poses(case["map"]), 1, seed=int(seed))[0]
        depth, rgba = _images(1, case["height"], case["width"])
        s.depth, s.rgba = depth[0], rgba[0]
    elif kind == "views":
        n, H, W = case["n"], case["height"], case["width"]
        s.scene, s.intr = _scene(case["map"]), _intr(case)
        s.poses = synth.query_poses(_world(case["map"]), _poses(case["map"]), n, seed=int(seed))
        s.depth, s.rgba = _images(n, H, W)
        s.noise = _noise(n, H, W, seed) if case["noise"] else None
        s.ws = torch.empty(B.raycast_views_workspace_size(n), dtype=torch.uint8, device="cuda")
    elif kind == "frame":
        H, W = case["height"], case["width"]
        s.scene, s.forest, s.intr = _scene(case["map"]), _forest(case["map"]), _intr(case)
        world = _world(case["map"])
        pose = synth.query_poses(world, _poses(case["map"]), 1, seed=int(seed))
        depth, rgba = _frames(world, s.intr, pose, seed)
        s.depth, s.rgba = depth[0], rgba[0]
        s.leaves = torch.zeros((s.forest.n_trees, H, W), dtype=torch.int16, device="cuda")
        s.params = B.ransac_params(n_hyps=case["hyps"], batch=case["pixels"], seed=int(seed))
        s.ws = torch.empty(B.ransac_workspace_size(W, H, s.params), dtype=torch.uint8, device="cuda")
        s.result = torch.zeros(B.RESULT_BYTES, dtype=torch.uint8, device="cuda")
        s.seen = torch.zeros((H, W), dtype=torch.int16, device="cuda")
    elif kind in ("attempt", "batch", "pairs"):
        s.keep, items = _pairs(case, seed) if kind == "pairs" else _attempts(case, seed)
        s.params = B.ransac_params(n_hyps=case.get("hyps", 1024), batch=case["pixels"])
        s.attempts = B.make_attempts(items)
        s.items = items
        s.ws = torch.empty(B.batch_workspace_size(s.attempts, s.params), dtype=torch.uint8, device="cuda")
        if kind == "batch":
            s.batch = B.Batch(s.attempts, s.params, s.ws)
            s.result = torch.zeros(case["n"] * B.RESULT_BYTES, dtype=torch.uint8, device="cuda")
        else:
            s.result = (B.PoseResult * case["n"])()
    elif kind == "training":
        p, world, s.intr = presets.TINY, _world(case["map"]), _intr(case)
        s.poses = synth.query_poses(world, _poses(case["map"]), case["n"], seed=int(seed))
        s.depth, s.rgba = _frames(world, s.intr, s.poses, seed)
        s.nodes = synth.random_forest_nodes(p.trees, p.depth, seed=int(seed) % 9973, depth_tau=100, colour_tau=32)
        s.forest = B.Forest(s.nodes, max_modes=p.max_modes)
        s.params = B.train_params(capacity=case["capacity"], stride=case["stride"], seed=int(seed))
    elif kind in ("reg_step", "reg_forward"):
        n, H, W = case["n"], case["height"], case["width"]
        s.intr, net = _intr(case), _network(seed)
        s.poses, s.depth, s.rgba = _views(case, seed)
        s.net = B.Regressor(net["params"], origin=ORIGIN)
        train = kind == "reg_step"
        s.ws = torch.empty(B.regressor_workspace_size(n, W, H, train), dtype=torch.uint8, device="cuda")
        if train:
            B.regressor_set_state(s.net, net)
            s.loss = torch.zeros(1, device="cuda")
        else:
            s.out = torch.zeros((n, H // 8, W // 8, 4), device="cuda")
    elif kind == "global":
        frags, world = _fragments()[:case["n"]], _world("house")
        rng = np.random.default_rng([int(seed), 9])
        every = [P for f in frags for P in f["train_w"]]
        s.scenes = [f["scene"] for f in frags]
        s.globals = [f["scene_to_world"] for f in frags]
        s.intr = _intr(case)
        s.pose = synth.query_poses(world, every, 1, seed=int(rng.integers(1 << 30)))[0]
        depth, rgba = _images(1, case["height"], case["width"])
        s.depth, s.rgba = depth[0], rgba[0]
        s.owner = torch.zeros((case["height"], case["width"]), dtype=torch.int8, device="cuda")
        s.ws = torch.empty(B.render_global_workspace_size(case["n"]), dtype=torch.uint8, device="cuda")
    else:
        n, world, s.intr = case["n"], _world("room"), _intr(case)
        s.poses = synth.query_poses(world, _poses("room"), n, seed=int(seed))
        s.depth, s.rgba = _frames(world, s.intr, s.poses, seed)
        s.scene = B.FusionScene(1 << 18, synth.VOXEL_SIZE, synth.TRUNCATION, 18)
        s.view, s.colour = _images(n, case["height"], case["width"])
    return s


# ------------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------------
_RESULT = np.dtype([("pose", "<f8", (4, 4)), ("rel", "<f8", (4, 4)), ("energy", "<f8"), ("small", "<i4", (6,)),
                    ("counts", "<u8", (6,)), ("path", "<i4", (2,))])


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "view":
        B.raycast_view(s.scene, s.intr, s.pose, s.depth, s.rgba)
        return dict(depth=s.depth, rgba=s.rgba)
    if kind == "views":
        B.raycast_views(s.scene, s.intr, s.poses, s.depth, s.rgba, noise_dev=s.noise, workspace_dev=s.ws)
        return dict(depth=s.depth, rgba=s.rgba)
    if kind == "frame":
        B.forest_eval(s.forest, s.depth, s.rgba, s.leaves)
        B.ransac_relocalise(s.forest, s.depth, s.leaves, s.intr, s.params, s.ws, s.result)
        B.verify(s.scene, s.intr, s.depth, s.result, s.seen)
        return dict(leaves=s.leaves, seen=s.seen, pose=s.result.view(torch.float64)[:33],
                    counts=s.result.view(torch.int32)[66:])
    if kind in ("attempt", "pairs"):
        B.relocalise_batch_into(s.attempts, s.params, s.ws, s.result)
        r = np.frombuffer(s.result, dtype=_RESULT)
        return dict(pose=r["pose"], rel=r["rel"], energy=r["energy"], small=r["small"],
                    counts=r["counts"].astype(np.int64))
    if kind == "batch":
        s.batch.run(s.result)
        return dict(pose=s.result.view(torch.float64).view(case["n"], -1)[:, :33],
                    counts=s.result.view(torch.int32).view(case["n"], -1)[:, 66:])
    if kind == "training":
        B.forest_train_begin(s.forest, s.params)
        for k in range(case["n"]):
            B.forest_train_frame(s.forest, s.intr, s.poses[k], s.depth[k], s.rgba[k])
        B.forest_train_finish(s.forest)
        samples, count = B.forest_train_reservoirs(s.forest, case["capacity"])
        modes, n_modes = s.forest.get_modes()
        return dict(samples=samples, count=count, modes=modes, n_modes=n_modes)
    if kind == "reg_step":
        B.regressor_train_step(s.net, s.depth, s.rgba, s.intr, s.poses, 5e-4, s.ws, loss_dev=s.loss)
        return dict(loss=s.loss, grads=s.net.grads(), params=s.net.params())
    if kind == "reg_forward":
        B.regressor_forward(s.net, s.depth, s.rgba, s.out, s.ws)
        return s.out
    if kind == "global":
        B.render_global(s.scenes, s.globals, s.intr, s.pose, s.depth, s.rgba, s.owner, workspace_dev=s.ws)
        return dict(depth=s.depth, rgba=s.rgba, owner=s.owner)
    for k in range(case["n"]):
        s.scene.fuse(s.intr, s.poses[k], s.depth[k], s.rgba[k] if case["colour"] else None)
        B.raycast_view(s.scene, s.intr, s.poses[k], s.view[k], s.colour[k] if case["colour"] else None)
    return dict(view=s.view, colour=s.colour)


# ------------------------------------------------------------------------------------------------
# Work and 64-bit values
# ------------------------------------------------------------------------------------------------
# Bytes a raycast cannot do without, per pixel, by exact count of the distinct voxels and table
# entries that the house views' rays need: with colour, and depth only.
_VIEW_BYTES, _DEPTH_BYTES = 50.7, 35.9


def work(case):
    kind, n = case["kind"], case.get("n", 1)
    px = case.get("width", 480) * case.get("height", 360)
    hyps, pixels = case.get("hyps", 640), case.get("pixels", 64)
    # rounds: K + K / 2 + ... scored on `pixels` draws each, about four modes in each of five trees
    rounds = 2.0 * hyps * pixels * 20 * 30
    if kind in ("view", "views", "global"):
        return dict(bytes=px * _VIEW_BYTES * (1 if kind == "global" else n), flops=px * n * 600.0)
    if kind == "frame":
        return dict(bytes=px * (16.0 + _DEPTH_BYTES + 2), flops=rounds + px * 5 * 15 * 10.0)
    if kind in ("attempt", "batch", "pairs"):
        return dict(bytes=n * px * (_VIEW_BYTES + 16 + _DEPTH_BYTES + (4 if case.get("noise", True) else 0)),
                    flops=n * (rounds + px * (5 * 15 * 10.0 + 1200)))
    if kind == "training":
        return dict(bytes=n * (px * 6.0 + 5 * 12.0 * px / case["stride"] ** 2) + 5 * 1024 * 10 * 48.0,
                    flops=5 * 1024 * 25 * 12.0 * case["capacity"] ** 2)
    if kind in ("reg_step", "reg_forward"):
        flops, w, h = 0.0, case["width"], case["height"]
        for cin, cout, stride in _LAYERS:
            w, h = (w - 1) // stride + 1, (h - 1) // stride + 1
            flops += 18.0 * w * h * cin * cout
        io = px * 6.0 + w * h * 16
        return dict(bytes=n * io + 5e6 * (kind == "reg_step"), flops=n * flops * (3 if kind == "reg_step" else 1))
    # mapping: each frame read, about 6000 blocks of 8-byte voxels and weights read and written, the view
    return dict(bytes=n * (px * 6.0 + 6000 * 512 * 20.0 + px * _VIEW_BYTES), flops=n * 6000 * 512 * 40.0)


def _net64(net, depth, rgba):
    """(weights, head output [n, 4, Hc, Wc]) of the network in 64 bits."""
    d = depth.to(torch.int32).bitwise_and(0xFFFF).double() * 0.001
    x = torch.cat([((d - 3.0) * 0.5)[:, None], (rgba[..., :3].double() / 255 - 0.5).movedim(-1, 1) * 4], 1)
    weights, at = [], 0
    flat = torch.as_tensor(net["params"], device="cuda").double()
    for cin, cout, stride in _LAYERS:
        w = flat[at:at + 9 * cin * cout].view(3, 3, cin, cout).clone().requires_grad_()
        b = flat[at + 9 * cin * cout:at + 9 * cin * cout + cout].clone().requires_grad_()
        at += 9 * cin * cout + cout
        weights += [w, b]
        x = F.conv2d(x, w.permute(3, 2, 0, 1), b, stride=stride, padding=1)
        x = x if cout == 4 else F.relu(x)
    return weights, x


def _step64(case, seed):
    net, intr = _network(seed), _intr(case)
    poses, depth, rgba = _views(case, seed)
    # view by view: the loss is a mean over the scored cells of all views
    centre = depth[:, 4::8, 4::8].to(torch.int32).bitwise_and(0xFFFF)
    scored = max(1, int((centre > 0).sum()))
    loss, grads = 0.0, None
    T = torch.as_tensor(np.stack(poses), device="cuda").double()
    Hc, Wc = centre.shape[1:]
    v, u = torch.meshgrid(torch.arange(Hc, device="cuda").double() * 8 + 4,
                          torch.arange(Wc, device="cuda").double() * 8 + 4, indexing="ij")
    for k in range(case["n"]):
        weights, out = _net64(net, depth[k:k + 1], rgba[k:k + 1])
        z = centre[k].double() / 1000
        cam = torch.stack([z * (u - intr.cx) / intr.fx, z * (v - intr.cy) / intr.fy, z])
        y = torch.einsum("ij,jhw->ihw", T[k, :3, :3], cam) + (T[k, :3, 3] - torch.tensor(ORIGIN, device="cuda").double())[:, None, None]
        e = out[0, :3] - y
        sq, s, on = (e * e).sum(0), out[0, 3], centre[k] > 0
        each = torch.sqrt(sq + 1e-6) + 0.5 * sq.detach() * torch.exp(-s) + 1.5 * s
        total = each[on].sum() / scored
        got = torch.autograd.grad(total, weights)
        loss += float(total.detach())
        got = torch.cat([g.reshape(-1) for g in got])
        grads = got if grads is None else grads + got
    m = 0.9 * torch.as_tensor(net["m"], device="cuda").double() + 0.1 * grads
    w = 0.999 * torch.as_tensor(net["v"], device="cuda").double() + 0.001 * grads * grads
    t = net["step"] + 1
    p = torch.as_tensor(net["params"], device="cuda").double()
    p = p - 5e-4 * (m / (1 - 0.9 ** t)) / (torch.sqrt(w / (1 - 0.999 ** t)) + 1e-8)
    return dict(loss=torch.tensor([loss], dtype=torch.float64), grads=grads.cpu().numpy(), params=p.cpu().numpy())


def _philox(c, key):
    """Philox4x32-10 on counters c (int64 tensors, 4 of them); the first output word."""
    low = 0xFFFFFFFF
    k0, k1 = key & low, key >> 32 & low

    def mul(a, x):  # (high, low) words of a 32 x 32-bit product, in 16-bit halves
        xl, xh = x & 0xFFFF, x >> 16
        l = a * xl
        h = a * xh + (l >> 16)
        return h >> 16, (h & 0xFFFF) << 16 | (l & 0xFFFF)

    c = list(c)
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c[0]


def _reservoirs64(case, seed):
    """The leaves' reservoirs after all frames: samples (scene coordinates in 64 bits)."""
    s = prepare(case, seed)
    H, W, st, cap, D = case["height"], case["width"], case["stride"], case["capacity"], presets.TINY.depth
    nodes = {k: torch.as_tensor(s.nodes[k].astype(np.int64)) for k in s.nodes.dtype.names}
    T, L = s.nodes.shape[0], 1 << D
    ids, points = [], []
    for k in range(case["n"]):
        depth = s.depth[k].cpu().to(torch.int64) & 0xFFFF
        rgba = s.rgba[k].cpu().to(torch.int64)
        v, u = (g.reshape(-1) for g in torch.meshgrid(torch.arange(0, H, st), torch.arange(0, W, st), indexing="ij"))
        d = depth[v, u]
        v, u, d = v[d > 0], u[d > 0], d[d > 0]
        leaf = []
        for t in range(T):
            at = torch.zeros_like(d)
            for _ in range(D):
                f = {q: nodes[q][t][at] for q in nodes}
                probe = lambda x, o, top: (x + torch.div(o * 1000, d, rounding_mode="trunc")).clamp(0, top)  # noqa: E731
                y1, x1 = probe(v, f["dy1"], H - 1), probe(u, f["dx1"], W - 1)
                y2, x2 = probe(v, f["dy2"], H - 1), probe(u, f["dx2"], W - 1)
                far = depth[y1, x1] - depth[y2, x2]
                hue = rgba[y1, x1].gather(1, f["c1"][:, None])[:, 0] - rgba[y2, x2].gather(1, f["c2"][:, None])[:, 0]
                at = 2 * at + torch.where(torch.where(f["kind"] == 0, far, hue) < f["tau"], 1, 2)
            leaf.append(t * L + at - (L - 1))
        z = d.double() / 1000
        cam = torch.stack([z * (u - s.intr.cx) / s.intr.fx, z * (v - s.intr.cy) / s.intr.fy, z], 1)
        P = torch.as_tensor(np.asarray(s.poses[k]))
        ids.append(torch.stack(leaf, 1).reshape(-1))
        points.append((cam @ P[:3, :3].T + P[:3, 3]).repeat_interleave(T, 0))
    ids, points = torch.cat(ids), torch.cat(points)
    order = torch.argsort(ids, stable=True)
    ids, points = ids[order], points[order]
    seen = torch.bincount(ids, minlength=T * L)
    nth = torch.arange(len(ids)) - (torch.cumsum(seen, 0) - seen)[ids]
    word = _philox([torch.full_like(ids, 3), ids, nth, torch.zeros_like(ids)], int(seed))
    high = (word >> 16) * (nth + 1) + ((word & 0xFFFF) * (nth + 1) >> 16)
    slot = torch.where(nth < cap, nth, high >> 16)
    kept = slot < cap
    at = (ids * cap + slot)[kept].numpy()
    samples = np.zeros((T * L * cap, 3))
    samples[at] = points[kept].numpy()  # the last offer of a slot stays, as in the order of offers
    return samples.reshape(T, L, cap, 3), seen.clamp(max=cap).view(T, L).numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "reg_forward":
        net = _network(seed)
        _, depth, rgba = _views(case, seed)
        with torch.no_grad():
            return torch.cat([_net64(net, depth[k:k + 1], rgba[k:k + 1])[1] for k in range(case["n"])]).movedim(1, -1)
    if kind == "reg_step":
        return _step64(case, seed)
    if kind == "training":
        samples, count = _reservoirs64(case, seed)
        # the modes come of comparisons (which ascents meet within a distance) that one bit can turn
        return dict(samples=samples, count=count, modes=None, n_modes=None)
    # views and maps are whole numbers; a whole attempt's 64-bit evaluation takes far too long
    return None
