"""Forest nodes as the device holds them (numbered from 1, a node's trees together, thresholds within
17 bits) and the tiled image that a batch's forest reads, against the oracle, bit for bit: every
unrolled width and its remainders, trees of one level, thresholds beyond any difference, every channel,
and images whose sides are no multiples of the 8-pixel tiles."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _nodes(trees, depth, seed, channels=3):
    """Random nodes, an eighth of them with thresholds past every possible difference of two probes."""
    nodes = synth.random_forest_nodes(trees, depth, seed=seed)
    rng = np.random.default_rng(seed + 1)
    for c in ("c1", "c2"):
        nodes[c] = rng.integers(0, channels, nodes.shape)
    extreme = np.array([2**31 - 1, -2**31, 65536, -65536, 65535, -65535, 70000, -70000], np.int32)
    at = rng.random(nodes.shape) < 0.125
    nodes["tau"][at] = rng.choice(extreme, int(at.sum()))
    return nodes


def _u16(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.uint16).view(np.int16)).to(DEV)


@pytest.mark.parametrize("trees,depth,W,H", [(1, 1, 33, 9), (2, 6, 8, 8), (4, 15, 65, 17), (5, 3, 1, 1), (7, 8, 31, 40),
                                             (16, 11, 70, 23)])
def test_images_in_rows(trees, depth, W, H):
    rng = np.random.default_rng(17 * trees + depth)
    d = rng.choice(np.array([0, 1, 9, 15, 16, 64, 65, 700, 2500, 30000, 65535], np.uint16), (H, W))
    c = rng.integers(0, 256, (H, W, 4)).astype(np.uint8)
    nodes = _nodes(trees, depth, 3 * trees + depth, channels=4)
    leaves = torch.zeros((trees, H, W), dtype=torch.int16, device=DEV)
    B.forest_eval(B.Forest(nodes, max_modes=1), _u16(d), torch.from_numpy(c).to(DEV), leaves)
    torch.cuda.synchronize()
    assert np.array_equal(leaves.cpu().numpy().view(np.uint16), oracle.forest_eval(nodes, d, c))


def test_tiled_images(room, room_training):
    """A batch's views of ragged sizes through forests of 1 to 16 trees."""
    world, blocks = room
    scene = B.Scene(blocks, 16)
    shapes = [(1, 7, 33, 25), (4, 9, 96, 72), (5, 10, 150, 101), (6, 1, 64, 48), (8, 12, 47, 83), (16, 5, 129, 65)]
    qs = synth.query_poses(world, [f[1] for f in room_training], len(shapes), seed=12)
    items, nodes = [], []
    for i, (T, D, W, H) in enumerate(shapes):
        nodes.append(_nodes(T, D, 40 + i))
        f = B.Forest(nodes[i], np.zeros((T, 1 << D, 1, 12)), np.zeros((T, 1 << D)), max_modes=1)
        items.append(dict(scene_b=scene, forest_a=f, scene_a=scene, intr=synth.Intrinsics.for_size(W, H), pose_b=qs[i],
                          noise=torch.from_numpy(synth.depth_noise(H, W, i)).to(DEV), n_hyps=4, seed=i))
    prm = B.ransac_params(n_hyps=4, batch=20, max_tries=5)
    for picks in ([0, 1, 2, 3, 4], list(range(6)), [5], [2]):  # the widest forest sets the unrolled width
        att = B.make_attempts([items[k] for k in picks])
        bt = B.Batch(att, prm, torch.empty(B.batch_workspace_size(att, prm), dtype=torch.uint8, device=DEV))
        out = torch.zeros(len(picks) * B.RESULT_BYTES, dtype=torch.uint8, device=DEV)
        for rows in (0, 1):
            bt.set_schedule(forest_tiles=rows)
            bt.run(out)
            torch.cuda.synchronize()
            for k, i in enumerate(picks):
                T, _, W, H = shapes[i]
                d, c, lv = (x.cpu().numpy() for x in bt.attempt_images(k, W, H, trees=T))
                assert np.array_equal(lv.view(np.uint16), oracle.forest_eval(nodes[i], d.view(np.uint16), c)), (i, rows)


def test_batches_read_alpha(room, room_training):
    """Forests whose nodes compare channel 3 (0 where a view's ray misses, 255 elsewhere), beside one that
    has no such node."""
    world, blocks = room
    scene = B.Scene(blocks, 16)
    shapes = [(5, 10, 150, 101, 4), (4, 9, 96, 72, 3), (8, 12, 47, 83, 4)]
    qs = synth.query_poses(world, [f[1] for f in room_training], len(shapes), seed=12)
    items, nodes = [], []
    for i, (T, D, W, H, channels) in enumerate(shapes):
        nodes.append(_nodes(T, D, 70 + i, channels))
        f = B.Forest(nodes[i], np.zeros((T, 1 << D, 1, 12)), np.zeros((T, 1 << D)), max_modes=1)
        items.append(dict(scene_b=scene, forest_a=f, scene_a=scene, intr=synth.Intrinsics.for_size(W, H), pose_b=qs[i],
                          n_hyps=4, seed=i))
    prm = B.ransac_params(n_hyps=4, batch=20, max_tries=5)
    att = B.make_attempts(items)
    bt = B.Batch(att, prm, torch.empty(B.batch_workspace_size(att, prm), dtype=torch.uint8, device=DEV))
    bt.run(torch.zeros(len(items) * B.RESULT_BYTES, dtype=torch.uint8, device=DEV))
    torch.cuda.synchronize()
    for i, (T, _, W, H, _) in enumerate(shapes):
        d, c, lv = (x.cpu().numpy() for x in bt.attempt_images(i, W, H, trees=T))
        assert np.array_equal(lv.view(np.uint16), oracle.forest_eval(nodes[i], d.view(np.uint16), c)), i
