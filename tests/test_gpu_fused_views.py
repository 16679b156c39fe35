"""Views of growing scenes through their cell words against the same blocks looked up in the hash alone:
a static scene made of the fused scene's exported blocks, without its grid and apron copy, walks block
by block through its hash.  Depth, colour and global renders equal bit for bit: with blocks at negative
coordinates, words shared by blocks 64 words apart, odd image sizes, and an empty scene."""
import numpy as np
import pytest
import torch

from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _render(scene, intr, pose):
    depth = torch.zeros((intr.height, intr.width), dtype=torch.int16, device=DEV)
    rgba = torch.zeros((intr.height, intr.width, 4), dtype=torch.uint8, device=DEV)
    owner = torch.zeros((intr.height, intr.width), dtype=torch.int8, device=DEV)
    B.raycast_view(scene, intr, pose, depth, rgba)
    alone = torch.zeros_like(depth)
    B.raycast_view(scene, intr, pose, alone)
    seen, colour = torch.zeros_like(depth), torch.zeros_like(rgba)
    B.render_global([scene, scene], [np.eye(4)] * 2, intr, pose, seen, colour, owner)
    torch.cuda.synchronize()
    assert torch.equal(depth, alone)
    return depth, rgba, seen, colour, owner


@pytest.mark.parametrize("size,shift", [((160, 120), 0.0), ((131, 97), -7.3), ((64, 48), 10.24)])
def test_cell_words_equal_the_hash_walk(room, size, shift):
    """shift: the agent's origin; 10.24 m is 64 words of 4 blocks of 8 voxels of 5 mm, so that frames of
    both origins, fused into one scene, share words."""
    world, blocks = room
    source = B.Scene(blocks, 16)
    W, H = size
    intr = synth.Intrinsics.for_size(W, H)
    fused = B.FusionScene(1 << 17, synth.VOXEL_SIZE, synth.TRUNCATION, 12)
    train = synth.training_poses(world, 4, seed=21)
    depth = torch.zeros((H, W), dtype=torch.int16, device=DEV)
    rgba = torch.zeros((H, W, 4), dtype=torch.uint8, device=DEV)
    empty = _render(fused, intr, train[0])
    assert int(empty[0].abs().max()) == 0 and int(empty[2].abs().max()) == 0
    moved = []
    for P in train:
        B.raycast_view(source, intr, P, depth, rgba)
        for s in {0.0, shift}:
            Q = P.copy()
            Q[:3, 3] += s
            fused.fuse(intr, Q, depth, rgba)
            moved.append(Q)
    coords, tsdf, colour, _ = fused.export()
    static = B.Scene(synth.SceneBlocks(coords, tsdf, colour, synth.VOXEL_SIZE, synth.TRUNCATION, np.eye(4)), 12)
    static.use_grid(False)
    static.use_apron(False)
    for P in moved + synth.query_poses(world, train, 2, seed=5):
        for a, b in zip(_render(fused, intr, P), _render(static, intr, P)):
            assert torch.equal(a, b)
    assert int((_render(fused, intr, moved[0])[0] != 0).sum()) > W * H // 3
