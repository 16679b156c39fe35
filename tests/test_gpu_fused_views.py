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


@pytest.mark.parametrize("shift", [0.0, -7.36])
def test_rays_along_block_edges(room, shift):
    """Rays in block faces, along block edges and through block and word corners: cameras on corners of the
    4 cm blocks and 16 cm words (and off them by less and by more than a walk's 1e-5 step past a face), axis
    aligned, with a pixel pitch of 1/32, so that rays run along the axes and the faces' diagonals."""
    world, blocks = room
    source = B.Scene(blocks, 16)
    W, H = 160, 120
    intr = synth.Intrinsics.for_size(W, H)
    fused = B.FusionScene(1 << 17, synth.VOXEL_SIZE, synth.TRUNCATION, 12)
    depth = torch.zeros((H, W), dtype=torch.int16, device=DEV)
    rgba = torch.zeros((H, W, 4), dtype=torch.uint8, device=DEV)
    for P in synth.training_poses(world, 6, seed=21):
        B.raycast_view(source, intr, P, depth, rgba)
        Q = P.copy()
        Q[:3, 3] += shift
        fused.fuse(intr, Q, depth, rgba)
    coords, tsdf, colour, _ = fused.export()
    static = B.Scene(synth.SceneBlocks(coords, tsdf, colour, synth.VOXEL_SIZE, synth.TRUNCATION, np.eye(4)), 12)
    static.use_grid(False)
    static.use_apron(False)
    grid = synth.Intrinsics(65, 49, 32.0, 32.0, 32.0, 24.0)
    axes = np.eye(3)
    hits = 0
    for centre in ((2.0, 2.0, 1.2), (1.92, 2.08, 1.28), (2.005, 2.0, 1.2)):
        for off in (0.0, 1e-6, -1e-6, 9e-6, -2e-5, 1e-4):
            for k in range(6):
                f = axes[k // 2] * (1 if k % 2 == 0 else -1)
                r = axes[(k // 2 + 1) % 3]
                P = np.eye(4)
                P[:3, 0], P[:3, 1], P[:3, 2] = r, np.cross(f, r), f
                P[:3, 3] = np.array(centre) + off + shift
                a, b = _render(fused, grid, P), _render(static, grid, P)
                assert all(torch.equal(x, y) for x, y in zip(a, b)), (centre, off, k)
                hits += int((a[0] != 0).sum())
    assert hits > 108 * 65 * 49 // 8
