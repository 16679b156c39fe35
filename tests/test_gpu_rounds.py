"""The forms that the rounds' kernels take for few and for many jobs (pixels split over CTAs or not,
solves by 16 lanes or by one thread, one to 32 lanes per survivor) give the same results bit for bit:
an attempt alone equals the same attempt among so many copies that no form for few jobs applies, at
hypothesis counts around each form's edges and pixel counts that are no multiple of the warps."""
import pytest
import torch

from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("hyps,pixels", [(2, 9), (3, 1), (5, 500), (17, 7), (33, 64), (65, 100), (257, 13), (1030, 8)])
def test_one_attempt_equals_many(room, room_training, room_forest, hyps, pixels):
    world, blocks = room
    scene = B.Scene(blocks, 16)
    forest = B.Forest(room_forest.nodes, room_forest.modes, room_forest.n_modes, max_modes=10)
    intr = synth.Intrinsics.for_size(96, 72)
    pose = synth.query_poses(world, [f[1] for f in room_training], 1, seed=12 + hyps)[0]
    item = dict(scene_b=scene, forest_a=forest, scene_a=scene, intr=intr, pose_b=pose, seed=hyps)
    prm = B.ransac_params(n_hyps=hyps, batch=pixels, max_tries=2000)
    got = []
    for n in (1, max(310, 4300 // hyps + 1)):  # above 304 chunks and 2048 solves in every round's first launches
        att = B.make_attempts([item] * n)
        ws = torch.full((B.batch_workspace_size(att, prm),), 0x7f, dtype=torch.uint8, device=DEV)
        out = torch.zeros(n * B.RESULT_BYTES, dtype=torch.uint8, device=DEV)
        bt = B.Batch(att, prm, ws)
        bt.run(out)
        torch.cuda.synchronize()
        got.append(out.view(n, -1))
    assert (got[1] == got[0][0]).all()
