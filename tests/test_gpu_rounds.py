"""The forms that the rounds' kernels take for few and for many jobs (pixels split over CTAs or not,
solves by 16 lanes or by one thread, one to 32 lanes per survivor) give the same results bit for bit:
an attempt alone equals the same attempt among so many copies that no form for few jobs applies, at
hypothesis counts around each form's edges and pixel counts that are no multiple of the warps."""
import numpy as np
import pytest
import torch

import oracle

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


@pytest.mark.parametrize("counts", [(15, 15, 15, 15), (16, 15, 15, 15), (16, 16, 16, 16), (8,) * 8, (4,) * 16])
@pytest.mark.parametrize("hyps,pixels", [(3, 17), (256, 40)])
def test_pixels_of_up_to_64_modes(room_training, room_forest, counts, hyps, pixels):
    """Scores from staged modes equal those read one by one: the same forest with further modes that never
    win (a score below any other's) has more than 64 a pixel, which are not staged."""
    intr, _, d, c = room_training[2]
    T, D, M = len(counts), 10, 32
    L = 1 << D
    rng = np.random.default_rng(hyps + T)
    trees = np.arange(T) % len(room_forest.modes)
    modes = np.repeat(room_forest.modes[trees, :, :1], M, 2).astype(np.float32)  # each leaf's first mode, moved about
    modes[:, :, 1:, :3] += rng.normal(0, 0.05, (T, L, M - 1, 3))
    real = oracle.forest_eval(room_forest.nodes, d, c)
    prm = B.ransac_params(n_hyps=hyps, batch=pixels, max_tries=2000, seed=5)
    ws = torch.empty(B.ransac_workspace_size(intr.width, intr.height, prm), dtype=torch.uint8, device=DEV)
    du, lu = (torch.from_numpy(np.ascontiguousarray(a, np.uint16).view(np.int16)).to(DEV) for a in (d, real[trees]))
    nodes = synth.random_forest_nodes(T, D, seed=3)
    got = []
    for extra in (0, 65 - sum(counts)):
        m, n = modes.copy(), np.zeros((T, L), np.uint8)
        for t, k in enumerate(counts):
            n[t] = np.where(room_forest.n_modes[trees[t]] > 0, k + (extra if t == 0 else 0), 0)
            m[t, :, k:, 9] = -1e30
        res = torch.zeros(B.RESULT_BYTES, dtype=torch.uint8, device=DEV)
        B.ransac_relocalise(B.Forest(nodes, m, n, max_modes=M), du, lu, intr, prm, ws, res)
        torch.cuda.synchronize()
        got.append(res)
    assert hyps == 3 or B.result_from_bytes(got[0])["status"] == 0  # (three draws may all fail)
    assert torch.equal(got[0], got[1])
