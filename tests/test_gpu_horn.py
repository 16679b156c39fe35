"""Hypothesis poses against the oracle's FP64 Jacobi rotations: the eigenvectors refined from FP32, and
the rotations that take over where the largest eigenvalue does not stand clear (a relative gap below
5e-4), with solves shared by lanes and one a thread.  Bars: a solve rounds to ten units of 2^-52 or so
over the gap.  A triple has camera-point cross products of 1e-3 m^2 or more and edges of a few metres, so
its gap is at least about (1e-3 / 16)^2 = 4e-9 (largest error 1e-6), and one triple in a hundred is
thinner than 1 : 100, a gap of 1e-4 (99 % within 1e-10)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_08361_gb300 import binding as B

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("hyps,frame", [(7, 0), (256, 1), (2049, 2)])
def test_poses_match_the_oracle(room_forest, room_training, hyps, frame):
    intr, _, d, c = room_training[frame]
    leaves = oracle.forest_eval(room_forest.nodes, d, c)
    want, ok, tries = oracle.generate_hypotheses(d, intr, leaves, room_forest, oracle.RansacParams(n_hyps=hyps, batch=8, seed=3))
    prm = B.ransac_params(n_hyps=hyps, batch=8, seed=3)
    forest = B.Forest(room_forest.nodes, room_forest.modes, room_forest.n_modes, max_modes=10)
    poses = torch.zeros((hyps, 12), dtype=torch.float64, device=DEV)
    valid = torch.zeros(hyps, dtype=torch.int32, device=DEV)
    n_tries = torch.zeros(hyps, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.ransac_workspace_size(intr.width, intr.height, prm), dtype=torch.uint8, device=DEV)
    du, lu = (torch.from_numpy(np.ascontiguousarray(a, np.uint16).view(np.int16)).to(DEV) for a in (d, leaves))
    B.ransac_hypotheses(forest, du, lu, intr, prm, ws, poses, valid, n_tries)
    torch.cuda.synchronize()
    assert np.array_equal(valid.cpu().numpy().astype(bool), ok) and np.array_equal(n_tries.cpu().numpy(), tries)
    assert ok.any()
    R = poses.cpu().numpy().reshape(hyps, 3, 4)[ok][:, :, :3]
    err = np.abs(R - want[ok][:, :3, :3]).max(axis=(1, 2))
    assert err.max() <= 1e-6 and np.quantile(err, 0.99) <= 1e-10, (err.max(), np.quantile(err, 0.99))
    assert np.abs(R @ R.transpose(0, 2, 1) - np.eye(3)).max() <= 1e-12
