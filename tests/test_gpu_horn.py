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
from paper_1801_08361_gb300 import synth

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


def _gaps(d, intr, leaves, forest, tries, seed):
    """Relative gap below the largest eigenvalue of each kept triple's 4 x 4 matrix, and its camera centroid."""
    key, valid, n = oracle.seed_key(seed), oracle.valid_pixels(d), len(tries)
    ctr = np.zeros((n, 4), np.uint32)
    ctr[:, 0], ctr[:, 1], ctr[:, 2] = oracle.TAG_HYP, np.arange(n), tries
    x = oracle.philox(ctr, key)
    pix = valid[oracle.uniform_below(x[:, :3], len(valid))]
    leaf = leaves.reshape(1, -1)[0, pix].astype(int)
    cam = oracle.camera_points(d, intr, pix.reshape(-1)).reshape(n, 3, 3)
    w = forest.modes[0, leaf, 0, :3].astype(float)
    c = cam.mean(1)
    S = np.einsum("nka,nkb->nab", cam - c[:, None], w - w.mean(1, keepdims=True))
    (xx, xy, xz), (yx, yy, yz), (zx, zy, zz) = np.moveaxis(S, 0, 2)
    N = np.array([[xx + yy + zz, yz - zy, zx - xz, xy - yx], [yz - zy, xx - yy - zz, xy + yx, zx + xz],
                  [zx - xz, xy + yx, yy - xx - zz, yz + zy], [xy - yx, zx + xz, yz + zy, zz - xx - yy]])
    e = np.linalg.eigvalsh(np.moveaxis(N, 2, 0))
    return (e[:, 3] - e[:, 2]) / np.abs(e).max(1), c


@pytest.mark.parametrize("hyps", [64, 257, 2048, 2049])
def test_thin_triples_match_the_oracle(hyps):
    """Four pixels in five lie on two neighbouring rows of a wall, so a third of the triples are lines but
    for 4 mm: their gaps (near 1e-5) take the FP64 rotations, in warps that also hold refined solves; up to
    2048 hypotheses the rotations are shared by 16 lanes.  A leaf a pixel, the wall moved rigidly and by half a
    millimetre of noise.  Bars: a solve rounds to some 50 units of 2^-52 over the gap (products, sums and
    rotations of a 4 x 4 matrix), two of them are compared, and the translation is the rotation's error times
    the centroid's distance."""
    W, H, D = 640, 48, 15
    intr = synth.Intrinsics.for_size(W, H)
    rng = np.random.default_rng(hyps)
    d = np.zeros((H, W), np.uint16)
    d[23:25, 100:420] = 2000
    other = rng.choice(np.setdiff1d(np.arange(W * H), np.arange(23 * W, 25 * W)), 160, replace=False)
    d.reshape(-1)[other] = rng.integers(1000, 3500, 160)
    pose = synth.look_pose(np.array([1.2, -0.7, 1.5]), 0.8, -0.3)
    cam = oracle.camera_points(d, intr, np.arange(W * H))
    modes = np.zeros((1, 1 << D, 1, 12), np.float32)
    modes[0, :W * H, 0, :3] = cam @ pose[:3, :3].T + pose[:3, 3] + rng.normal(0, 5e-4, cam.shape)
    n_modes = np.zeros((1, 1 << D), np.uint8)
    n_modes[0, :W * H] = 1
    leaves = np.arange(W * H, dtype=np.uint16).reshape(1, H, W)
    nodes = synth.random_forest_nodes(1, D, seed=3)
    want, ok, tries = oracle.generate_hypotheses(d, intr, leaves, oracle.Forest(nodes, modes, n_modes),
                                                 oracle.RansacParams(n_hyps=hyps, batch=8, seed=3))
    assert ok.all()
    gap, centre = _gaps(d, intr, leaves, oracle.Forest(nodes, modes, n_modes), tries, 3)
    thin, clear = gap < 4e-4, gap > 6e-4
    pair = np.arange(hyps // 2) * 2
    assert thin.sum() >= hyps // 8 and ((thin[pair] & clear[pair + 1]) | (clear[pair] & thin[pair + 1])).any()
    prm = B.ransac_params(n_hyps=hyps, batch=8, seed=3)
    poses = torch.zeros((hyps, 12), dtype=torch.float64, device=DEV)
    valid = torch.zeros(hyps, dtype=torch.int32, device=DEV)
    n_tries = torch.zeros(hyps, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.ransac_workspace_size(W, H, prm), dtype=torch.uint8, device=DEV)
    du, lu = (torch.from_numpy(a.view(np.int16)).to(DEV) for a in (d, leaves))
    B.ransac_hypotheses(B.Forest(nodes, modes, n_modes, max_modes=1), du, lu, intr, prm, ws, poses, valid, n_tries)
    torch.cuda.synchronize()
    assert np.array_equal(n_tries.cpu().numpy(), tries) and valid.cpu().numpy().all()
    got = poses.cpu().numpy().reshape(hyps, 3, 4)
    bar = 100 * 2.0**-52 / gap
    err = np.abs(got - want[:, :3])
    assert (err[:, :, :3].max(axis=(1, 2)) <= bar).all(), (err[:, :, :3].max(axis=(1, 2)) / bar).max()
    assert (err[:, :, 3].max(axis=1) <= bar * (1 + np.linalg.norm(centre, axis=1))).all()
