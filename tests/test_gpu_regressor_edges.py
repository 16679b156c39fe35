"""The regressor's convolutions, backward-weight and loss kernels where their tiles are cut: one cell,
rows and columns of partial tiles (8 x 16 cells forward, 8 x 8 backward-weight, 16 x 8 outputs of layer
1), more images than one tile each, and a map with more tiles than CTAs."""
import numpy as np
import pytest
import torch

from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth
from test_gpu_regressor import ORIGIN, _cosines, _flat, _oracle_gradients, _unflat
from test_gpu_regressor import params  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _views(W, H, n, seed):
    rng = np.random.default_rng(seed)
    depth = rng.integers(800, 4000, (n, H, W)).astype(np.uint16)
    depth[rng.random((n, H, W)) < 0.1] = 0
    colour = rng.integers(0, 256, (n, H, W, 4)).astype(np.uint8)
    poses = [synth.look_pose(np.array([1.5, 2.0, 1.2]), 0.7 * k, 0.0) for k in range(n)]
    return synth.Intrinsics.for_size(W, H), poses, depth, colour


def _step(view, flat):
    intr, poses, depth, colour = view
    n, H, W = depth.shape
    reg = B.Regressor(flat, origin=ORIGIN)
    ws = torch.empty(B.regressor_workspace_size(n, W, H, True), dtype=torch.uint8, device=DEV)
    ws.fill_(0xFF)  # NaNs where a kernel reads what none has written
    loss = torch.zeros(1, dtype=torch.float32, device=DEV)
    d = torch.from_numpy(depth.view(np.int16)).to(DEV)
    c = torch.from_numpy(colour).to(DEV)
    out = []
    for _ in range(2):  # the second pass finds the first one's counters and partial sums
        B.regressor_gradients(reg, d, c, intr, poses, ws, loss)
        torch.cuda.synchronize()
        out.append((float(loss.item()), reg.grads().copy()))
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
    return out[0]


SHAPES = [(8, 8, 1), (8, 136, 3), (136, 8, 2), (72, 40, 5), (264, 72, 2), (648, 328, 1)]


@pytest.mark.parametrize("W,H,n", SHAPES)
def test_both_convolution_paths_give_the_same_bits(params, W, H, n):  # noqa: F811
    view, flat = _views(W, H, n, W + H + n), _flat(params)
    try:
        B.debug_conv_path(False)
        want = _step(view, flat)
    finally:
        B.debug_conv_path(True)
    got = _step(view, flat)
    assert np.isfinite(got[1]).all()
    assert got[0] == want[0] and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("W,H,n", [(8, 136, 2), (72, 40, 3)])
def test_gradients_match_the_oracle(params, W, H, n):  # noqa: F811
    """Every layer's cosine at least 0.99: activations and their gradients are kept in BF16 (2^-9
    relative each) through sixteen passes, sqrt(16) 2^-9 = 0.8 % of noise at most: a cosine of 0.9999."""
    view = _views(W, H, n, 7)
    intr, poses, depth, colour = view
    reg_loss, grads = _step(view, _flat(params))
    lo, want = _oracle_gradients(view, params, bf16_storage=True)
    assert abs(reg_loss - lo) <= 1e-2 * abs(lo)
    assert min(_cosines(_unflat(grads, params), want)) >= 0.99


@pytest.mark.parametrize("n,W,H", [(1, 64, 48), (16, 160, 120), (64, 640, 480)])
def test_workspaces_hold_one_padded_image(n, W, H):
    """Activations of 64 channels at 1/2, 1/4 and (six times) 1/8 of the size and the head's 32 bytes a cell; the
    padded input of the mma.sync path, 32 bytes a pixel, of one image; 256 bytes of alignment per buffer."""
    px = W * H
    forward = 128 * n * (px // 4 + px // 16 + 5 * px // 64) + 32 * n * px // 64
    assert B.regressor_workspace_size(n, W, H, False) <= forward + 32 * px + 16 * 256
