"""The regressor's convolutions, backward-weight and loss kernels where their tiles are cut: one cell,
rows and columns of partial tiles (8 x 16 cells forward, 8 x 8 backward-weight, 16 x 8 outputs of layer
1), more images than one tile each, and a map with more tiles than CTAs."""
import numpy as np
import pytest
import torch

from oracle import regressor as R
from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth
from test_gpu_regressor import ORIGIN, _cosines, _flat, _operands, _oracle_gradients, _unflat
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


# A layer's gradients against the FP64 oracle on the kernels' own activations (an oracle's own would round, and
# pass the ReLU, differently here and there): at most nine gradients are rounded to BF16 on the way (2^-9 at
# most each, 0.6 % together; 0.3 % in the mean square), doubled for what sums cancel
GRADIENT_BAR = 1.2e-2


def _activations(view, flat):
    """The stored activations and the output of a forward pass, from its workspace: the padded input of an image,
    then every layer's input, each on a 256-byte boundary."""
    _, _, depth, colour = view
    n, H, W = depth.shape
    ws = torch.zeros(B.regressor_workspace_size(n, W, H, False), dtype=torch.uint8, device=DEV)
    out = torch.zeros((n, H // 8, W // 8, 4), dtype=torch.float32, device=DEV)
    B.regressor_forward(B.Regressor(flat, origin=ORIGIN), torch.from_numpy(depth.view(np.int16)).to(DEV),
                        torch.from_numpy(colour).to(DEV), out, ws)
    torch.cuda.synchronize()
    acts, at = [], -(-H * W * 32 // 256) * 256
    for layer in range(1, 8):
        H, W = ((H - 1) // 2 + 1, (W - 1) // 2 + 1) if layer <= 3 else (H, W)
        size = n * H * W * 128
        acts.append(ws[at:at + size].view(torch.bfloat16).view(n, H, W, 64).double().cpu().numpy())
        at += -(-size // 256) * 256
    return acts, out.double().cpu().numpy()


def _operand_chain(view, params):
    """(weights, activations) for the oracle's backward pass, each layer's checked against the one before it."""
    _, _, depth, colour = view
    pq, x = _operands(params, np.stack([R.network_input(d, c) for d, c in zip(depth, colour)]))
    stored, out = _activations(view, _flat(params))
    acts = [x] + stored + [out]
    for k, (w, b) in enumerate(zip(pq.w, pq.b)):
        z = R.conv3x3(acts[k], w, b, R.STRIDES[k])
        z = np.maximum(z, 0.0) if k < 7 else z
        assert np.linalg.norm(acts[k + 1] - z) <= 2.0**-8 * np.linalg.norm(z), k  # (one rounding to BF16)
    return pq, acts


def _relative_errors(got, want):
    out = []
    for gw, ww, gb, wb in zip(got.w, want.w, got.b, want.b):
        a, b = np.concatenate([gw.ravel(), gb.ravel()]), np.concatenate([ww.ravel(), wb.ravel()])
        out.append(float(np.linalg.norm(a - b) / np.linalg.norm(b)))
    return out


@pytest.mark.parametrize("W,H,n", [(8, 136, 3), (136, 8, 2), (72, 40, 5), (264, 72, 2)])
def test_gradients_of_ragged_maps(params, W, H, n):  # noqa: F811
    view = _views(W, H, n, W + n)
    intr, poses, d, _ = view
    _, grads = _step(view, _flat(params))
    pq, acts = _operand_chain(view, params)
    tg = [R.cell_targets(d[k], intr, poses[k], ORIGIN) for k in range(n)]
    _, g = R.loss_and_grad_output(acts[8], np.stack([t[0] for t in tg]), np.stack([t[1] for t in tg]))
    assert max(_relative_errors(_unflat(grads, params), R.backward(pq, acts, g))) <= GRADIENT_BAR


def test_gradients_of_more_tiles_than_ctas(params):  # noqa: F811
    """700 images of 64 x 64, one backward-weight tile each in the inner layers (152 CTAs with a ring of four
    stages) and sixteen in the first (608 CTAs, three stages): five different images in no order and
    unequal numbers, so that the oracle needs those five alone, their gradients weighted."""
    few = _views(64, 64, 5, 3)
    order = np.random.default_rng(8).choice(5, 700, p=[0.4, 0.25, 0.2, 0.1, 0.05])
    times = np.bincount(order, minlength=5)
    intr, poses, d, c = few
    loss, grads = _step((intr, [poses[k] for k in order], d[order], c[order]), _flat(params))
    pq, acts = _operand_chain(few, params)
    tg = [R.cell_targets(d[k], intr, poses[k], ORIGIN) for k in range(5)]
    mask = np.stack([t[1] for t in tg])
    scored = mask.reshape(5, -1).sum(1)
    parts = [R.loss_and_grad_output(acts[8][k:k + 1], tg[k][0][None], mask[k:k + 1]) for k in range(5)]
    weight = times * scored / (times * scored).sum()  # (each part is a mean over its image's scored cells)
    want = R.backward(pq, acts, np.concatenate([w * g for w, (_, g) in zip(weight, parts)]))
    assert abs(loss - float(weight @ [p[0] for p in parts])) <= 1e-3 * abs(loss)
    assert max(_relative_errors(_unflat(grads, params), want)) <= GRADIENT_BAR
