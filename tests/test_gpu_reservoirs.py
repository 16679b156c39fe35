"""The reservoirs of forest training against the oracle's (which offers pixel by pixel), at the edges
of the device's sort: one and two digits of leaf ids, grids below one block and not a multiple of it,
the largest leaf id, many offers to one leaf (every pixel in the same leaf: offers compete for slots
within and across steps of 32), frames without depth, and a second training of the same forest."""
import numpy as np
import pytest
import torch

import oracle
from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth
from test_gpu_allocator import Counting

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _frames(W, H, flat, seed):
    rng = np.random.default_rng(seed)
    for k in range(3):
        depth = np.full((H, W), 1500, np.uint16) if flat else rng.integers(300, 6000, (H, W)).astype(np.uint16)
        if not flat:
            depth[rng.random((H, W)) < 0.3] = 0
        if k == 1:
            depth[:] = 0
        rgba = np.full((H, W, 4), 90, np.uint8) if flat else rng.integers(0, 256, (H, W, 4)).astype(np.uint8)
        yield depth, rgba


@pytest.mark.parametrize("trees,depth,capacity,stride,W,H,flat", [
    (1, 3, 5, 1, 17, 11, False), (2, 8, 4, 1, 64, 32, False), (3, 9, 3, 2, 131, 97, False),
    (2, 16, 2, 1, 90, 50, False), (2, 16, 3, 1, 64, 65, True), (5, 10, 64, 3, 200, 152, False),
    (1, 1, 40, 1, 96, 72, True)])
def test_reservoirs_match_the_oracle(trees, depth, capacity, stride, W, H, flat):
    nodes = synth.random_forest_nodes(trees, depth, seed=depth, offset=130, depth_tau=300, colour_tau=64)
    if flat:  # equal probes everywhere and thresholds below zero: every pixel goes right, to the last leaf
        nodes["tau"] = -1
    intr = synth.Intrinsics.for_size(W, H, 12.0)
    pose = synth.look_pose(np.array([1.0, 2.0, 1.5]), 0.3, -0.1)
    f = B.Forest(nodes, max_modes=4)
    for seed in (5, (7 << 32) + 9):  # the second training starts from empty reservoirs
        want = oracle.Reservoirs(nodes, oracle.LeafParams(capacity=capacity, max_modes=4, seed=seed, stride=stride))
        B.forest_train_begin(f, B.train_params(capacity=capacity, stride=stride, seed=seed))
        for d, c in _frames(W, H, flat, seed % 1000):
            want.add_frame(intr, pose, d, c)
            B.forest_train_frame(f, intr, pose, torch.from_numpy(d.view(np.int16)).to(DEV), torch.from_numpy(c).to(DEV))
        samples, count = B.forest_train_reservoirs(f, capacity)
        so, co = want.contents()
        assert np.array_equal(count, co)
        assert np.array_equal(samples, so)
        if flat:
            assert count[:, -1].min() == min(capacity, 2 * len(range(0, W, stride)) * len(range(0, H, stride)))


class Limited(Counting):
    limit = 0

    def alloc(self, n):
        return super().alloc(n) if n <= self.limit else 0


@pytest.fixture
def limited():
    a = Limited()
    yield a
    B.set_allocator()


def test_a_frame_without_room_leaves_nothing_behind(limited):
    """Room for the reservoirs (4 KB) but not for the frame's scratch (16 bytes a pixel at least): the frame
    fails with nothing allocated or under way, so the next one, on another stream, starts a training."""
    W, H = 64, 48
    nodes = synth.random_forest_nodes(2, 4, seed=9)
    f = B.Forest(nodes, max_modes=4)
    intr, pose = synth.Intrinsics.for_size(W, H, 12.0), synth.look_pose(np.array([1.0, 2.0, 1.5]), 0.3, -0.1)
    (d, c), *_ = _frames(W, H, False, 3)
    dd, cc = torch.from_numpy(d.view(np.int16)).to(DEV), torch.from_numpy(c).to(DEV)
    torch.cuda.synchronize()
    B.forest_train_begin(f, B.train_params(capacity=8, stride=1, seed=5))
    limited.limit = 16 * W * H
    B.set_allocator(limited.alloc, limited.free)
    with pytest.raises(B.ReloError) as e:
        B.forest_train_frame(f, intr, pose, dd, cc)
    assert e.value.status == B.ENOMEM
    assert not limited.live
    samples, count = B.forest_train_reservoirs(f, 8)
    assert not samples.any() and not count.any()
    B.set_allocator()
    B.forest_train_frame(f, intr, pose, dd, cc, torch.cuda.Stream())
    want = oracle.Reservoirs(nodes, oracle.LeafParams(capacity=8, max_modes=4, seed=5, stride=1))
    want.add_frame(intr, pose, d, c)
    samples, count = B.forest_train_reservoirs(f, 8)
    so, co = want.contents()
    assert np.array_equal(count, co) and np.array_equal(samples, so)


@pytest.mark.parametrize("W,H,kept", [(64, 48, 16 << 20), (700, 600, 0)])
def test_training_gives_its_memory_back(limited, W, H, kept):
    """finish gives a scratch of over 16 MB back (700 x 600 pixels take 12 + 2 * 18 bytes each), end the
    reservoirs and the rest; reading and going on after finish are as before it, after end the training is over
    and the modes stay."""
    nodes = synth.random_forest_nodes(2, 4, seed=9)
    intr, pose = synth.Intrinsics.for_size(W, H, 12.0), synth.look_pose(np.array([1.0, 2.0, 1.5]), 0.3, -0.1)
    limited.limit = 1 << 30
    B.set_allocator(limited.alloc, limited.free)
    f = B.Forest(nodes, max_modes=4)
    own = dict(limited.live)
    want = oracle.Reservoirs(nodes, oracle.LeafParams(capacity=8, max_modes=4, seed=5, stride=1))
    B.forest_train_begin(f, B.train_params(capacity=8, stride=1, seed=5))
    for d, c in _frames(W, H, False, 3):
        want.add_frame(intr, pose, d, c)
        B.forest_train_frame(f, intr, pose, torch.from_numpy(d.view(np.int16)).to(DEV), torch.from_numpy(c).to(DEV))
        B.forest_train_finish(f)
        held = sum(n for q, (_, n) in limited.live.items() if q not in own)
        assert held <= 2 * 16 * (12 * 8 + 20) + kept
        samples, count = B.forest_train_reservoirs(f, 8)
        so, co = want.contents()
        assert np.array_equal(count, co) and np.array_equal(samples, so)
    modes = f.get_modes()
    B.forest_train_end(f)
    assert limited.live == own
    assert all(np.array_equal(a, b) for a, b in zip(f.get_modes(), modes)) and modes[1].any()
    with pytest.raises(B.ReloError) as e:
        B.forest_train_frame(f, intr, pose, torch.zeros((H, W), dtype=torch.int16, device=DEV),
                             torch.zeros((H, W, 4), dtype=torch.uint8, device=DEV))
    assert e.value.status == B.EINVAL
    B.forest_train_end(f)
