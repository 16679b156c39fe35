"""relo_batch_launch_count against the kernel nodes of the batch's graph: forest and learned attempts, the
learned ones on both convolution paths, RANSAC in stages and in one persistent launch, and enough attempts
that a round's pixels are not split over CTAs (four launches a round, five where a further one adds the
split scores)."""
import ctypes

import pytest
import torch

from paper_1801_08361_gb300 import binding as B
from paper_1801_08361_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _kernel_nodes(bt, n):
    out = torch.zeros(n * B.RESULT_BYTES, dtype=torch.uint8, device=DEV)
    bt.run(out)
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bt.run(out)
        status, graph, nodes = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_size_t()
        assert cu.cuStreamGetCaptureInfo_v3(ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), ctypes.byref(status),
                                            None, ctypes.byref(graph), None, None, None) == 0
        assert status.value == 1
        assert cu.cuGraphGetNodes(graph, None, ctypes.byref(nodes)) == 0
        all_nodes = (ctypes.c_void_p * nodes.value)()
        assert cu.cuGraphGetNodes(graph, all_nodes, ctypes.byref(nodes)) == 0
        kinds = []
        for node in all_nodes:
            kind = ctypes.c_int()
            assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
            kinds.append(kind.value)
    return kinds.count(0)  # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.mark.parametrize("n,learned,tcgen05,persistent", [(1, 0, True, 0), (3, 2, True, 0), (2, 2, False, 0), (3, 1, True, 1),
                                                          (310, 0, True, 0)])
def test_launch_count_is_the_graphs(room, room_training, room_forest, n, learned, tcgen05, persistent):
    world, blocks = room
    scene = B.Scene(blocks, 16)
    forest = B.Forest(room_forest.nodes, room_forest.modes, room_forest.n_modes, max_modes=10)
    reg = B.Regressor(seed=9, origin=(2.0, 2.0, 1.5))
    intr = synth.Intrinsics.for_size(64, 48)
    pose = synth.query_poses(world, [f[1] for f in room_training], 1, seed=4)[0]
    items = [dict(scene_b=scene, forest_a=forest, scene_a=scene, intr=intr, pose_b=pose, seed=k) for k in range(n)]
    for k in range(learned):
        items[k]["regressor_a"] = reg
    prm = B.ransac_params(n_hyps=32, batch=40, max_tries=500)
    att = B.make_attempts(items)
    bt = B.Batch(att, prm, torch.empty(B.batch_workspace_size(att, prm), dtype=torch.uint8, device=DEV))
    bt.set_schedule(persistent=persistent)
    try:
        B.debug_conv_path(tcgen05)
        count = _kernel_nodes(bt, n)
        assert bt.launch_count == count
    finally:
        B.debug_conv_path(True)
    if n > 300:
        assert count == 2 + 1 + 1 + n // 257 + 2 + 2 + 4 * 5 + 1 + 2
