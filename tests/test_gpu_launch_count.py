"""Problem.launches_per_epoch against the kernel nodes of a captured epoch: dense
fields, fields of many sparse super cells (whose item order takes two launches
although they hold few points), and the rebuild's levels."""
import ctypes as C

import numpy as np
import pytest

import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _kernel_nodes(torch, fn):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    cu = C.CDLL("libcuda.so.1")
    raw, n = C.c_void_p(g.raw_cuda_graph()), C.c_size_t(0)
    assert cu.cuGraphGetNodes(raw, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(raw, nodes, C.byref(n)) == 0
    kinds = []
    for v in nodes[:n.value]:
        k = C.c_int(-1)
        assert cu.cuGraphNodeGetType(C.c_void_p(v), C.byref(k)) == 0
        kinds.append(k.value)
    return sum(k == 0 for k in kinds)  # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.mark.parametrize("n,cells,sf,levels", [(4000, 8, 4, 1), (4000, 8, 4, 2), (30000, 16, 2, 3), (60000, 40, 1, 1),
                                               (200000, 41, 1, 1), (40000, 64, 1, 0)])
def test_launches_of_an_epoch(n, cells, sf, levels):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build, field
    build.build()
    g = np.random.default_rng(n)
    x, y, z = (g.uniform(-1, 1, n).astype(np.float32) for _ in range(3))
    S = (np.sqrt(x * x + y * y + z * z) - 0.5).astype(np.float32) - np.float32(1.0)
    P = synth.init_kernels(3, 12, length_range=(0.1, 0.3), rotate=True)
    pb = field.Problem(x, y, z, S, P, 12, spacing=2.0 / (4 * cells - 1), super_factor=sf, super_cap=32, cap=64,
                       cfg=N.config_default(rebuild_levels=levels))
    assert pb.grid.n[0] == cells
    pb.epoch()
    torch.cuda.synchronize()
    assert _kernel_nodes(torch, pb.epoch) == pb.launches_per_epoch()
