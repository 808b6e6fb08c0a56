"""The standalone adjoint on fields of very many super cells (more than a grid's
y dimension holds), where the binning and the fused pass work as well."""
import numpy as np
import pytest

import synth
from gpu_util import rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [40, 41])  # 64000 and 68921 super cells
def test_backward_with_many_super_cells(orc, cells):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import build, field
    build.build()
    n, m = 6000, 20
    g = np.random.default_rng(cells)
    x, y, z = (g.uniform(-1, 1, n).astype(np.float32) for _ in range(3))
    S = (np.sqrt(x * x + y * y + z * z) - 0.5).astype(np.float32) - np.float32(1.0)
    P = synth.init_kernels(4, m, length_range=(0.1, 0.3), rotate=True)
    pb = field.Problem(x, y, z, S, P, m, spacing=2.0 / (4 * cells - 1), super_factor=1, super_cap=32)
    assert pb.grid.n[0] == cells
    E = g.normal(size=n).astype(np.float32)
    perm = pb.perm[:n].cpu().numpy().astype(np.int64)
    pb.build_neighbors()
    pb.backward(torch.as_tensor(E, device="cuda"))
    want, pairs = orc.backward(x[perm], y[perm], z[perm], E.astype(np.float64), np.asarray(P, np.float64), m)
    assert int(pb.stats[5].item()) == pairs
    got = pb.grad[:, :m].cpu().numpy()
    for a, b in ((0, 3), (3, 6), (6, 9), (9, 10)):
        assert rel_l2(got[a:b], want[a:b]) <= 1e-4


@pytest.mark.parametrize("n,half", [(90011, 0.5), (60000, 0.98), (33000, 0.03)])
@pytest.mark.parametrize("kahan", [0, 1])
def test_backward_with_one_dense_super_cell(orc, n, half, kahan):
    """Rows of several chunks: a share of the points in one super cell, the rest scattered."""
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build, field
    build.build()
    m = 18
    g = np.random.default_rng(n)
    x, y, z = (g.uniform(-1, 1, n).astype(np.float32) for _ in range(3))
    k = int(half * n)
    for v in (x, y, z):
        v[:k] = (0.31 + 0.03 * v[:k]).astype(np.float32)
    S = (np.sqrt(x * x + y * y + z * z) - 0.5).astype(np.float32) - np.float32(1.0)
    P = synth.init_kernels(4, m, length_range=(0.1, 0.4), rotate=True)
    P[0:3, :6] = 0.3  # several kernels on the dense super cell
    pb = field.Problem(x, y, z, S, P, m, spacing=0.03, super_factor=2, cfg=N.config_default(kahan=kahan))
    E = np.where(g.uniform(size=n) < 0.9, g.normal(size=n), 0.0).astype(np.float32)
    perm = pb.perm[:n].cpu().numpy().astype(np.int64)
    pb.build_neighbors()
    pb.backward(torch.as_tensor(E, device="cuda"))
    want, pairs = orc.backward(x[perm], y[perm], z[perm], E.astype(np.float64), np.asarray(P, np.float64), m)
    assert int(pb.stats[5].item()) == pairs
    got = pb.grad[:, :m].cpu().numpy()
    for a, b in ((0, 3), (3, 6), (6, 9), (9, 10)):
        assert rel_l2(got[a:b], want[a:b]) <= 1e-4
