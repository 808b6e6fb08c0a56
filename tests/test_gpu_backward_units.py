"""The standalone adjoint deals 32-tile chunks of super cells to its warps:
one super cell with all points (many chunks), one chunk per super cell, fewer
chunks than warps, sparse residuals (empty chunks), one point."""
import numpy as np
import pytest

import synth
from gpu_util import rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,spacing,sf,keep", [(1, 2, 0.1, 4, 1.0), (40000, 24, 1.0, 4, 1.0), (20000, 24, 0.05, 1, 1.0),
                                                 (9000, 70, 0.06, 2, 0.03), (33, 5, 0.2, 4, 1.0), (30011, 9, 0.02, 4, 0.5)])
@pytest.mark.parametrize("kahan", [0, 1])
def test_backward_matches_oracle(orc, n, m, spacing, sf, keep, kahan):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build, field
    build.build()
    g = np.random.default_rng(n)
    x, y, z = (g.uniform(-0.9, 0.9, n).astype(np.float32) for _ in range(3))
    S = (np.sqrt(x * x + y * y + z * z) - 0.5).astype(np.float32) - np.float32(1.0)
    P = synth.init_kernels(4, m, length_range=(0.1, 0.3), rotate=True)
    pb = field.Problem(x, y, z, S, P, m, spacing=spacing, super_factor=sf, cfg=N.config_default(kahan=kahan))
    E = np.where(g.uniform(size=n) < keep, g.normal(size=n), 0.0).astype(np.float32)
    perm = pb.perm[:n].cpu().numpy().astype(np.int64)
    pb.build_neighbors()
    pb.backward(torch.as_tensor(E, device="cuda"))
    want, pairs = orc.backward(x[perm], y[perm], z[perm], E.astype(np.float64), np.asarray(P, np.float64), m)
    assert int(pb.stats[5].item()) == pairs
    got = pb.grad[:, :m].cpu().numpy()
    for a, b in ((0, 3), (3, 6), (6, 9), (9, 10)):
        if np.abs(want[a:b]).max() > 0:
            assert rel_l2(got[a:b], want[a:b]) <= 1e-4
