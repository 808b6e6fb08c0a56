"""Tiles, boxes and work items of fields with few points per super cell, where a
warp takes a super cell and a block's warps together the dense ones: the edges of
the rule, of a warp's own tiles and of the last block, and empty super cells.
The lists and both item sets must hold exactly the oracle's pairs."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

# supers per axis at super factor 1: 1331 = 83 x 16 + 3 super cells, 8, and 512 and
# 729 to either side of the number that is on the chip at once
@pytest.mark.parametrize("cells,n,dense", [(11, 64 * 1331, 0), (11, 64 * 1331 + 1, 0), (11, 3000, 128), (11, 3000, 129),
                                           (11, 6000, 5000), (8, 4000, 2000), (9, 4000, 2000), (9, 64 * 729, 0),
                                           (2, 64 * 8, 0), (2, 40, 0), (11, 1, 0)])
def test_sparse_super_cells(orc, cells, n, dense):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build, field
    build.build()
    g = np.random.default_rng(n + dense)
    x, y, z = (g.uniform(-1, 1, n).astype(np.float32) for _ in range(3))
    for v in (x, y, z):
        v[:dense] = (0.2 + 0.01 * v[:dense]).astype(np.float32)  # inside one cell
    S = (np.sqrt(x * x + y * y + z * z) - 0.5).astype(np.float32) - np.float32(1.0)
    m = 30
    P = synth.init_kernels(3, m, length_range=(0.03, 0.2), centre=1.0, rotate=True)
    P[0:3, :4] = 0.2
    pb = field.Problem(x, y, z, S, P, m, spacing=2.0 / (4 * cells - 1), super_factor=1)
    assert pb.grid.n[0] == cells
    perm = pb.perm[:n].cpu().numpy().astype(np.int64)
    krow, kcol, prow, pcol = orc.neighbors(x[perm], y[perm], z[perm], np.asarray(P, np.float64), m)
    tot = int(krow[-1])
    kr, pr = torch.zeros(m + 1, dtype=torch.int64, device="cuda"), torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    kc, pc = (torch.zeros(max(tot, 1), dtype=torch.int32, device="cuda") for _ in range(2))
    rc, pairs = pb.build_neighbors(N.csr(kr, kc), N.csr(pr, pc))
    assert rc == N.SERBF_OK and pairs == tot
    np.testing.assert_array_equal(kr.cpu().numpy(), krow)
    np.testing.assert_array_equal(pr.cpu().numpy(), prow)
    np.testing.assert_array_equal(kc[:tot].cpu().numpy().astype(np.uint32), kcol)
    np.testing.assert_array_equal(pc[:tot].cpu().numpy().astype(np.uint32), pcol)
    t = pb.tb[:n].cpu().numpy()
    want = orc.forward(x[perm], y[perm], z[perm], t, np.asarray(P, np.float64), m)[0]
    for warps in (1, 2):  # items of four and of two tiles
        pb.cfg.fwd_warps = warps
        pb.psi.fill_(7.0)
        pb.forward()
        assert int(pb.stats[N.STAT_PAIRS_FWD].item()) == tot
        assert np.abs(pb.psi[:n].cpu().numpy() - want).max() <= 1e-5 * np.abs(t).max()
