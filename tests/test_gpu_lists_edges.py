"""Explicit neighbour lists where their launches can go wrong: one kernel, rows
whose super cells do not divide among the row's warps, kernels that reach
nothing or everything, row counts at the scan's tile (4096 points), ragged
clouds, no kernels at all."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,length,sf", [(1, 1, 0.1, 4), (33, 3, 0.4, 1), (4095, 40, 0.1, 2), (4096, 40, 0.1, 4), (4097, 65, 0.02, 3),
                                           (20011, 300, 0.05, 1), (20011, 0, 0.05, 4), (9000, 12, 5.0, 2)])
def test_lists_match_oracle(orc, n, m, length, sf):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build, field
    build.build()
    g = np.random.default_rng(n + m)
    x, y, z = (g.uniform(-1, 1, n).astype(np.float32) for _ in range(3))
    S = (np.sqrt(x * x + y * y + z * z) - 0.5).astype(np.float32) - np.float32(1.0)
    P = synth.init_kernels(3, max(m, 1), length=length, centre=1.4)
    pb = field.Problem(x, y, z, S, P, m, spacing=0.05, super_factor=sf)
    perm = pb.perm[:n].cpu().numpy().astype(np.int64)
    krow, kcol, prow, pcol = orc.neighbors(x[perm], y[perm], z[perm], np.asarray(P, np.float64), m)
    tot = int(krow[-1])
    kr, pr = torch.full((m + 1,), -1, dtype=torch.int64, device="cuda"), torch.full((n + 1,), -1, dtype=torch.int64, device="cuda")
    kc, pc = (torch.zeros(max(tot, 1), dtype=torch.int32, device="cuda") for _ in range(2))
    rc, pairs = pb.build_neighbors(N.csr(kr, kc), N.csr(pr, pc))
    assert rc == N.SERBF_OK and pairs == tot
    np.testing.assert_array_equal(kr.cpu().numpy(), krow)
    np.testing.assert_array_equal(pr.cpu().numpy(), prow)
    np.testing.assert_array_equal(kc[:tot].cpu().numpy().astype(np.uint32), kcol)
    np.testing.assert_array_equal(pc[:tot].cpu().numpy().astype(np.uint32), pcol)
    if tot > 1:  # a capacity one short: the size comes back, the rows are valid
        rc, pairs = pb.build_neighbors(N.csr(kr, kc[:tot - 1]))
        assert rc == N.SERBF_ECAPACITY and pairs == tot
        np.testing.assert_array_equal(kr.cpu().numpy(), krow)
