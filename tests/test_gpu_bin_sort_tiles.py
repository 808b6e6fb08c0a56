"""Binning where the sort's tile changes (1024 elements up to 32768 points, 4096
beyond) and at the small tile's own edges, and coordinates that are not finite
(they must take the exact path of the cell index)."""
import numpy as np
import pytest

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _check(orc, p, cells, sf, h, origin):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build
    build.build()
    n = p.shape[1]
    grid = N.Grid()
    for k in range(3):
        grid.origin[k], grid.n[k] = origin, cells[k]
    grid.h = h
    x, y, z = (torch.as_tensor(v, device="cuda") for v in p)
    perm = torch.zeros(n, dtype=torch.int32, device="cuda")
    b = [torch.zeros(n, device="cuda") for _ in range(3)]
    sizes = N.WsSizes(n, 8, 40 ** 3, 0, 64, sf, 0)
    nbytes = N.serbf_workspace_bytes(sizes)
    mem = torch.zeros(nbytes + 256, dtype=torch.uint8, device="cuda")
    off = (-mem.data_ptr()) % 256
    ws = N.workspace_struct()
    N.serbf_workspace_init(ws, mem[off:off + nbytes], sizes)
    try:
        N.serbf_bin_points(x, y, z, grid, perm, *b, ws)
        want = orc.bin_points(p[0], p[1], p[2], (origin,) * 3, h, cells, sf).astype(np.int64)
        np.testing.assert_array_equal(perm.cpu().numpy().astype(np.int64), want)
        for k in range(3):
            np.testing.assert_array_equal(b[k].cpu().numpy(), p[k][want])
    finally:
        torch.cuda.synchronize()
        N.serbf_workspace_release(ws)


@pytest.mark.parametrize("n", [1023, 1024, 1025, 32767, 32768, 32769])
@pytest.mark.parametrize("cells,sf", [((5, 5, 5), 4), ((37, 20, 11), 3)])
def test_sort_tile_edges(orc, n, cells, sf):
    g = np.random.default_rng(n)
    _check(orc, g.uniform(-1, 1, (3, n)).astype(np.float32), cells, sf, np.float32(2.0 / max(cells)), np.float32(-1.0))


@pytest.mark.parametrize("sf", [1, 3, 4])
@pytest.mark.parametrize("h", [0.0731, 1e-3, 30.0])
def test_coordinates_that_are_not_finite(orc, sf, h):
    g = np.random.default_rng(7)
    p = g.uniform(-2, 2, (3, 3000)).astype(np.float32)
    odd = np.float32([np.nan, np.inf, -np.inf, 3e38, -3e38, 1e-42, -1e-42])
    for k in range(3):
        p[k, g.integers(0, 3000, 400)] = g.choice(odd, 400)
    _check(orc, p, (37, 20, 11), sf, np.float32(h), np.float32(-1.3))
