"""Binning at the sizes where its kernels change: one point, tile and sort-tile
edges, the largest number of sort blocks that sum the histograms themselves and
one more, a single cell, and grids with long runs of empty cells.  Order, cell
ranges (through the neighbour lists' tiles) and the tight boxes are whole or
selected values: they must be exact."""
import numpy as np
import pytest

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 4095, 4096, 4097, 32 * 4096, 32 * 4096 + 1, 300007])
@pytest.mark.parametrize("cells,sf", [((1, 1, 1), 4), ((7, 5, 9), 2), ((64, 64, 40), 4)])
def test_binned_order_at_edges(orc, n, cells, sf):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build
    build.build()
    g = np.random.default_rng(n + cells[0])
    p = g.uniform(-1, 1, (3, n)).astype(np.float32)
    p[:, : n // 2] *= np.float32(0.05)  # half of the points in few cells, the rest scattered
    grid = N.Grid()
    for k in range(3):
        grid.origin[k], grid.n[k] = -1.0, cells[k]
    grid.h = 2.0 / max(cells)
    x, y, z = (torch.as_tensor(v, device="cuda") for v in p)
    perm = torch.zeros(n, dtype=torch.int32, device="cuda")
    b = [torch.zeros(n, device="cuda") for _ in range(3)]
    sizes = N.WsSizes(n, 8, cells[0] * cells[1] * cells[2] * 8, 0, 64, sf, 0)
    nbytes = N.serbf_workspace_bytes(sizes)
    mem = torch.zeros(nbytes + 256, dtype=torch.uint8, device="cuda")
    off = (-mem.data_ptr()) % 256
    ws = N.workspace_struct()
    N.serbf_workspace_init(ws, mem[off:off + nbytes], sizes)
    try:
        for _ in range(2):  # a second binning of the same workspace finds its counters clear
            N.serbf_bin_points(x, y, z, grid, perm, *b, ws)
        want = orc.bin_points(p[0], p[1], p[2], (-1.0, -1.0, -1.0), grid.h, cells, sf).astype(np.int64)
        np.testing.assert_array_equal(perm.cpu().numpy().astype(np.int64), want)
        for k in range(3):
            np.testing.assert_array_equal(b[k].cpu().numpy(), p[k][want])
    finally:
        torch.cuda.synchronize()
        N.serbf_workspace_release(ws)


@pytest.mark.parametrize("sf", [1, 3, 4])
def test_points_on_and_beside_cell_faces(orc, sf):
    """Quotients at integers and one float to either side, beyond the grid on both
    sides and at magnitudes where the quotient has no fraction bits."""
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build
    build.build()
    cells, h, origin = (37, 20, 11), np.float32(0.0731), np.float32(-1.3)
    k = np.arange(-3, 60, dtype=np.float32)
    face = (origin + k * h).astype(np.float32)
    v = np.concatenate([face, np.nextafter(face, np.float32(9)), np.nextafter(face, np.float32(-9)),
                        np.float32([3e5, -3e5, 1e9, -1e9, 3e38, 0.0, -0.0])])
    g = np.random.default_rng(sf)
    p = np.stack([g.permutation(np.tile(v, 8)) for _ in range(3)]).astype(np.float32)
    n = p.shape[1]
    grid = N.Grid()
    for a in range(3):
        grid.origin[a], grid.n[a] = origin, cells[a]
    grid.h = h
    x, y, z = (torch.as_tensor(q, device="cuda") for q in p)
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
    finally:
        torch.cuda.synchronize()
        N.serbf_workspace_release(ws)
