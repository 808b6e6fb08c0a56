"""Surface metrics through the point grid against the oracle's all-pairs search:
the set sizes where the search changes, flat, collinear and coincident sets
(empty axes of the box), duplicated points (ties go to the lowest index), far
apart sets, outliers that stretch the grid, and coordinates far from zero."""
import numpy as np
import pytest

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _unit(g, n):
    v = g.normal(size=(n, 3))
    return (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.float32)


def _set(g, kind, n):
    p = g.uniform(-1, 1, (n, 3))
    if kind == "sphere":
        p /= np.linalg.norm(p, axis=1, keepdims=True)
    elif kind == "flat":
        p[:, 2] = 0.25
    elif kind == "line":
        p[:, 1:] = 0.5
    elif kind == "point":
        p[:] = 0.125
    elif kind == "twice":
        p[n // 2:2 * (n // 2)] = p[:n // 2]
    elif kind == "outlier":
        p *= 0.01
        p[n // 3] = 50.0
    elif kind == "away":
        p = p * 0.1 + 1000.0
    return p.astype(np.float32)


CASES = [("sphere", 1, "sphere", 1), ("sphere", 7, "sphere", 2000), ("sphere", 1023, "sphere", 1024),
         ("sphere", 1025, "sphere", 8193), ("flat", 3000, "sphere", 3000), ("line", 1500, "flat", 1500),
         ("point", 1200, "sphere", 1100), ("twice", 4097, "twice", 3001), ("outlier", 2048, "sphere", 2049),
         ("away", 2000, "sphere", 2000), ("away", 1500, "away", 5000)]


@pytest.mark.parametrize("ka,na,kb,nb", CASES)
def test_metrics_match_all_pairs(orc, ka, na, kb, nb):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build
    build.build()
    g = np.random.default_rng(na * 7 + nb)
    A, B, nA, nB = _set(g, ka, na), _set(g, kb, nb), _unit(g, na), _unit(g, nb)
    if ka == "twice":
        B[: nb // 3] = A[: nb // 3]  # exact hits, several candidates at distance zero
    d = [torch.as_tensor(v, device="cuda") for v in (A, nA, B, nB)]
    guard = 64
    scr = torch.full((2 * (na + nb) + 6 + guard,), 7.0, dtype=torch.float64, device="cuda")
    got = N.serbf_surface_metrics(d[0], d[1], na, d[2], d[3], nb, scr)
    want = orc.surface_metrics(A, nA, B, nB)
    assert got[0] == want[0]  # a selected value
    assert got[1] == pytest.approx(want[1], rel=1e-12) and got[2] == pytest.approx(want[2], rel=1e-12)
    assert bool((scr[-guard:] == 7.0).all())  # nothing beyond the documented scratch
    assert N.serbf_surface_metrics(d[0], d[1], na, d[2], d[3], nb, scr) == got


@pytest.mark.parametrize("n", [2, 17, 18, 40])
def test_extraction_scan_edges(orc, n):
    """Cube counts below, at and above a scan tile (16^3 = 4096 cubes), every cube crossed."""
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build
    build.build()
    g = np.random.default_rng(n)
    f = g.normal(size=n ** 3).astype(np.float32)
    want = orc.marching_tets(f, (n, n, n), (-1, -1, -1), 2.0 / (n - 1))
    fd = torch.as_tensor(f, device="cuda")
    scratch = torch.zeros((n - 1) ** 3 + 1, dtype=torch.int64, device="cuda")
    tri = torch.zeros(max(len(want), 1), 9, device="cuda")
    rc, nt = N.serbf_marching_tets(fd, (n, n, n), (-1.0, -1.0, -1.0), 2.0 / (n - 1), 0.0, tri, len(tri), scratch)
    assert rc == N.SERBF_OK and nt == len(want)
    np.testing.assert_array_equal(tri.cpu().numpy()[:nt], want)
    ns = 5000
    u = g.uniform(size=(ns, 3))
    pts, nrm = torch.zeros(ns, 3, device="cuda"), torch.zeros(ns, 3, device="cuda")
    cum = torch.zeros(nt + 1, dtype=torch.int64, device="cuda")
    N.serbf_sample_surface(tri, nt, torch.as_tensor(u, device="cuda"), ns, pts, nrm, cum)
    p_o, n_o = orc.sample_surface(want, u)
    np.testing.assert_array_equal(pts.cpu().numpy(), p_o)
    np.testing.assert_array_equal(nrm.cpu().numpy(), n_o)
