"""Surface metrics of sets whose points lie in few cells of their grid (streamed
instead, from an eighth of the points in one cell on) against the oracle's
all-pairs search: shares around that eighth in one set or in both, equal
distances in the cluster, and the same sets in turn with even ones (the count
of the densest cell starts anew with every call)."""
import numpy as np
import pytest

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _set(g, n, share, step=0.0):
    """n points, `share` of them in one small cluster; step: on a lattice, so that distances tie."""
    p = g.uniform(-1, 1, (n, 3))
    k = int(round(share * n))
    q = g.uniform(-1, 1, (k, 3)) * 1e-3
    p[:k] = 0.3 + (np.round(q / step) * step if step else q)
    return g.permutation(p).astype(np.float32)


@pytest.mark.parametrize("na,sa,nb,sb", [(4096, 0.12, 4096, 0.13), (1024, 0.124, 9000, 0.126), (5000, 1.0, 5000, 0.0),
                                         (3000, 0.5, 1500, 0.5), (900, 0.5, 3000, 0.9), (8200, 0.125, 8200, 0.125)])
@pytest.mark.parametrize("step", [0.0, 2.5e-4])
def test_clusters_match_all_pairs(orc, na, sa, nb, sb, step):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, build
    build.build()
    g = np.random.default_rng(na + nb)
    unit = lambda n: (lambda v: (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.float32))(g.normal(size=(n, 3)))
    scr = torch.zeros(2 * (na + nb) + 6, dtype=torch.float64, device="cuda")
    nA, nB = unit(na), unit(nb)
    for A, B in ((_set(g, na, sa, step), _set(g, nb, sb, step)), (_set(g, na, 0.0), _set(g, nb, 0.0)),
                 (_set(g, na, sb, step), _set(g, nb, sa, step))):
        d = [torch.as_tensor(v, device="cuda") for v in (A, nA, B, nB)]
        got = N.serbf_surface_metrics(d[0], d[1], na, d[2], d[3], nb, scr)
        want = orc.surface_metrics(A, nA, B, nB)
        assert got[0] == want[0]
        assert got[1] == pytest.approx(want[1], rel=1e-12) and got[2] == pytest.approx(want[2], rel=1e-12)
