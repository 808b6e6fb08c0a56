"""The fused adjoint leaves out kernels whose quadratic form makes every
moment over an item's residual points a fixed-point zero.  Where that bound
can go wrong: needle kernels (large forms right next to the centre; thin discs
are in the CPU test of the bound, their float forms are too coarse for this bar),
supports wider than 1 (moments scale with r^2), large and tiny residuals, and
items whose kernels do not fit the remembered list."""
import numpy as np
import pytest

import synth
from gpu_util import oracle_view, per_kernel_errors, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


def _kernels(m, lengths, w, seed=11):
    P = synth.init_kernels(seed, m, length_range=(0.1, 0.2), rotate=True)
    g = synth.rng(seed + 1)
    P[3:6] = 1.0 / np.stack([np.full(m, v) * g.uniform(0.8, 1.25, m) for v in lengths]).astype(np.float32)
    P[9] = g.normal(0.0, w, m)
    return P


CASES = [
    ("needle", 96, (0.30, 0.02, 0.02), 0.1, 24),
    ("wide", 64, (0.9, 0.3, 0.05), 0.1, 24),       # r^2 well above 1
    ("loud", 96, (0.30, 0.05, 0.02), 6.0, 24),     # residuals of order 100
    ("quiet", 96, (0.30, 0.05, 0.02), 1e-4, 24),
    ("many", 640, (0.60, 0.30, 0.10), 0.05, 17),   # every kernel reaches every item: the list is walked again
]


@pytest.mark.parametrize("name,m,lengths,w,n", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("warps", [1, 2, 4])
def test_fused_gradients_of_stretched_kernels(orc, name, m, lengths, w, n, warps):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import build, field
    build.build()
    x, y, z = synth.grid(n)
    S = synth.sdf_torus(x, y, z)
    P = _kernels(m, lengths, w)
    pb = field.Problem(x, y, z, S, P, m, synth.spacing(n))
    pb.test_src = (x, y, z, S, np.asarray(P, np.float64))
    pb.cfg.fwd_warps = warps
    pb.build_neighbors()
    pb.forward_backward()
    fused = pb.grad.cpu().numpy()
    assert pb.status()[0] == 0
    h = oracle_view(pb, orc)
    E = pb.err[:pb.n].cpu().numpy().astype(np.float64)
    g_o, _ = orc.backward(h["x"], h["y"], h["z"], E, np.asarray(P, np.float64), m)
    for a, b in ((0, 3), (3, 6), (6, 9), (9, 10)):
        assert rel_l2(fused[a:b], g_o[a:b]) <= 1e-4
    # kernel by kernel: a kernel left out wrongly cannot hide under the norm
    assert max(per_kernel_errors(fused, g_o)) <= 1.0
