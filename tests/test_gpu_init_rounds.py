"""Algorithm 1 in rounds (the next 1024 points settled at a time) against the
oracle's walk: fewer interior points than a round, rounds cut in the middle of
a sphere's points, dense rounds and the sparse ones that look for conflicts
first, super cells of other sizes."""
import numpy as np
import pytest

import synth
from gpu_util import oracle_view, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n,sf", [("sphere", 12, 4), ("sphere", 30, 2), ("torus", 40, 4), ("prims9", 44, 3), ("prims40", 52, 4)])
def test_centres_of_rounds_match_the_walk(orc, shape, n, sf):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import build, field
    build.build()
    x, y, z = synth.grid(n)
    S = synth.shape_sdf(shape, 7, x, y, z)
    P = np.zeros((10, 1), np.float32)
    pb = field.Problem(x, y, z, S, P, 1, synth.spacing(n), cap=1 << 14, super_factor=sf)
    pb.test_src = (x, y, z, S, None)
    for _ in range(2):  # the second walk starts from a used workspace
        found = pb.init_kernels()
    torch.cuda.synchronize()
    h = oracle_view(pb, orc)
    idx, want = orc.inscribed(h["x"], h["y"], h["z"], h["t"], h["S"])
    assert found == want == pb.m()
    got = pb.p[:3, :found].cpu().numpy()
    np.testing.assert_array_equal(got, np.stack([h[k][idx] for k in "xyz"]))
