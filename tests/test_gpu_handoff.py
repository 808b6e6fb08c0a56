"""Work items handed between the warps of a forward block: fields whose blocks
take one item or two (the first record is the one that a block makes itself),
with 2, 4 and 8 warps per item.  A batch of one field is handed its items by
other code; both must give the same bits, and the oracle's values."""
import numpy as np
import pytest

import synth
from gpu_util import oracle_view, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(3, 4), (9, 40), (24, 96), (44, 200)])
@pytest.mark.parametrize("warps", [2, 4, 8])
def test_first_items_with_several_warps(orc, n, m, warps):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import _native as N, batch, build, field
    build.build()
    x, y, z = synth.grid(n)
    S = synth.sdf_torus(x, y, z) + np.float32(0.01)
    P = synth.init_kernels(5, m, length_range=(0.1, 0.4), rotate=True)
    made = []
    for _ in range(2):
        pb = field.Problem(x, y, z, S, P, m, synth.spacing(n), cap=2 * m, cfg=N.config_default(fwd_warps=warps))
        pb.test_src = (x, y, z, S, None)
        made.append(pb)
    one, other = made
    b = batch.Batch([other], fwd_warps=warps)
    for _ in range(3):
        one.epoch()
        b.epoch()
    torch.cuda.synchronize()
    assert torch.equal(one.psi, other.psi) and torch.equal(one.err, other.err) and torch.equal(one.mask, other.mask)
    assert torch.equal(one.p, other.p) and torch.equal(one.stats[:10], other.stats[:10])
    one.build_neighbors()
    one.forward_backward()
    h = oracle_view(one, orc)
    P1 = one.p[:, :one.m()].cpu().numpy().astype(np.float64)
    psi, _, mask, st = orc.forward(h["x"], h["y"], h["z"], h["t"], P1, one.m())
    assert np.abs(one.psi[:one.n].cpu().numpy() - psi).max() <= 1e-5 * float(np.abs(h["t"]).max())
    assert int(one.stats[4].item()) == int(st[4])
