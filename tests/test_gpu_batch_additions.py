"""Batched epochs in which some fields add kernels and others do not: one field,
a few, more fields than a launch has blocks per SM, all at once and none.
Additions are spread over the blocks in another way than in the single-field
call; the kernels, their order and all state must be the same bits."""
import numpy as np
import pytest

import synth
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _fields(count, due):
    from paper_2505_02350_gb300 import _native as N, field
    out = []
    for i in range(count):
        n = (9, 14, 21, 33)[i % 4]
        x, y, z = synth.grid(n)
        S = synth.shape_sdf("prims%d" % (5 + i % 7), 3 + i, x, y, z)
        m = 6 + i % 5
        P = synth.init_kernels(40 + i, m, length_range=(0.1, 0.4), rotate=True)
        pb = field.Problem(x, y, z, S, P, m, synth.spacing(n), cap=m + (3 if i % 6 == 5 else 200), super_cap=256)
        pb.cfg.k_l2, pb.cfg.tau_l2 = 2, 1e30  # the L1 term goes on at epoch 2
        pb.cfg.k_l1, pb.cfg.tau_l1 = (3, 1e30) if due(i) else (200, 0.0)
        pb.cfg.topk_frac = (0.01, 0.3, 0.0)[i % 3]
        pb.cfg.fwd_warps = 2
        N.serbf_state_init(pb.state, pb.cfg)
        out.append(pb)
    return out


@pytest.mark.parametrize("count,due", [(1, "all"), (5, "one"), (23, "all"), (23, "some"), (70, "some"), (33, "none"), (180, "some")])
def test_batched_additions_equal_single_field_additions(count, due):
    torch = torch_cuda()
    from paper_2505_02350_gb300 import batch, build
    build.build()
    is_due = {"all": lambda i: True, "none": lambda i: False, "one": lambda i: i == 3, "some": lambda i: i % 3 != 1}[due]
    singles, batched = _fields(count, is_due), _fields(count, is_due)
    bt = batch.Batch(batched, fwd_warps=2)
    grew = set()
    for e in range(7):
        before = [pb.m() for pb in singles]
        for pb in singles:
            pb.epoch()
        bt.epoch()
        torch.cuda.synchronize()
        for i, (a, b) in enumerate(zip(singles, batched)):
            if a.m() > before[i]:
                grew.add(i)
            assert a.m() == b.m(), (e, i)
            m = a.m()
            assert torch.equal(a.p[:, :m], b.p[:, :m]), (e, i)
            assert torch.equal(a.adam_m[:, :m], b.adam_m[:, :m]) and torch.equal(a.adam_v[:, :m], b.adam_v[:, :m])
            assert torch.equal(a.state, b.state) and torch.equal(a.stats[:10], b.stats[:10]), (e, i)
    assert all(is_due(i) for i in grew) and (len(grew) > 0 or due == "none")
    for a, b in zip(singles, batched):
        assert a.status() == b.status()
