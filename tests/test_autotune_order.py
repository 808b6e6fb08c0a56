"""The autotuners time every split in the order that an epoch of a fit runs in:
the item order of a split needs two forwards (the mean cost, then the classes)
and a rebuild after them, before the timed calls."""
import types

import pytest

from paper_2505_02350_gb300 import batch, field


@pytest.fixture
def calls(monkeypatch):
    log = []

    class Event:
        def __init__(self, **kw):
            pass

        def record(self):
            log.append("record")

        def elapsed_time(self, other):
            return 1.0 + len(log)

    for mod in (field, batch):
        monkeypatch.setattr(mod.torch.cuda, "synchronize", lambda *a: None)
        monkeypatch.setattr(mod.torch.cuda, "Event", Event)
    return log


def _timed(log):
    """Calls before each split's first timed one, and the timed ones."""
    at = [i for i, v in enumerate(log) if v == "record"]
    assert len(at) == 8
    starts = [0] + [at[k] + 1 for k in (1, 3, 5)]
    return [(log[s:at[2 * k]], log[at[2 * k] + 1:at[2 * k + 1]]) for k, s in enumerate(starts)]


@pytest.mark.parametrize("fused", [True, False])
def test_problem(calls, fused):
    pb = types.SimpleNamespace(fused=fused, cfg=types.SimpleNamespace(fwd_warps=0), dev=None,
                               build_neighbors=lambda: calls.append("build"), forward=lambda: calls.append("run"),
                               forward_backward=lambda: calls.append("run"))
    times = field.Problem.autotune(pb, reps=3)
    assert list(times) == [1, 2, 4, 8] and pb.cfg.fwd_warps == 1
    for before, timed in _timed(calls):
        assert before[-3:] == ["run", "run", "build"]
        assert timed == ["run"] * 3


def test_batch(calls):
    restored = []
    bt = types.SimpleNamespace(snapshot=lambda: "snap", restore=restored.append, _init=lambda g: calls.append("init"),
                               epoch=lambda: calls.append("epoch"))
    times = batch.Batch.autotune(bt, reps=2)
    assert list(times) == [1, 2, 4, 8] and restored == ["snap"] * 4
    for before, timed in _timed(calls):
        assert before[-4:] == ["init"] + ["epoch"] * 3  # every epoch rebuilds and sorts first
        assert timed == ["epoch"] * 2
