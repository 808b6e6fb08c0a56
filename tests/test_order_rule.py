"""Launches of the item order: the library's rule (order_rule.cuh, the code
itself, compiled for the host) against Problem.launches_per_epoch and against
the items that fields really have."""
import ctypes as C
import os
import subprocess
import types

import numpy as np
import pytest

from paper_2505_02350_gb300 import field

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_02350_gb300", "csrc")
HARNESS = """
#include "order_rule.cuh"
extern "C" int direct(long long points, long long supers) { return serbf::order_direct(points, supers); }
"""


@pytest.fixture(scope="module")
def direct(tmp_path_factory):
    d = tmp_path_factory.mktemp("order_rule")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")])
    lib = C.CDLL(str(d / "h.so"))
    lib.direct.argtypes = [C.c_longlong, C.c_longlong]
    return lambda n, s: bool(lib.direct(n, s))


def _launches(n, cells, sf):
    cfg = types.SimpleNamespace(rebuild_levels=1)
    pb = types.SimpleNamespace(n=n, cap=8, cfg=cfg, sizes=types.SimpleNamespace(super_factor=sf), grid=types.SimpleNamespace(n=[cells] * 3))
    return field.Problem.launches_per_epoch(pb)


@pytest.mark.parametrize("cells,sf", [(1, 4), (33, 4), (50, 1), (51, 1), (64, 1), (128, 2), (256, 4)])
@pytest.mark.parametrize("n", [1, 4096, 200000, 2_000_000, (1 << 22) - 64 * 729, (1 << 22) - 64, 1 << 22, 9_400_000])
def test_launch_count_follows_the_rule(direct, n, cells, sf):
    supers = (-(-cells // sf)) ** 3
    assert _launches(n, cells, sf) == (10 if direct(n, supers) else 11)


@pytest.mark.parametrize("supers", [1, 1000, 40000, 300000])
def test_one_launch_never_meets_more_items_than_its_counters_hold(direct, supers):
    """The most items that a number of points can make: as many super cells as
    possible hold one point more than whole items."""
    for n in (1, 63, 64, 65, 65536, 65537, 131072, 200000, 4_000_000, 1 << 22):
        used = np.minimum(n, supers)
        whole, extra = divmod(max(n - used, 0), 64)
        items = used + whole  # one point each, then 64 for every further item
        if direct(n, supers):
            assert items <= 128 * 1024
