"""Warps per forward work item: the library's rule (warps_rule.cuh, the code
itself, compiled for the host) must choose a split within a tenth of the fastest
one measured, for fields of full and of sparse super cells, and a fixed split
must stand."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_02350_gb300", "csrc")
HARNESS = """
#include "warps_rule.cuh"
extern "C" int warps(long long items4, int sms, int fixed) { return serbf::forward_warps(items4, sms, fixed); }
"""
SMS = 152


@pytest.fixture(scope="module")
def warps(tmp_path_factory):
    d = tmp_path_factory.mktemp("warps_rule")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")])
    lib = C.CDLL(str(d / "h.so"))
    lib.warps.argtypes = [C.c_longlong, C.c_int, C.c_int]
    return lib.warps


# items of up to four tiles, and us of the fused call with 1, 2 and 4 warps
@pytest.mark.parametrize("items4,us", [
    # full super cells
    (256, (36, 35, 35)), (2304, (104, 59, 61)), (4096, (133, 82, 89)), (7200, (163, 148, 159)), (7200, (248, 193, 201)),
    (9100, (145, 137, 164)), (13500, (275, 251, 297)), (16384, (337, 309, 365)), (21500, (384, 385, 458)), (26500, (467, 476, 568)),
    (74000, (1671, 1817, 2109)), (41000, (552, 718, 979)),
    # a tile or less in each
    (8000, (55, 52, 62)), (15625, (90, 96, 117)), (29791, (134, 147, 189)), (39304, (166, 186, 241)),
    # the forward alone on those
    (8000, (37, 40, 47)), (29791, (88, 102, 131)), (39304, (111, 128, 166))])
def test_choice_is_near_the_fastest_split(warps, items4, us):
    took = dict(zip((1, 2, 4), us))[warps(items4, SMS, 0)]
    assert took <= 1.1 * min(us)


@pytest.mark.parametrize("fixed", [1, 2, 4, 8])
def test_fixed_split_stands(warps, fixed):
    assert warps(10, SMS, fixed) == fixed and warps(10 ** 7, SMS, fixed) == fixed


def test_edges(warps):
    assert [warps(v, SMS, 0) for v in (0, 50 * SMS - 1, 50 * SMS, 160 * SMS - 1, 160 * SMS)] == [4, 4, 2, 2, 1]
