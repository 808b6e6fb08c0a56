"""The rows into which the standalone adjoint deals the chunks of a super cell
(chunk_rows.cuh, the code itself, compiled for the host): a row per chunk on
even sets, and a number of rows bounded by the average super cell on sets with
one dense super cell, where a row per chunk made every kernel look at as many
empty rows in all other super cells of its support."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_02350_gb300", "csrc")
HARNESS = """
#include "chunk_rows.cuh"
extern "C" int rows(long long tiles, long long supers, int most) { return serbf::chunk_rows(tiles, supers, most); }
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunk_rows")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "h.so"), str(d / "h.cpp")])
    lib = C.CDLL(str(d / "h.so"))
    lib.rows.argtypes = [C.c_longlong, C.c_longlong, C.c_int]
    return lib.rows


@pytest.mark.parametrize("supers", [1, 27, 125, 4913, 68921])
@pytest.mark.parametrize("chunks", [1, 4, 9])
def test_even_sets_have_a_row_per_chunk(rows, supers, chunks):
    assert rows(32 * chunks * supers, supers, chunks) == chunks


@pytest.mark.parametrize("supers", [64, 4913, 68921])
@pytest.mark.parametrize("dense", [40, 977, 65535, 1 << 21])
def test_one_dense_super_cell_does_not_add_rows_to_the_others(rows, supers, dense):
    tiles = 32 * dense + supers  # the others hold one tile each
    r = rows(tiles, supers, dense)
    assert 1 <= r <= dense
    assert r * supers <= 4 * (tiles // 32) + 4 * supers


def test_no_points(rows):
    assert rows(0, 27, 0) == 0
