"""The bound by which the fused adjoint leaves a kernel out (form_bound.cuh, the
code itself, compiled for the host) where its terms change sign: residuals so
small that the limit is below zero, boxes around the kernel's centre, supports
much wider than 1 (moments grow with r^2), as many residual points as an item
can hold.  Whenever it holds, every moment is below half a unit of 2^-36."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import synth
from test_form_floor import records

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_02350_gb300", "csrc")
HARNESS = """
struct float4 { float x, y, z, w; };
#include "form_bound.cuh"
extern "C" void floors(const float *k, const float *box, float *out, int m) {
    const float4 b = {box[0], box[1], box[2], 0.f};
    for (int j = 0; j < m; ++j) {
        const float *r = k + 12 * j;
        out[j] = serbf::form_floor({r[0], r[1], r[2], r[3]}, {r[4], r[5], r[6], r[7]}, {r[8], r[9], r[10], r[11]}, b, box[3]);
    }
}
extern "C" float limit(float emax, int cnt) { return serbf::form_limit(emax, cnt); }
"""
f32 = np.float32


@pytest.fixture(scope="module")
def bound(tmp_path_factory):
    d = tmp_path_factory.mktemp("form_bound")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o",
                           str(d / "h.so"), str(d / "h.cpp")])
    lib = C.CDLL(str(d / "h.so"))
    lib.limit.restype, lib.limit.argtypes = C.c_float, [C.c_float, C.c_int]
    return lib


def _floors(lib, P, Q, r2, l, mid, hd):
    k = np.stack([P[0], P[1], P[2], r2, Q[0, 0], Q[1, 1], Q[2, 2], P[9] * np.abs(P[9]), 2 * Q[0, 1], 2 * Q[0, 2],
                  2 * Q[1, 2], l], 1).astype(f32)
    box, out = np.append(mid, hd).astype(f32), np.zeros(P.shape[1], f32)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    lib.floors(ptr(np.ascontiguousarray(k)), ptr(box), ptr(out), P.shape[1])
    return out


@pytest.mark.parametrize("lengths,spread", [((0.15, 0.15, 0.15), 0.3), ((3.0, 2.0, 0.5), 6.0), ((20.0, 20.0, 20.0), 16.0), ((40.0, 3.0, 0.2), 30.0)])
@pytest.mark.parametrize("emax", [1e-16, 1e-14, 1e-13, 1e-12, 1e-11, 1e-9, 0.02])
@pytest.mark.parametrize("n", [1, 64, 128])
def test_left_out_kernels_add_nothing(bound, lengths, spread, emax, n):
    g = synth.rng(8)
    m = 200
    P = synth.init_kernels(6, m, length_range=(0.1, 0.2), rotate=True)
    P[3:6] = (1.0 / np.stack([v * g.uniform(0.7, 1.4, m) for v in lengths])).astype(f32)
    Q, r2, l = records(P)
    err = 16 * 2.0 ** -24 * l.astype(np.float64) ** 2  # float error of a form, per |Delta|^2
    for k in range(12):
        p = (g.uniform(-1, 1, 3) * spread * (k % 3) + g.uniform(-0.5, 0.5, (n, 3)) * g.choice([0.01, 0.3, 1.0]) * spread).astype(f32)
        E = (g.choice([-1.0, 1.0], n) * emax).astype(f32)
        lo, hi = p.min(0), p.max(0)
        mid = (f32(0.5) * (lo + hi)).astype(f32)
        hd = f32(0.5001) * np.sqrt(((hi - lo) ** 2).sum(dtype=f32))
        gone = _floors(bound, P, Q, r2, l, mid, hd) > bound.limit(float(np.abs(E).max()), n)
        D = p.astype(np.float64)[:, :, None] - P[0:3].astype(np.float64)  # n x 3 x m
        d2 = (D ** 2).sum(1)
        q = np.maximum(np.einsum("nam,abm,nbm->nm", D, Q, D) - err * d2, 0.0)  # the least the pair loop can see
        s = np.where(d2 < r2, np.abs(E)[:, None].astype(np.float64) * np.exp2(-q), 0.0)
        most = (s * np.maximum(1.0, d2)).sum(0) * (1 + 1e-4)
        assert (most[gone] < 2.0 ** -37).all()


def test_bound_says_something_and_nothing_for_what_is_not_finite(bound):
    P = synth.init_kernels(6, 4, length_range=(0.1, 0.2), rotate=True)
    P[0:3] = 0.0
    Q, r2, l = records(P)
    assert (_floors(bound, P, Q, r2, l, (1.1, 0.0, 0.0), 0.01) > 20).all()  # a box far down the form
    near = _floors(bound, P, Q, r2, l, (0.0, 0.0, 0.0), 0.5)  # a box around the centres: no bound, or NaN
    assert not (near > 0).any()
    for bad in (np.nan, np.inf):
        assert np.isnan(_floors(bound, P, Q, r2, l, (bad, 0.0, 0.0), np.inf)).all()
        assert bound.limit(float(bad), 3) == np.inf
