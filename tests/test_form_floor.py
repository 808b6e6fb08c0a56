"""The bound by which the fused adjoint leaves a kernel out (forward.cu,
form_floor and form_limit), restated in float32 numpy, against float64
moments: whenever it holds, every moment of the kernel over the item's
residual points, as the float pair loop may compute it, is below half a unit
of the 2^-36 fixed point."""
import numpy as np
import pytest

import synth

f32 = np.float32
LOG2E = 1.4426950408889634


def rotation(P):
    sx, cx, sy, cy, sz, cz = (fn(P[r].astype(np.float64)) for r in (6, 7, 8) for fn in (np.sin, np.cos))
    return np.array([[cx * cy, -cz * sx - sy * sz * cx, sx * sz - cx * cz * sy],
                     [cy * sx, cx * cz - sx * sy * sz, -sz * cx - cz * sx * sy],
                     [sy, cy * sz, cy * cz]])


def records(P):
    R, e = rotation(P), LOG2E * P[3:6].astype(np.float64) ** 2
    Q = np.einsum("kam,km,kbm->abm", R, e, R)
    r2 = (f32(-np.log(1e-7)) / (P[3:6] * P[3:6]).min(0)).astype(f32)
    return Q, r2, np.sqrt(e.max(0)).astype(f32)


def floor_of(c, Q, r2, l, mid, hd):
    with np.errstate(invalid="ignore"):
        d = (mid[:, None] - c).astype(f32)
        q = np.einsum("am,abm,bm->m", d.astype(np.float64), Q, d.astype(np.float64)).astype(f32)
        eps = f32(1.6e-5) * l * l * r2
        s = np.sqrt(q - eps) - f32(1.0001) * l * f32(hd)
        lg = np.maximum((r2.view(np.uint32) >> 23).astype(np.int64) - 126, 0)
        return np.where(s > 0, s * s - eps - lg, f32(0) * s)


def limit_of(emax, cnt):
    e = int(f32(emax).view(np.uint32)) >> 23
    return np.inf if e >= 255 else 38 + (e - 126) + int(cnt).bit_length()


@pytest.mark.parametrize("lengths", [(0.15, 0.15, 0.15), (0.3, 0.02, 0.02), (0.25, 0.25, 0.004), (0.9, 0.3, 0.05), (3.0, 0.5, 0.001)])
@pytest.mark.parametrize("emax", [1e-6, 0.02, 1.5, 300.0])
def test_left_out_kernels_add_nothing(lengths, emax):
    g = synth.rng(5)
    m, out = 400, 0
    P = synth.init_kernels(6, m, length_range=(0.1, 0.2), rotate=True)
    P[3:6] = (1.0 / np.stack([v * g.uniform(0.7, 1.4, m) for v in lengths])).astype(f32)
    Q, r2, l = records(P)
    err = 16 * 2.0 ** -24 * l.astype(np.float64) ** 2  # float error of a form, per |Delta|^2
    for k in range(40):
        n = int(g.integers(1, 65))
        p = (g.uniform(-1, 1, 3) + g.uniform(-0.5, 0.5, (n, 3)) * g.choice([0.01, 0.05, 0.3])).astype(f32)
        E = (g.uniform(-1, 1, n) * emax).astype(f32)
        lo, hi = p.min(0), p.max(0)
        mid = (f32(0.5) * (lo + hi)).astype(f32)
        hd = f32(0.5001) * np.sqrt(((hi - lo) ** 2).sum(dtype=f32))
        gone = floor_of(P[0:3], Q, r2, l, mid, hd) > limit_of(np.abs(E).max(), n)
        D = p.astype(np.float64)[:, :, None] - P[0:3].astype(np.float64)  # n x 3 x m
        d2 = (D ** 2).sum(1)
        q = np.einsum("nam,abm,nbm->nm", D, Q, D) - err * d2  # the least the pair loop can see
        s = np.where(d2 < r2, np.abs(E)[:, None] * np.exp2(-q), 0.0)
        most = (s * np.maximum(1.0, d2)).sum(0) * (1 + 1e-4)
        assert (most[gone] < 2.0 ** -37).all()
        reach = (d2 < r2).any(0)
        out += int((gone & reach).sum())
    assert out > 0 or lengths[0] == lengths[2]  # stretched kernels do get left out


def test_residuals_that_are_not_finite_leave_nothing_out():
    assert limit_of(np.inf, 3) == np.inf and limit_of(np.nan, 64) == np.inf
