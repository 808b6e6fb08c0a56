"""Workloads of the SE-RBFNet fitting path, each through the calls that a program makes.

A fit is a sequence of Algorithm 3 epochs (neighbour rebuild, forward, adjoint, optimiser step, deletion and
addition checks), replayed as a CUDA graph; around it stand the initial kernels, mini-batches, batches of
fields, the autograd function, the evaluation of a fit at new points, the explicit neighbour lists and the
surface metrics.  Sizes are those of the repository's own workloads (synth.CONFIGS, synth.batch_workload, the
paper's 40 000 samples in batches of 10 000, 10^5 samples per surface) and sizes between them.

Inputs are analytic signed distances (sphere, torus, unions of random primitives) and random kernels, all
made from the seed.  An epoch is measured as one of a resumed fit: the checkpoint (parameters, Adam moments,
optimiser state, kernel count) is restored at its beginning, so that every pass does the same epoch.
"""
import math

import numpy as np
import torch

from paper_2505_02350_gb300 import _native as N
from paper_2505_02350_gb300 import autograd, batch, field

EPS, TAU1, TAU2 = 1e-7, 0.9, 1.1
LR, BETA1, BETA2, ADAM_EPS = 0.01, 0.9, 0.999, 1e-8
RESUMED = 25  # optimiser steps done before the measured epoch
FWD_FLOPS, ADJ_FLOPS = 26, 52  # arithmetic of one forward and of one adjoint pair
RESIDUAL = 0.3  # about the share of the points that carry a residual


def spacing(n):
    return 2.0 / (n - 1)


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest fit: a sphere on 32^3 with 64 equal kernels (latency and launches)
        dict(name="epoch_32", kind="epoch", shape="sphere", grid=32, coarse=0, band=0.0, m=64, iso=True, sf=4, kahan=0),
        # a small fit after its coarse-to-fine refinement, 32^3 + 64^3 points
        dict(name="epoch_64", kind="epoch", shape="torus", grid=64, coarse=32, band=0.0, m=512, iso=False, sf=4, kahan=0),
        # an odd grid with compensated sums, on default-sized super cells
        dict(name="epoch_97_comp", kind="epoch", shape="prims12", grid=97, coarse=0, band=0.0, m=1500, iso=False, sf=4, kahan=1),
        # an ordinary fit of a complex shape, 128^3 points
        dict(name="epoch_128", kind="epoch", shape="prims20", grid=128, coarse=0, band=0.0, m=4096, iso=False, sf=2, kahan=0),
        # the largest single field: a narrow band of 256^3 and every 8th far point, 9.4 million points
        dict(name="epoch_256_band", kind="epoch", shape="prims60", grid=256, coarse=0, band=0.56, m=16384, iso=False, sf=2, kahan=0),
        # many small fits advanced together, uneven grids and kernel counts
        dict(name="batch_16", kind="batch", fields=16, grid_max=96, m_max=1024),
        # Algorithm 3 with the paper's mini-batches: 40 000 samples, batches of 10 000
        dict(name="minibatch_40k", kind="minibatch", n=40000, size=10000, m=900),
        # the field inside a user's own loss: forward and adjoint of an arbitrary upstream gradient
        dict(name="autograd_64", kind="autograd", shape="torus", grid=64, n=0, m=512),
        # a fit evaluated at new points (the extraction grid), in the caller's order
        dict(name="query_129", kind="query", grid=129, n=0, m=2048),
        # initial kernels of a fit (Algorithm 1), once per shape
        dict(name="init_64", kind="init", grid=64),
        # explicit neighbour lists, both orders (analysis, export)
        dict(name="lists_64", kind="lists", grid=64, m=512),
        # surface of a fit against the true one: extraction, samples, HD / CD / CS
        dict(name="surface_129", kind="surface", grid=129, samples=100000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["epoch", "epoch", "epoch", "batch", "minibatch", "autograd", "query", "init", "lists", "surface"])
    if kind == "epoch":
        g = _log(rng, 24, 200)
        band = 0.56 if g > 140 else 0.0
        m = _log(rng, 48, 40 * g)
        return dict(kind=kind, shape=rng.choice(["sphere", "torus", "prims7", "prims33"]), grid=g,
                    coarse=g // 2 if rng.random() < 0.3 and not band else 0, band=band, m=m,
                    iso=rng.random() < 0.3 and m < 400, sf=rng.choice([2, 3, 4, 4]), kahan=int(rng.random() < 0.25))
    if kind == "batch":
        return dict(kind=kind, fields=rng.randint(3, 20), grid_max=rng.choice([48, 64, 96]), m_max=_log(rng, 100, 1500))
    if kind == "minibatch":
        return dict(kind=kind, n=_log(rng, 9000, 80000), size=rng.choice([4096, 8192, 10000, 12345]), m=_log(rng, 100, 2000))
    if kind == "autograd":
        g = _log(rng, 24, 100)
        return dict(kind=kind, shape=rng.choice(["torus", "prims9"]), grid=g, n=rng.choice([0, _log(rng, 5000, 400000)]), m=_log(rng, 64, 2500))
    if kind == "query":
        return dict(kind=kind, grid=_log(rng, 33, 160), n=rng.choice([0, _log(rng, 3000, 2000000)]), m=_log(rng, 64, 4096))
    if kind == "init":
        return dict(kind=kind, grid=rng.randint(24, 80))
    if kind == "lists":
        return dict(kind=kind, grid=rng.randint(24, 80), m=_log(rng, 48, 700))
    return dict(kind=kind, grid=rng.randint(40, 150), samples=_log(rng, 5000, 120000))


# ---------------------------------------------------------------- inputs
def _generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed + 1) + salt)
    return g


def _rotation(g):
    q = torch.randn(4, generator=g, device="cuda")
    a, b, c, d = (q / q.norm()).tolist()
    return torch.tensor([[a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c)],
                         [2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b)],
                         [2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d]], device="cuda")


def _shape(name, g):
    """A function (points n x 3) -> signed distances (float32), the shape drawn from g."""
    u = torch.rand(2, generator=g, device="cuda").tolist()
    if name == "sphere":
        return lambda p: p.norm(dim=1) - (0.4 + 0.2 * u[0])
    if name == "torus":
        R, r = 0.45 + 0.1 * u[0], 0.17 + 0.06 * u[1]
        return lambda p: torch.hypot(torch.hypot(p[:, 0], p[:, 1]) - R, p[:, 2]) - r
    parts = [(k % 3, torch.rand(3, generator=g, device="cuda") * 1.4 - 0.7, _rotation(g),
              torch.rand(3, generator=g, device="cuda") * 0.25 + 0.05) for k in range(int(name[5:]))]

    def sdf(p):
        out = torch.full((p.shape[0],), math.inf, device="cuda")
        for kind, c, R, s in parts:
            l = (p - c) @ R
            if kind == 0:  # ellipsoid
                d = ((l / s).norm(dim=1) - 1.0) * s.min()
            elif kind == 1:  # box
                q = l.abs() - s
                d = q.clamp(min=0.0).norm(dim=1) + q.max(dim=1).values.clamp(max=0.0)
            else:  # capsule
                z = torch.maximum(torch.minimum(l[:, 2], s[2]), -s[2])
                d = torch.sqrt(l[:, 0] ** 2 + l[:, 1] ** 2 + (l[:, 2] - z) ** 2) - s[0]
            out = torch.minimum(out, d)
        return out
    return sdf


def _grid(n):
    """Vertex grid n^3 over [-1, 1]^3, x fastest."""
    a = (-1.0 + 2.0 * torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1)).float()
    z, y, x = torch.meshgrid(a, a, a, indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _cloud(n, sdf, g):
    """n scattered points, half of them drawn towards the surface."""
    p = torch.rand(n, 3, generator=g, device="cuda") * 2.0 - 1.0
    near = p[: n // 2]
    for _ in range(3):
        near = (near - 0.8 * sdf(near)[:, None] * near / near.norm(dim=1, keepdim=True).clamp(min=1e-3)).clamp(-1.0, 1.0)
    p[: n // 2] = (near + 0.02 * torch.randn(near.shape, generator=g, device="cuda")).clamp(-1.0, 1.0)
    return p


def _points(case, sdf, g):
    if case.get("n"):
        p = _cloud(case["n"], sdf, g)
        return p, sdf(p)
    p = _grid(case["grid"])
    if case.get("coarse"):
        p = torch.cat([_grid(case["coarse"]), p])
    S = sdf(p)
    if case.get("band"):
        # every 8th point, and of the others those nearest to the surface, `band` of all points in all
        near = S.abs()
        near[::8] = -1.0
        keep = torch.argsort(near, stable=True)[:int(case["band"] * S.numel())].sort().values
        p, S = p[keep], S[keep]
    return p, S


def _kernels(m, g, iso=False):
    """Random initial kernels (10 x m): centres, axis parameters, angles, weights."""
    P = torch.zeros(10, m, device="cuda")
    P[0:3] = torch.rand(3, m, generator=g, device="cuda") * 1.2 - 0.6
    w = torch.randn(m, generator=g, device="cuda") * 0.1
    if iso:
        P[3:6] = 1.0 / 0.15
    else:
        scale = (512.0 / m) ** (1.0 / 3.0)
        P[3:6] = 1.0 / ((torch.rand(3, m, generator=g, device="cuda") * 0.15 + 0.05) * scale)
        u = torch.rand(3, m, generator=g, device="cuda") * 2.0 - 1.0
        P[6], P[7], P[8] = math.pi * u[0], torch.asin(u[1]), math.pi * u[2]
    P[9] = w
    return P


def _np(t):
    return t.cpu().numpy()


def _problem(p, S, P, step, **kw):
    x, y, z = _np(p.t().contiguous())
    return field.Problem(x, y, z, _np(S), _np(P), P.shape[1], step, **kw)


def _moments(m, g):
    """Adam moments of a fit that has run for a while."""
    return 2.0 * torch.randn(10, m, generator=g, device="cuda"), 25.0 + 400.0 * torch.rand(10, m, generator=g, device="cuda")


def _resume(pb, am, av):
    """The problem as a checkpoint leaves it after RESUMED optimiser steps."""
    m = am.shape[1]
    pb.adam_m[:, :m] = am
    pb.adam_v[:, :m] = av
    st = pb.state_host()
    st.epoch = st.adam_t = RESUMED
    pb.state.copy_(torch.frombuffer(bytearray(bytes(st)), dtype=torch.uint8))


def _checkpoint(pbs):
    """(live buffers, saved copies) of everything an epoch changes, grouped by type."""
    groups = {}
    for pb in pbs:
        for t, c in zip((pb.p, pb.adam_m, pb.adam_v, pb.state, pb.m_dev), pb.snapshot()):
            live, saved = groups.setdefault(t.dtype, ([], []))
            live.append(t)
            saved.append(c)
    return list(groups.values())


def _restore(groups):
    for live, saved in groups:
        torch._foreach_copy_(live, saved)


def _graph(groups, epoch):
    """One CUDA graph: restore the checkpoint, then the epoch."""
    epoch()
    _restore(groups)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _restore(groups)
        epoch()
    torch.cuda.synchronize()
    return g


def _batch_sizes(case):
    grids = [v for v in (32, 48, 64, 96) if v <= case["grid_max"]]
    k = case["fields"]
    return [(grids[(3 * i) % len(grids)], int(round(64 * (case["m_max"] / 64.0) ** (i / max(1, k - 1))))) for i in range(k)]


def _epoch_inputs(case, seed):
    g = _generator(seed)
    p, S = _points(case, _shape(case["shape"], g), g)
    P = _kernels(case["m"], g, case["iso"])
    return p, S, P, _moments(case["m"], g)


def _field_inputs(seed, i, n, m):
    g = _generator(seed, 17 * (i + 1))
    p = _grid(n)
    S = _shape("prims%d" % (5 + (7 * i) % 36), g)(p)
    return p, S, _kernels(m, g), _moments(m, g)


def _minibatch_inputs(case, seed):
    g = _generator(seed)
    sdf = _shape("prims20", g)
    p = _cloud(case["n"], sdf, g)
    return p, sdf(p), _kernels(case["m"], g), _moments(case["m"], g)


def _points_inputs(case, seed):
    """Points, distances, kernels and an upstream gradient."""
    g = _generator(seed)
    p, S = _points(case, _shape(case.get("shape", "prims20"), g), g)
    P = _kernels(case["m"], g)
    return p, S, P, torch.randn(p.shape[0], generator=g, device="cuda")


# ---------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind == "epoch":
        p, S, P, (am, av) = _epoch_inputs(case, seed)
        cfg = N.config_default(kahan=case["kahan"])
        pb = _problem(p, S, P, spacing(case["grid"]), cfg=cfg, cap=2 * case["m"], super_factor=case["sf"])
        _resume(pb, am, av)
        groups = _checkpoint([pb])
        return dict(kind=kind, pb=pb, groups=groups, graph=_graph(groups, pb.epoch))
    if kind == "batch":
        pbs = []
        for i, (n, m) in enumerate(_batch_sizes(case)):
            p, S, P, (am, av) = _field_inputs(seed, i, n, m)
            pbs.append(_problem(p, S, P, spacing(n), cap=2 * m, super_cap=4096))
            _resume(pbs[-1], am, av)
        groups = _checkpoint(pbs)
        b = batch.Batch(pbs)
        return dict(kind=kind, b=b, pbs=pbs, groups=groups, graph=_graph(groups, b.epoch))
    if kind == "minibatch":
        p, S, P, (am, av) = _minibatch_inputs(case, seed)
        pb = _problem(p, S, P, spacing(64), cap=2 * case["m"])
        _resume(pb, am, av)
        return dict(kind=kind, pb=pb, groups=_checkpoint([pb]), mb=field.MiniBatch(pb, case["size"], seed=seed))
    if kind == "autograd":
        p, S, P, up = _points_inputs(case, seed)
        pb = _problem(p, S, P, spacing(case["grid"]))
        return dict(kind=kind, pb=pb, p=pb.p.clone().requires_grad_(True), up=up)
    if kind == "query":
        # the fitted field's own points come first; the query points replace them in every pass
        p, S, P, _ = _points_inputs(case, seed)
        pb = _problem(p, S, P, spacing(case["grid"]))
        xyz = p.t().contiguous()
        return dict(kind=kind, pb=pb, xyz=xyz, psi=torch.zeros_like(S))
    if kind == "init":
        g = _generator(seed)
        p, S = _points(case, _shape("prims20", g), g)
        return dict(kind=kind, pb=_problem(p, S, torch.zeros(10, 1, device="cuda"), spacing(case["grid"]), cap=8192))
    if kind == "lists":
        p, S, P, _ = _points_inputs(case, seed)
        pb = _problem(p, S, P, spacing(case["grid"]))
        n, m = pb.n, case["m"]
        kptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
        pptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        room = int(min(n * m, 3.0 * _pairs(n, m)))
        kcol = torch.zeros(room, dtype=torch.int32, device="cuda")
        pcol = torch.zeros(room, dtype=torch.int32, device="cuda")
        return dict(kind=kind, pb=pb, kptr=kptr, kcol=kcol, pptr=pptr, pcol=pcol)
    n, ns = case["grid"], case["samples"]
    g = _generator(seed)
    sdf = _shape("prims8", g)
    p = _grid(n)
    wave = 0.01 * torch.sin(9.0 * p[:, 0] + 1.0) * torch.cos(7.0 * p[:, 1]) * torch.sin(8.0 * p[:, 2] + 2.0)
    true = sdf(p)
    scratch = torch.zeros((n - 1) ** 3 + 1, dtype=torch.int64, device="cuda")
    room = 60 * n * n
    sides = []
    for f in (true, true + wave):
        sides.append(dict(f=f, tri=torch.zeros(room, 9, device="cuda"), cum=torch.zeros(room + 1, dtype=torch.int64, device="cuda"),
                          u=torch.rand(ns, 3, generator=g, dtype=torch.float64, device="cuda"),
                          pts=torch.zeros(ns, 3, device="cuda"), nrm=torch.zeros(ns, 3, device="cuda")))
    return dict(kind=kind, n=n, ns=ns, sides=sides, scratch=scratch, scr=torch.zeros(4 * ns + 6, dtype=torch.float64, device="cuda"))


# ---------------------------------------------------------------- run
def _fit_outputs(pb):
    return dict(psi=pb.psi[:pb.n], err=pb.err[:pb.n], grad=pb.grad, p=pb.p, adam_m=pb.adam_m, adam_v=pb.adam_v)


def run(s):
    kind = s["kind"]
    if kind == "epoch":
        s["graph"].replay()
        return _fit_outputs(s["pb"])
    if kind == "batch":
        s["graph"].replay()
        return [dict(psi=pb.psi[:pb.n], grad=pb.grad, p=pb.p) for pb in s["pbs"]]
    if kind == "minibatch":
        _restore(s["groups"])
        s["mb"].epoch()
        pb = s["pb"]
        return dict(grad=pb.grad, p=pb.p, adam_m=pb.adam_m, adam_v=pb.adam_v)
    if kind == "autograd":
        psi = autograd.erbf_field(s["pb"], s["p"])
        (grad,) = torch.autograd.grad(psi, s["p"], s["up"])
        return dict(psi=psi.detach(), grad=grad)
    pb = s.get("pb")
    if kind == "query":
        n = pb.n
        for dst, src in zip((pb.x_all, pb.y_all, pb.z_all), s["xyz"]):
            dst[:n] = src
        pb.bin()
        pb.build_neighbors()
        pb.forward()
        N.serbf_scatter(pb.psi[:n], pb.perm[:n], s["psi"], n)
        return s["psi"]
    if kind == "init":
        found = pb.init_kernels()
        return dict(found=found, p=pb.p, m=pb.m_dev)
    if kind == "lists":
        pb.build_neighbors(kmajor=N.csr(s["kptr"], s["kcol"]), pmajor=N.csr(s["pptr"], s["pcol"]))
        return dict(kptr=s["kptr"], kcol=s["kcol"], pptr=s["pptr"], pcol=s["pcol"])
    n, ns = s["n"], s["ns"]
    for d in s["sides"]:
        _rc, nt = N.serbf_marching_tets(d["f"], (n, n, n), (-1.0, -1.0, -1.0), spacing(n), 0.0, d["tri"], len(d["tri"]), s["scratch"])
        N.serbf_sample_surface(d["tri"], nt, d["u"], ns, d["pts"], d["nrm"], d["cum"])
    a, b = s["sides"]
    hd, cd, cs = N.serbf_surface_metrics(a["pts"], a["nrm"], ns, b["pts"], b["nrm"], ns, s["scr"])
    return dict(tri=[a["tri"], b["tri"]], pts=[a["pts"], b["pts"]], nrm=[a["nrm"], b["nrm"]], hd=hd, cd=cd, cs=cs)


# ---------------------------------------------------------------- work
def _pairs(n, m, iso=False):
    """Expected support pairs: n points of [-1, 1]^3, m kernels with centres in [-0.6, 0.6]^3."""
    r = math.sqrt(-math.log(EPS)) * (0.15 if iso else 0.1625 * (512.0 / m) ** (1.0 / 3.0))
    return n * m * min(1.0, 4.0 / 3.0 * math.pi * r ** 3 / 8.0) * 0.8


def _case_points(case):
    if case.get("n"):
        return case["n"]
    n = case["grid"] ** 3 + case.get("coarse", 0) ** 3
    return int(n * case["band"]) if case.get("band") else n


def _epoch_work(n, m, iso=False):
    pairs = _pairs(n, m, iso)
    return n * 25 + m * 320, pairs * (FWD_FLOPS + RESIDUAL * ADJ_FLOPS)


def work(case):
    kind = case["kind"]
    if kind == "epoch":
        b, f = _epoch_work(_case_points(case), case["m"], case["iso"])
    elif kind == "batch":
        w = [_epoch_work(n ** 3, m) for n, m in _batch_sizes(case)]
        b, f = sum(v[0] for v in w), sum(v[1] for v in w)
    elif kind == "minibatch":
        b, f = _epoch_work(case["n"], case["m"])
        b += (math.ceil(case["n"] / case["size"]) - 1) * case["m"] * 320 + case["n"] * 4
    elif kind == "autograd":
        n, pairs = _case_points(case), _pairs(_case_points(case), case["m"])
        b, f = n * 36 + case["m"] * 80, pairs * (FWD_FLOPS + ADJ_FLOPS)
    elif kind == "query":
        n = _case_points(case)
        b, f = n * 16 + case["m"] * 40, _pairs(n, case["m"]) * FWD_FLOPS
    elif kind == "init":
        b, f = case["grid"] ** 3 * 20, case["grid"] ** 3 * 10
    elif kind == "lists":
        n, pairs = _case_points(case), _pairs(_case_points(case), case["m"])
        b, f = n * 20 + case["m"] * 24 + pairs * 8, pairs * 9
    else:
        n, ns = case["grid"], case["samples"]
        b, f = 2 * (n ** 3 * 4 + 60 * n * n * 36 / 4 + ns * 48), 2 * ns * 17 * 9
    return dict(bytes=float(b), flops=float(f))


# ---------------------------------------------------------------- 64-bit values
def _rotations(P):
    sx, cx, sy, cy, sz, cz = P[6].sin(), P[6].cos(), P[7].sin(), P[7].cos(), P[8].sin(), P[8].cos()
    o = torch.zeros_like(sx)
    R = torch.stack([cx * cy, -cz * sx - sy * sz * cx, sx * sz - cx * cz * sy, cy * sx, cx * cz - sx * sy * sz,
                     -sz * cx - cz * sx * sy, sy, cy * sz, cy * cz]).reshape(3, 3, -1)
    Ry = torch.stack([-cx * sy, -cx * cy * sz, -cx * cy * cz, -sx * sy, -sx * cy * sz, -sx * cy * cz, cy, -sy * sz,
                      -sy * cz]).reshape(3, 3, -1)
    Rx = torch.stack([-R[1, 0], -R[1, 1], -R[1, 2], R[0, 0], R[0, 1], R[0, 2], o, o, o]).reshape(3, 3, -1)
    Rz = torch.stack([o, R[0, 2], -R[0, 1], o, R[1, 2], -R[1, 1], o, R[2, 2], -R[2, 1]]).reshape(3, 3, -1)
    return R, (Rx, Ry, Rz)


def _field64(p, P, residual=None):
    """Psi (Eq. 3-26 over the supports of Eq. 3-15-1) and, with residual(psi, first, last) -> E, the App. A
    gradients of sum E^2 as float64 (10 x m), E held fixed."""
    p, P = p.double(), P.double()
    n, m = p.shape[0], P.shape[1]
    R, dR = _rotations(P)
    d2 = P[3:6] ** 2
    A = torch.einsum("kam,km,kbm->abm", R, d2, R)
    c = P[0:3]
    Ac = torch.einsum("abm,bm->am", A, c)
    coef = torch.stack([(c * Ac).sum(0), -2 * Ac[0], -2 * Ac[1], -2 * Ac[2], A[0, 0], 2 * A[0, 1], 2 * A[0, 2], A[1, 1],
                        2 * A[1, 2], A[2, 2]])
    r2 = -math.log(EPS) / d2.min(0).values
    ball = torch.stack([(c * c).sum(0) - r2, -2 * c[0], -2 * c[1], -2 * c[2]])
    a = P[9] * P[9].abs()
    psi = torch.empty(n, dtype=torch.float64, device="cuda")
    M = torch.zeros(10, m, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // m)
    for i in range(0, n, step):
        x, y, z = p[i:i + step].t()
        one = torch.ones_like(x)
        mono = torch.stack([one, x, y, z, x * x, x * y, x * z, y * y, y * z, z * z], 1)
        phi = mono @ coef
        phi.neg_().exp_()
        phi *= (mono[:, :4] @ ball + (x * x + y * y + z * z)[:, None]) < 0
        psi[i:i + step] = phi @ a
        if residual is not None:
            E = residual(psi[i:i + step], i, min(n, i + step))
            M += (mono * E[:, None]).t() @ phi
    if residual is None:
        return psi, None
    # moments about the kernels' centres, in their frames
    S0, W1 = M[0], M[1:4] - c * M[0]
    X2 = torch.stack([M[4], M[5], M[6], M[5], M[7], M[8], M[6], M[8], M[9]]).reshape(3, 3, m)
    W2 = X2 - torch.einsum("am,bm->abm", M[1:4], c) - torch.einsum("am,bm->abm", c, M[1:4]) + torch.einsum("am,bm->abm", c, c) * S0
    M2 = torch.einsum("kam,abm,lbm->klm", R, W2, R)
    G = torch.zeros(10, m, dtype=torch.float64, device="cuda")
    G[9] = 4 * P[9].abs() * S0
    for k in range(3):
        G[3 + k] = -4 * a * P[3 + k] * M2[k, k]
        K = torch.einsum("kam,lam->klm", dR[k], R)
        G[6 + k] = -4 * a * (d2[:, None] * K * M2).sum((0, 1))
    G[0:3] = 4 * a * torch.einsum("kam,km,kbm,bm->am", R, d2, R, W1)
    return psi, G


def _targets(S):
    """Eq. 3-10, rounded to the stored float."""
    S = S.double()
    m = S.min()
    return (2 * torch.exp(-math.log(2.0) / m ** 2 * (S - m) ** 2)).float().double()


def _masked(t):
    def residual(psi, i, j):
        u = t[i:j]
        return torch.where(((u > TAU1) & (u < TAU2)) | ((u <= TAU1) & (psi > TAU1)) | ((u >= TAU2) & (psi < TAU2)), psi - u, 0.0)
    return residual


def _adam(P, G, m, v, t):
    """One Adam update in place (t: steps done after it)."""
    m.mul_(BETA1).add_(G, alpha=1 - BETA1)
    v.mul_(BETA2).addcmul_(G, G, value=1 - BETA2)
    P -= LR * (m / (1 - BETA1 ** t)) / ((v / (1 - BETA2 ** t)).sqrt() + ADAM_EPS)


def _binned(p, step, sf):
    """Order of the points by (super cell, cell, index), cells of 4 grid spacings."""
    h = np.float32(4 * step)
    o = np.float32(-1.0 - 0.5 * step)
    n = int(math.ceil((2.0 + step) / (4 * step) - 1e-6))
    k = torch.floor((p - float(o)) / torch.tensor(float(h), device="cuda")).clamp(0, n - 1).long()
    s, l = k // sf, k % sf
    ns = -(-n // sf)
    key = ((s[:, 2] * ns + s[:, 1]) * ns + s[:, 0]) * sf ** 3 + (l[:, 2] * sf + l[:, 1]) * sf + l[:, 0]
    return torch.argsort(key, stable=True)


def _padded(G, cap):
    return torch.nn.functional.pad(G, (0, cap - G.shape[1]))


def _epoch64(p, S, P, am, av, step, sf):
    o = _binned(p, step, sf)
    p, t = p[o], _targets(S)[o]
    residual = _masked(t)
    psi, G = _field64(p, P, residual)
    P, am, av = P.double(), am.double(), av.double()
    _adam(P, G, am, av, RESUMED + 1)
    cap = 2 * P.shape[1]
    return dict(psi=psi, err=residual(psi, 0, psi.numel()), grad=_padded(G, cap), p=_padded(P, cap), adam_m=_padded(am, cap),
                adam_v=_padded(av, cap))


def _init64(case, seed):
    """Algorithm 1 and Eq. 3-12; the spheres' membership is decided on float distances, as it is defined."""
    g = _generator(seed)
    p, S = _points(case, _shape("prims20", g), g)
    o = _binned(p, spacing(case["grid"]), 4)
    p, S, t = p[o], S[o], _targets(S)[o]
    inside = torch.nonzero((t > 1.0) & (t < 2.0)).reshape(-1)
    inside = inside[torch.argsort(S[inside].abs(), descending=True, stable=True)]
    q, r = p[inside], S[inside].abs()
    r2 = (r * r).tolist()
    alive = torch.ones(inside.numel(), dtype=torch.bool, device="cuda")
    chosen = []
    for k in range(inside.numel()):
        if k % 64 == 0:
            left = alive[k:].cpu().numpy()
            base = k
        if not left[k - base]:
            continue
        if not bool(alive[k]):
            continue
        chosen.append(k)
        d = (q - q[k]).double()
        e = (d[:, 0] * d[:, 0]).float().double()
        e = (d[:, 1] * d[:, 1] + e).float().double()
        e = (d[:, 2] * d[:, 2] + e).float()
        alive &= e > r2[k]
        alive[k] = False
    c = q[chosen].double()
    w = t[inside[chosen]]
    m = len(chosen)
    near = torch.full((m,), math.inf, dtype=torch.float64, device="cuda")
    for i in range(0, m, 1024):
        D = torch.cdist(c[i:i + 1024], c, compute_mode="donot_use_mm_for_euclid_dist")
        D[torch.arange(D.shape[0], device="cuda"), torch.arange(i, i + D.shape[0], device="cuda")] = math.inf
        near[i:i + 1024] = D.min(1).values
    P = torch.zeros(10, 8192, dtype=torch.float64, device="cuda")
    k = min(m, 8192)
    P[0:3, :k] = c.t()[:, :k]
    P[3:6, :k] = (2 * torch.sqrt(-torch.log(1e-3 / (w * w))) / near)[:k]
    P[9, :k] = w[:k]
    return dict(found=None, p=P, m=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "epoch":
        if _case_points(case) * case["m"] > 2e10:
            return None
        p, S, P, (am, av) = _epoch_inputs(case, seed)
        return _epoch64(p, S, P, am, av, spacing(case["grid"]), case["sf"])
    if kind == "batch":
        out = []
        for i, (n, m) in enumerate(_batch_sizes(case)):
            p, S, P, (am, av) = _field_inputs(seed, i, n, m)
            r = _epoch64(p, S, P, am, av, spacing(n), 4)
            out.append(dict(psi=r["psi"], grad=r["grad"], p=r["p"]))
        return out
    if kind == "minibatch":
        p, S, P, (am, av) = _minibatch_inputs(case, seed)
        o = _binned(p, spacing(64), 4)
        p, t = p[o], _targets(S)[o]
        order = torch.as_tensor(np.random.default_rng(seed).permutation(case["n"]).astype(np.int64), device="cuda")
        P, am, av = P.double(), am.double(), av.double()
        for k, i in enumerate(range(0, case["n"], case["size"])):
            sel = order[i:i + case["size"]]
            _, G = _field64(p[sel], P, _masked(t[sel]))
            _adam(P, G, am, av, RESUMED + 1 + k)
        cap = 2 * case["m"]
        return dict(grad=_padded(G, cap), p=_padded(P, cap), adam_m=_padded(am, cap), adam_v=_padded(av, cap))
    if kind == "autograd":
        p, _, P, up = _points_inputs(case, seed)
        o = _binned(p, spacing(case["grid"]), 4)
        psi, G = _field64(p[o], P, lambda v, i, j: 0.5 * up[i:j].double())
        return dict(psi=psi, grad=G)
    if kind == "query":
        p, _, P, _ = _points_inputs(case, seed)
        return _field64(p, P)[0]
    if kind == "init":
        return _init64(case, seed)
    return None  # neighbour lists are whole numbers; a surface's triangles and samples follow float decisions
