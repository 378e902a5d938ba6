"""Timed cases of the RPM-FFT library: what its users call, over the sizes
they call it with.

Four kinds of case, each through the package's public entry points:

  gamma   one application of the Lippmann-Schwinger map (rpm.Context.apply_gamma)
  solve   one cell problem to tolerance (rpm.Context.solve)
  batch   effective stiffness of several cells (rpm.rpm_effective_stiffness_batch)
  fno     the learned warm start's network: a forward pass, or loss and gradients

Cells are periodic, with spheres (circles in 2D) of radius 5-10 % of the cell
side in a matrix of Young's modulus 1, Poisson ratio 0.3: the recipe of the
batched sweep.  `exact` restates each path in 64 bits with torch alone: the
map by torch.fft, the solution of the cell problem by conjugate gradients on
the compatible fields (the map's fixed point), the network by torch.fft and
autograd.
"""
import math
import random

import numpy as np
import torch

from paper_2003_07720_gb300 import fno, rpm

MODES = {"full": rpm.RPM_GAMMA_FULL_MAP, "linear": rpm.RPM_GAMMA_LINEAR,
         "raw": rpm.RPM_GAMMA_RAW_TAU}
XY_SIZES = (4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256)
Z_SIZES = (1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256)
NU = 0.3


def _gamma(name, nz, ny, nx, mode, phases=2, contrast=10.0):
    return {"name": name, "kind": "gamma", "nz": nz, "ny": ny, "nx": nx, "mode": mode,
            "phases": phases, "contrast": contrast}


def listed():
    return [
        # the smallest cells (unit cells of a materials scan, checks): launches and latency
        _gamma("gamma_16", 16, 16, 16, "full"),
        # a middle grid of the batched sweep; F_u z, which every growth of the basis applies
        _gamma("gamma_48", 48, 48, 48, "linear", contrast=100.0),
        # Gamma0 on a given polarization, on the grid the network is trained on
        _gamma("gamma_64", 64, 64, 64, "raw"),
        # the benchmark's grid, one fixed-point step of Eq. 3.9
        _gamma("gamma_128", 128, 128, 128, "full", contrast=1e-3),
        # the largest grid: stiff inclusions, the spectrum larger than the L2 cache
        _gamma("gamma_256", 256, 256, 256, "full", contrast=1e4),
        # a 2D plane-strain cell, as in the fibre study
        _gamma("gamma_plane_256", 1, 256, 256, "full", contrast=1e3),
        # a box with three different sides and three phases
        _gamma("gamma_box_24_96_48", 24, 96, 48, "linear", phases=3),
        # cold start with a growing basis: map, projections and small Newton solves
        {"name": "solve_cold_96", "kind": "solve", "n": 96, "contrast": 30.0, "warm": False,
         "steps": 65},
        # the benchmark's form: Algorithm 3 first, then RPM, on its grid
        {"name": "solve_warm_128", "kind": "solve", "n": 128, "contrast": 0.03, "warm": True,
         "steps": 50},
        # the batched sweep: small cells of two sizes, six loads each, eight workers
        {"name": "batch_32_48", "kind": "batch", "cells": 6, "small": 32, "large": 48,
         "contrast": 10.0, "workers": 8, "steps": 25},
        # one guess of the learned warm start at its training size
        {"name": "fno_forward_64", "kind": "fno", "n": 64, "modes": 12, "layers": 4, "batch": 1,
         "precision": "bf16", "grad": False},
        # one small training batch: loss and gradients of every parameter
        {"name": "fno_grad_32", "kind": "fno", "n": 32, "modes": 12, "layers": 4, "batch": 2,
         "precision": "bf16", "grad": True},
    ]


def draw(rng):
    kind = rng.random()
    if kind < 0.6:
        goal = math.exp(rng.uniform(math.log(16 ** 3), math.log(256 ** 3)))
        while True:
            shape = rng.random()
            if shape < 0.4:       # cube
                n = min(XY_SIZES, key=lambda s: abs(math.log(s ** 3 / goal)))
                nz, ny, nx = n, n, n
                goal = math.exp(rng.uniform(math.log(16 ** 3), math.log(256 ** 3)))
            elif shape < 0.55:    # plane
                nx = ny = rng.choice((64, 96, 128, 256))
                nz = 1
            elif shape < 0.75:    # square column or slab
                nx = ny = rng.choice(XY_SIZES[4:])
                nz = rng.choice(Z_SIZES[3:])
            else:                 # box
                nz, ny, nx = rng.choice(Z_SIZES[4:]), rng.choice(XY_SIZES[2:]), rng.choice(XY_SIZES[2:])
            if 4096 <= nz * ny * nx <= 256 ** 3:
                break
        c = _gamma("", nz, ny, nx, rng.choice(("full", "full", "linear", "raw")),
                   rng.choice((2, 2, 3, 5)), round(10.0 ** rng.uniform(-3.0, 3.0), 4))
    elif kind < 0.75:
        warm = rng.random() < 0.5
        c = {"name": "", "kind": "solve", "n": rng.choice((24, 32, 48, 64, 96)),
             "contrast": round(10.0 ** rng.uniform(-1.0, 1.3), 3), "warm": warm,
             "steps": 40}
    elif kind < 0.8:
        c = {"name": "", "kind": "batch", "cells": rng.randint(2, 6),
             "small": rng.choice((16, 24, 32)), "large": rng.choice((32, 48)),
             "contrast": round(10.0 ** rng.uniform(-1.0, 1.0), 3),
             "workers": rng.choice((4, 8)), "steps": 25}
    else:
        grad = rng.random() < 0.5
        n = rng.choice((24, 32, 40) if grad else (24, 32, 40, 48, 56, 64, 80, 96))
        room = max(1, (2 * 32 ** 3 if grad else 8 * 64 ** 3) // n ** 3)
        c = {"name": "", "kind": "fno", "n": n, "modes": rng.randint(4, 12),
             "layers": rng.randint(1, 4), "batch": min(room, rng.randint(1, 8)),
             "precision": rng.choice(("bf16", "bf16", "fp32")), "grad": grad}
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class Cell:
    """What the package asks of a cell: phase map, moduli, reference medium."""

    def __init__(self, phase, lam, mu, lam0, mu0):
        self.phase, self.lam, self.mu, self.lam0, self.mu0 = phase, lam, mu, lam0, mu0


def _lame(young):
    return young * NU / ((1 + NU) * (1 - 2 * NU)), young / (2 * (1 + NU))


def _cell(shape, contrast, phases, r, vf=0.2):
    """Spheres of radius U[0.05, 0.10] (at least two voxels) of the cell side,
    up to about a volume fraction vf; sphere k has phase 1 + k mod (phases - 1).
    Phase j's modulus is contrast ** (j / (phases - 1))."""
    dev = "cuda"
    axes = [(torch.arange(n, device=dev, dtype=torch.float32) + 0.5) / n for n in shape]
    solid = [n > 1 for n in shape]
    low = max(0.05, 2.0 / max(shape))
    phase = torch.zeros(shape, dtype=torch.uint8, device=dev)
    volume, k = 0.0, 0
    while volume < -math.log(1.0 - vf):   # overlapping spheres cover 1 - exp(-volume)
        rad = r.uniform(low, max(low, 0.10))
        d2 = torch.zeros((1, 1, 1), device=dev)
        for a, x in enumerate(axes):
            c = r.random()
            if solid[a]:
                d = x - c
                d = (d - torch.round(d)) ** 2
                d2 = d2 + d.view([-1 if b == a else 1 for b in range(3)])
        phase.masked_fill_(d2 < rad * rad, 1 + k % (phases - 1))
        volume += math.pi * rad ** 2 if sum(solid) == 2 else 4.0 / 3.0 * math.pi * rad ** 3
        k += 1
    young = [contrast ** (j / (phases - 1)) for j in range(phases)]
    lam, mu = zip(*(_lame(y) for y in young))
    lam0, mu0 = _lame(0.5 * (min(young) + max(young)))
    return Cell(phase, np.array(lam), np.array(mu), lam0, mu0)


def _load(r):
    """A macroscopic strain of unit Frobenius norm (shears counted twice)."""
    e = np.array([r.gauss(0.0, 1.0) for _ in range(6)])
    return e / math.sqrt(float(np.sum(np.array([1, 1, 1, 2, 2, 2]) * e * e)))


def _column(v):
    return torch.tensor(np.asarray(v), dtype=torch.float32, device="cuda").view(6, 1, 1, 1)


def _inputs(case, seed):
    """Everything that is made from the seed, before any object of the package."""
    r = random.Random(1000003 * seed + 17)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["kind"] == "gamma":
        shape = (case["nz"], case["ny"], case["nx"])
        cell = _cell(shape, case["contrast"], case["phases"], r)
        E = _load(r)
        field = torch.randn((6,) + shape, generator=g, device="cuda")
        if case["mode"] != "raw":        # an iterate: the mean strain and a fluctuation
            field = _column(E) + 0.2 * field
        return cell, E, field.contiguous()
    if case["kind"] == "solve":
        cell = _cell((case["n"],) * 3, case["contrast"], 2, r)
        return cell, _load(r)
    if case["kind"] == "batch":
        cells = [_cell((case["small"] if k % 2 == 0 else case["large"],) * 3, case["contrast"], 2, r)
                 for k in range(case["cells"])]
        for c in cells:
            c.phase = c.phase.cpu().numpy()   # the batch takes host maps
        return cells
    n, B, W = case["n"], case["batch"], fno.WIDTH
    feat = torch.empty((B, 2, n, n, n), device="cuda")
    for b in range(B):
        c = _cell((n, n, n), 10.0 ** r.uniform(-3.0, 3.0), 2, r, r.uniform(0.1, 0.35))
        fno.features(c.phase, list(zip(c.lam, c.mu)), feat[b])
    E = np.stack([_load(r) for _ in range(B)]).astype(np.float32)
    target = 0.5 * torch.randn((B, 6, n, n, n), generator=g, device="cuda")
    count = fno.param_count(case["modes"], case["layers"])
    p = torch.zeros(count, device="cuda")

    def normal(at, size, scale):
        p[at:at + size] = scale * torch.randn(size, generator=g, device="cuda")

    normal(0, 2 * W, 1 / math.sqrt(2))                        # P
    normal(2 * W, W, 0.1)                                     # p
    normal(3 * W, fno.COUT * W, 1 / math.sqrt(W))             # Q
    normal(3 * W + fno.COUT * W, fno.COUT, 0.1)               # q
    per = (count - fno.HEADER) // case["layers"]
    for l in range(case["layers"]):
        at = fno.HEADER + l * per
        normal(at, W * W, 1 / math.sqrt(W))                   # A
        normal(at + W * W, W, 0.1)                            # a
        size = per - W * W - W
        p[at + per - size:at + per] = torch.rand(size, generator=g, device="cuda") / (W * W)
    return feat, E, target, p


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gamma":
        cell, E, field = _inputs(case, seed)
        ctx = rpm.Context(cell, rpm.rpm_default_options(p_max=0))
        return {"kind": kind, "ctx": ctx, "E": E, "in": field, "out": torch.empty_like(field),
                "mode": MODES[case["mode"]]}
    if kind == "solve":
        cell, E = _inputs(case, seed)
        opts = rpm.rpm_default_options(warm_tol=1e-4 if case["warm"] else 0.0)
        eps = torch.empty((6,) + tuple(cell.phase.shape), device="cuda")
        return {"kind": kind, "ctx": rpm.Context(cell, opts), "E": E, "eps": eps,
                "sig": torch.empty_like(eps)}
    if kind == "batch":
        return {"kind": kind, "cells": _inputs(case, seed), "workers": case["workers"],
                "opts": rpm.rpm_default_options()}
    feat, E, target, p = _inputs(case, seed)
    net = fno.Fno(case["n"], case["modes"], case["layers"], case["batch"],
                  precision=case["precision"])
    net.set_params(p.cpu().numpy())
    s = {"kind": kind, "net": net, "feat": feat, "E": E, "target": target, "grad": case["grad"]}
    if case["grad"]:   # the host buffer a training program reads gradients into
        s["host"] = torch.empty(net.nparam, dtype=torch.float32, pin_memory=True)
    else:
        s["out"] = torch.empty_like(target)
    return s


def run(s):
    if s["kind"] == "gamma":
        s["ctx"].apply_gamma(s["in"], s["E"], s["out"], s["mode"])
        return s["out"]
    if s["kind"] == "solve":
        s["ctx"].solve(s["E"], eps_out=s["eps"], sig_out=s["sig"])
        return {"eps": s["eps"], "sig": s["sig"]}
    if s["kind"] == "batch":
        C, _, _, _ = rpm.rpm_effective_stiffness_batch(s["cells"], s["opts"], s["workers"])
        return C.astype(np.float32)   # means of float32 stress fields
    if not s["grad"]:
        s["net"].forward(s["feat"], s["E"], s["out"])
        return s["out"]
    loss = s["net"].loss_grad(s["feat"], s["E"], s["target"])
    net = s["net"]
    fno._ck(net.h, fno.lib().rpm_fno_get_grads(net.h, s["host"].data_ptr()))
    return {"loss": loss, "grads": s["host"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _map_flops(n):
    """Forward and inverse real 3D transforms of six components (2.5 n log2 n
    each), the polarization and the Green operator."""
    return n * (2 * 6 * 2.5 * math.log2(n) + 20 + 60)


def work(case):
    if case["kind"] == "gamma":
        n = case["nz"] * case["ny"] * case["nx"]
        return {"bytes": n * (48 + (case["mode"] != "raw")), "flops": _map_flops(n)}
    if case["kind"] == "solve":   # phase map in, strain and stress out; `steps` typical maps
        n = case["n"] ** 3
        return {"bytes": n * 49, "flops": case["steps"] * _map_flops(n)}
    if case["kind"] == "batch":
        half = (case["cells"] + 1) // 2
        sizes = [case["small"] ** 3] * half + [case["large"] ** 3] * (case["cells"] - half)
        return {"bytes": sum(sizes) + 288 * len(sizes),
                "flops": 6 * case["steps"] * sum(_map_flops(n) for n in sizes)}
    n, m, L, B, W = case["n"], case["modes"], case["layers"], case["batch"], fno.WIDTH
    modes = 4 * m ** 3
    params = fno.param_count(m, L)
    layer = 2 * W * 2.5 * n ** 3 * math.log2(n ** 3) + 8 * modes * W * W + n ** 3 * (2 * W * W + 10 * W)
    flops = B * (L * layer + n ** 3 * (4 * W + 12 * W))
    if not case["grad"]:
        return {"bytes": 4 * (params + B * n ** 3 * 8), "flops": flops}
    # back through every layer: the input gradient and the parameter gradient
    return {"bytes": 4 * (2 * params + B * n ** 3 * 8), "flops": 3 * flops}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _tr(x):
    return x[0] + x[1] + x[2]


def _isotropic(lam, mu, x):
    """lam tr(x) I + 2 mu x; lam, mu numbers or fields."""
    y = 2 * mu * x
    y[:3] += lam * _tr(x)
    return y


class _Green:
    """Gamma0 of the reference medium on a grid with unit cell lengths; mixed
    frequencies with a Nyquist component, and the zero frequency, give zero."""

    def __init__(self, shape, lam0, mu0):
        nz, ny, nx = shape
        self.shape = shape
        k = [torch.fft.fftfreq(nz, 1 / nz, dtype=torch.float64, device="cuda").view(-1, 1, 1),
             torch.fft.fftfreq(ny, 1 / ny, dtype=torch.float64, device="cuda").view(1, -1, 1),
             torch.fft.rfftfreq(nx, 1 / nx, dtype=torch.float64, device="cuda").view(1, 1, -1)]
        nyq = [(n % 2 == 0 and n > 1) & (2 * torch.abs(q) == n) for n, q in zip(shape, k)]
        count = sum((q != 0).to(torch.int32) for q in k)
        zero = (count == 0) | ((count >= 2) & (nyq[0] | nyq[1] | nyq[2]))
        norm = torch.sqrt(k[0] ** 2 + k[1] ** 2 + k[2] ** 2)
        norm = torch.where(norm == 0, torch.ones_like(norm), norm)
        self.n = [torch.where(zero, torch.zeros_like(norm), q / norm) for q in (k[2], k[1], k[0])]
        self.a, self.mu0 = (lam0 + mu0) / (lam0 + 2 * mu0), mu0

    def __call__(self, tau):
        t = torch.fft.rfftn(tau, dim=(1, 2, 3))
        n1, n2, n3 = self.n
        v = [t[0] * n1 + t[5] * n2 + t[4] * n3, t[5] * n1 + t[1] * n2 + t[3] * n3,
             t[4] * n1 + t[3] * n2 + t[2] * n3]
        s = self.a * (n1 * v[0] + n2 * v[1] + n3 * v[2])
        w = [(x - n * s) / self.mu0 for x, n in zip(v, self.n)]
        t[0], t[1], t[2] = n1 * w[0], n2 * w[1], n3 * w[2]
        t[3] = 0.5 * (n2 * w[2] + n3 * w[1])
        t[4] = 0.5 * (n1 * w[2] + n3 * w[0])
        t[5] = 0.5 * (n1 * w[1] + n2 * w[0])
        return torch.fft.irfftn(t, s=self.shape, dim=(1, 2, 3))


def _moduli(cell):
    phase = torch.as_tensor(cell.phase, device="cuda").long()
    return (torch.tensor(cell.lam, dtype=torch.float64, device="cuda")[phase],
            torch.tensor(cell.mu, dtype=torch.float64, device="cuda")[phase])


def _solution(cell, E):
    """Strain of the cell problem: conjugate gradients for Gamma0 C (E + e) = 0
    over the compatible fields e, in the energy of C0."""
    lam, mu = _moduli(cell)
    green = _Green(tuple(cell.phase.shape), cell.lam0, cell.mu0)
    weight = torch.tensor([1.0, 1, 1, 2, 2, 2], dtype=torch.float64, device="cuda").view(6, 1, 1, 1)

    def dot(x, y):
        return torch.sum(weight * x * y)

    eps = torch.tensor(np.asarray(E), dtype=torch.float64, device="cuda").view(6, 1, 1, 1)
    eps = eps.expand((6,) + tuple(cell.phase.shape)).clone()
    res = -green(_isotropic(lam, mu, eps))
    d = res.clone()
    rr = dot(res, _isotropic(cell.lam0, cell.mu0, res))
    stop = 1e-24 * float(rr)
    for _ in range(400):
        Cd = _isotropic(lam, mu, d)
        alpha = rr / dot(d, Cd)
        eps += alpha * d
        res -= alpha * green(Cd)
        new = dot(res, _isotropic(cell.lam0, cell.mu0, res))
        d = res + (new / rr) * d
        rr = new
        if float(rr) <= stop:
            break
    return eps, _isotropic(lam, mu, eps)


def _network(case, p, feat, E):
    """out [B][6][n][n][n] of the network for the parameter vector p."""
    n, m, W = case["n"], case["modes"], fno.WIDTH
    P, b = p[:2 * W].view(W, 2), p[2 * W:3 * W]
    Q, q = p[3 * W:3 * W + fno.COUT * W].view(fno.COUT, W), p[3 * W + fno.COUT * W:][:fno.COUT]
    per = (p.numel() - fno.HEADER) // case["layers"]
    keep = torch.tensor(list(range(m)) + list(range(n - m, n)), device="cuda")
    v = torch.einsum("oc,bcxyz->boxyz", P, feat) + b.view(1, W, 1, 1, 1)
    for l in range(case["layers"]):
        at = fno.HEADER + l * per
        A, a = p[at:at + W * W].view(W, W), p[at + W * W:at + W * W + W]
        R = torch.view_as_complex(p[at + W * W + W:at + per].view(2 * m, m, 2 * m, W, W, 2))
        F = torch.fft.rfftn(v, dim=(2, 3, 4))[..., :m].index_select(2, keep).index_select(3, keep)
        F = torch.einsum("bizyx,yxzio->bozyx", F, R)
        full = torch.zeros((v.shape[0], W, n, n, n // 2 + 1), dtype=F.dtype, device="cuda")
        row = torch.zeros((v.shape[0], W, 2 * m, n, m), dtype=F.dtype, device="cuda")
        row = row.index_copy(3, keep, F)
        col = torch.zeros((v.shape[0], W, n, n, m), dtype=F.dtype, device="cuda")
        col = col.index_copy(2, keep, row)
        full = torch.cat((col, full[..., m:]), dim=-1)
        u = torch.fft.irfftn(full, s=(n, n, n), dim=(2, 3, 4))
        v = torch.einsum("oc,bcxyz->boxyz", A, v) + a.view(1, W, 1, 1, 1) + u
        if l < case["layers"] - 1:
            v = torch.nn.functional.gelu(v, approximate="tanh")
    H = torch.einsum("oc,bcxyz->boxyz", Q, v) + q.view(1, -1, 1, 1, 1)
    return torch.einsum("bojxyz,bj->boxyz", H.view(v.shape[0], 6, 6, n, n, n), E)


def exact(case, seed):
    kind = case["kind"]
    if kind == "gamma":
        cell, E, field = _inputs(case, seed)
        x = field.double()
        if case["mode"] != "raw":
            lam, mu = _moduli(cell)
            x = _isotropic(lam - cell.lam0, mu - cell.mu0, x)
        y = -_Green(tuple(cell.phase.shape), cell.lam0, cell.mu0)(x)
        if case["mode"] == "full":
            y += torch.tensor(E, device="cuda").view(6, 1, 1, 1)
        return y
    if kind == "solve":
        cell, E = _inputs(case, seed)
        eps, sig = _solution(cell, E)
        return {"eps": eps, "sig": sig}
    if kind == "batch":
        cells = _inputs(case, seed)
        C = np.empty((len(cells), 6, 6))
        for i, cell in enumerate(cells):
            for j in range(6):
                E = np.zeros(6)
                E[j] = 1.0 if j < 3 else 0.5
                C[i, :, j] = _solution(cell, E)[1].mean(dim=(1, 2, 3)).cpu().numpy()
        return C
    feat, E, target, p = _inputs(case, seed)
    E = torch.tensor(E, dtype=torch.float64, device="cuda")
    p = p.double()
    if not case["grad"]:
        return _network(case, p, feat.double(), E)
    p.requires_grad_(True)
    total, count = 0.0, target.numel()
    for b in range(case["batch"]):   # one sample at a time: the loss is a sum over them
        out = _network(case, p, feat[b:b + 1].double(), E[b:b + 1])
        part = torch.sum((out - target[b:b + 1].double()) ** 2) / count
        part.backward()
        total += float(part.detach())
    return {"loss": total, "grads": p.grad}
