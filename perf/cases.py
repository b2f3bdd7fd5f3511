"""Cases by which the speed of the projection library is measured.

A case is one step that a flow solver asks of the library: a pressure
projection, an implicit viscous step, a gradient through a projection, and so
on, on fields of the kinds and sizes of this repository's configurations,
tests and benchmark.  All of them go through the Python entry points
(Context, Batch, projection).  ``prepare`` makes what a flow solver holds
before the call: the fields on the GPU and a context for its grid; ``run`` is
one call, on copies of the predicted velocity (the step updates it in place)
and from zero pressure; ``exact`` solves the same discrete equations in plain
FP64 torch, without the library.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2012_11744_gb300 as paris

PERIODIC, WALL = 0, 1
F64 = torch.float64


def _case(name, kind, n, bc, **more):
    return {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2],
            "bcx": bc[0], "bcy": bc[1], "bcz": bc[2], **more}


def listed():
    P, W = PERIODIC, WALL
    return [
        # the smallest grid in use: one drop in a 32^3 periodic box, where launches and latency count
        _case("step_drop32", "step", (32, 32, 32), (P, P, P), field="random", drops=1, ratio=10.0, fp64=False),
        # a box whose axes are not powers of two, walls all round (odd counts, no regular halving)
        _case("step_ragged", "step", (150, 100, 75), (W, W, W), field="drops", drops=12, ratio=1000.0, fp64=False),
        # the headline step: 64 drops at density ratio 1000, walls in z
        _case("step_drops256", "step", (256, 256, 256), (P, P, W), field="drops", drops=64, ratio=1000.0, fp64=False),
        # the largest step: a jet along x between walls in y and z
        _case("step_jet512", "step", (512, 256, 256), (P, W, W), field="jet", drops=0, ratio=1000.0, fp64=False),
        # the FP64 form, for callers that ask for double precision throughout
        _case("step_fp64", "step", (128, 128, 128), (P, P, W), field="drops", drops=24, ratio=1000.0, fp64=True),
        # the step with surface tension and gravity in its predictor
        _case("step_forced", "forced", (192, 192, 192), (P, P, W), field="drops", drops=32, ratio=1000.0),
        # forward and backward through the differentiable projection (an inverse problem)
        _case("adjoint128", "adjoint", (128, 128, 128), (P, P, P), field="random", drops=1, ratio=100.0),
        # many uneven boxes in one call (a parameter study, a training set)
        {"name": "batch64", "kind": "batch", "count": 64, "ratio": 1000.0},
        # the implicit viscous step of the three components, multigrid and plain conjugate gradients
        _case("viscous_mg", "viscous", (256, 256, 256), (P, P, W), drops=64, multigrid=True),
        _case("viscous_cg", "viscous", (128, 128, 128), (P, W, W), drops=24, multigrid=False),
        # bubbles as free surfaces: the liquid's projection, then the phantom projection in the gas
        _case("free_surface", "surface", (128, 128, 128), (P, P, W), drops=24),
        # the steps around a caller's own pressure solve: coefficients, divergence, correction
        _case("fields", "fields", (256, 256, 256), (P, P, W), drops=64, ratio=1000.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def even(lo, hi, by):  # sizes as users choose them: multiples that can be halved a few times
        return max(lo, by * round(size(lo, hi) / by))

    kind = rng.choice(["step", "step", "ragged", "ragged", "fp64", "forced", "adjoint", "batch", "viscous_mg",
                       "viscous_cg", "surface", "fields"])
    bc = tuple(rng.choice((PERIODIC, WALL)) for _ in range(3))
    ratio = round(math.exp(rng.uniform(0.0, math.log(1000.0))), 3)
    drops = rng.randint(1, 40)
    if kind == "batch":
        return {"kind": "batch", "count": size(4, 64), "ratio": max(ratio, 2.0)}
    if kind == "ragged":
        n = tuple(size(24, 128) for _ in range(3))
        return _unnamed("step", n, bc, field=rng.choice(("drops", "random")), drops=drops, ratio=ratio,
                        fp64=rng.random() < 0.25)
    if kind in ("step", "fp64"):
        hi = 320 if kind == "step" else 144
        n = tuple(even(32, hi, rng.choice((4, 8, 16))) for _ in range(3))
        field = rng.choice(("drops", "random", "jet"))
        if field == "jet":
            bc = (PERIODIC, WALL, WALL)
        return _unnamed("step", n, bc, field=field, drops=drops, ratio=ratio, fp64=kind == "fp64")
    if kind == "forced":
        return _unnamed("forced", tuple(even(32, 224, 4) for _ in range(3)), bc, field="drops", drops=drops,
                        ratio=ratio)
    if kind == "adjoint":
        return _unnamed("adjoint", tuple(even(32, 160, 4) for _ in range(3)), bc, field="random", drops=drops,
                        ratio=ratio)
    if kind in ("viscous_mg", "viscous_cg"):
        n = tuple(size(32, 256 if kind == "viscous_mg" else 144) for _ in range(3))
        return _unnamed("viscous", n, bc, drops=drops, multigrid=kind == "viscous_mg")
    if kind == "surface":
        return _unnamed("surface", tuple(even(32, 160, 4) for _ in range(3)), bc, drops=drops)
    return _unnamed("fields", tuple(size(48, 320) for _ in range(3)), bc, drops=drops, ratio=ratio)


def _unnamed(kind, n, bc, **more):
    c = _case("", kind, n, bc, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs ---

RHO2, DT, SIGMA, GRAVITY = 1.0, 1e-4, 0.07, (0.0, 0.0, -9.81)
MU1, MU2 = 1e-3, 1.8e-5          # water- and air-like viscosities
RHO_L = 1000.0                   # the liquid of the free-surface steps
BATCH_AXES = (32, 48, 64, 96, 128)


def _grid(case):
    return paris.Grid(case["nx"], case["ny"], case["nz"], 1.0 / max(case["nx"], case["ny"], case["nz"]),
                      (case["bcx"], case["bcy"], case["bcz"]))


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(gen, shape, lo=-1.0, hi=1.0):
    return torch.rand(shape, generator=gen, device="cuda", dtype=F64) * (hi - lo) + lo


def _spheres(rng, grid, count, rmin, rmax):
    """Non-overlapping spheres (as many as fit in 4000 tries), clear of the walls by two cells."""
    n = (grid.nx, grid.ny, grid.nz)
    L = [m * grid.h for m in n]
    gap, out = 2.0 * grid.h, []
    rmax = min(rmax, 0.5 * min(L) - gap - 0.5 * grid.h)
    rmin = min(rmin, rmax)
    for _ in range(4000):
        if len(out) >= count:
            break
        r = rng.uniform(rmin, rmax)
        c = [rng.uniform(r + gap, L[a] - r - gap) if grid.bc[a] == WALL else rng.uniform(0.0, L[a]) for a in range(3)]
        for c2, r2 in out:
            d2 = 0.0
            for a in range(3):
                d = c[a] - c2[a]
                if grid.bc[a] == PERIODIC:
                    d -= L[a] * round(d / L[a])
                d2 += d * d
            if d2 < (r + r2 + gap) ** 2:
                break
        else:
            out.append((c, r))
    return out


def _fraction(grid, spheres):
    """The spheres' volume fraction on 4 x 4 x 4 sub-cells per cell."""
    n, h = (grid.nx, grid.ny, grid.nz), grid.h
    C = torch.zeros(grid.shape, device="cuda", dtype=F64)
    sub = (torch.arange(4, device="cuda", dtype=F64) + 0.5) / 4
    for c, r in spheres:
        d2, ix = [], []
        for a in range(3):
            lo, hi = math.floor((c[a] - r) / h) - 1, math.floor((c[a] + r) / h) + 2
            if grid.bc[a] == WALL:
                lo, hi = max(lo, 0), min(hi, n[a])
            i = torch.arange(lo, hi, device="cuda")
            d2.append(((i[:, None].double() + sub) * h - c[a]) ** 2)
            ix.append(i % n[a])
        s = (d2[0][None, None, None, None] + d2[1][None, None, :, :, None, None]) + d2[2][:, :, None, None, None, None]
        C[ix[2][:, None, None], ix[1][None, :, None], ix[0]] += (s < r * r).sum((1, 3, 5)).double() / 64
    return C.clamp_(0.0, 1.0)


def _jet(rng, grid):
    """A jet along x whose radius is modulated by four sines."""
    n, h = (grid.nx, grid.ny, grid.nz), grid.h
    m, ph = [rng.randint(2, 16) for _ in range(4)], [rng.uniform(0.0, 2 * math.pi) for _ in range(4)]
    sub = (torch.arange(4, device="cuda", dtype=F64) + 0.5) / 4
    x, y, z = ((torch.arange(k, device="cuda", dtype=F64)[:, None] + sub) * h for k in n)
    Lx, rad = n[0] * h, 0.16 * min(n[1], n[2]) * h
    R = rad * (1.0 + 0.05 * sum(torch.sin(2 * math.pi * k * x / Lx + p) for k, p in zip(m, ph)))
    d2 = ((y - 0.5 * n[1] * h) ** 2)[None, None] + ((z - 0.5 * n[2] * h) ** 2)[:, :, None, None]
    C = torch.zeros(grid.shape, device="cuda", dtype=F64)
    for i in range(4):
        for j in range(4):
            for k in range(4):
                C += d2[:, k, :, j, None] < R[:, i] ** 2
    return C / 64


def _zero_walls(grid, vel):
    for a in range(3):
        if grid.bc[a] == WALL:
            vel[a].select(2 - a, 0).zero_()
            vel[a].select(2 - a, vel[a].shape[2 - a] - 1).zero_()
    return vel


def _waves(rng, gen, grid, noise=0.01):
    """16 random Fourier modes of unit amplitude plus noise, zero on the walls."""
    n = (grid.nx, grid.ny, grid.nz)
    modes = []
    for _ in range(16):
        k = [0, 0, 0]
        while not any(k):
            k = [rng.randint(-4, 4) for _ in range(3)]
        e = [rng.gauss(0, 1) for _ in range(3)]
        s = math.sqrt(sum(v * v for v in e))
        modes.append((k, [v / s for v in e], rng.uniform(0.0, 2 * math.pi)))
    vel = []
    for a in range(3):
        ph = []
        for b in range(3):
            m = grid.face_shape(a)[2 - b]
            x = (torch.arange(m, device="cuda", dtype=F64) + (0.0 if a == b else 0.5)) / n[b]
            ph.append(torch.stack([2 * math.pi * k[b] * x + (p if b == 2 else 0.0) for k, _, p in modes]))
        e = torch.tensor([d[a] for _, d, _ in modes], device="cuda", dtype=F64)
        yz = ph[2][:, :, None] + ph[1][:, None, :]
        left = torch.cat([e[:, None, None] * torch.cos(yz), -e[:, None, None] * torch.sin(yz)]).flatten(1)
        right = torch.cat([torch.cos(ph[0]), torch.sin(ph[0])])
        f = (left.t() @ right).view(grid.face_shape(a))
        vel.append(f + _uniform(gen, f.shape, -noise, noise))
    return _zero_walls(grid, vel)


def _noise(gen, grid):
    return _zero_walls(grid, [_uniform(gen, grid.face_shape(a)) for a in range(3)])


def _flow(case, grid, seed):
    """Volume fraction, spheres and predicted velocity of a single-grid case."""
    rng, gen = random.Random(seed), _generator(seed)
    field = case.get("field", "drops")
    if field == "jet":
        C, spheres = _jet(rng, grid), []
        u = 0.5 * (C + torch.roll(C, 1, 2))
        vel = [torch.zeros(grid.face_shape(a), device="cuda", dtype=F64) for a in range(3)]
        vel[0] += u
        vel = _zero_walls(grid, [f + _uniform(gen, f.shape, -0.1, 0.1) for f in vel])
        return C, spheres, vel
    L = min(grid.nx, grid.ny, grid.nz) * grid.h
    few = case["drops"] <= 4
    rmin, rmax = (0.1 if few else 0.02) * L, (0.25 if few else 0.08) * L
    if case["kind"] == "surface":  # bubbles that reach beyond the two gas layers of the phantom projection
        rmin, rmax = max(rmin, 5.0 * grid.h), max(rmax, 6.0 * grid.h)
    spheres = _spheres(rng, grid, case["drops"], rmin, rmax)
    C = _fraction(grid, spheres)
    return C, spheres, _noise(gen, grid) if field == "random" else _waves(rng, gen, grid)


def _curvature(grid, spheres):
    """-2/r of the sphere whose surface is nearest."""
    n = (grid.nx, grid.ny, grid.nz)
    best = torch.full(grid.shape, math.inf, device="cuda", dtype=F64)
    kappa = torch.zeros(grid.shape, device="cuda", dtype=F64)
    for c, r in spheres:
        d2 = []
        for a in range(3):
            d = (torch.arange(n[a], device="cuda", dtype=F64) + 0.5) * grid.h - c[a]
            if grid.bc[a] == PERIODIC:
                d = d - n[a] * grid.h * torch.round(d / (n[a] * grid.h))
            d2.append(d * d)
        dist = (torch.sqrt(d2[2][:, None, None] + d2[1][:, None] + d2[0]) - r).abs()
        kappa = torch.where(dist < best, torch.full_like(kappa, -2.0 / r), kappa)
        best = torch.minimum(best, dist)
    return kappa


def _batch_problems(case, seed):
    rng, gen = random.Random(seed), _generator(seed)
    # the sizes belong to the case, the fields to the seed
    shapes = random.Random(case["count"])
    out = []
    for _ in range(case["count"]):
        n = [shapes.choice(BATCH_AXES) for _ in range(3)]
        g = paris.Grid(*n, 1.0 / 64)
        L = min(n) / 64
        C = _fraction(g, _spheres(rng, g, rng.randint(1, 8), 0.05 * L, 0.2 * L))
        rho1 = math.exp(rng.uniform(0.0, math.log(case["ratio"])))
        out.append((g, C, rho1, _noise(gen, g)))
    return out


def _inputs(case, seed):
    """Everything of a case but the context: the same for prepare and exact."""
    kind = case["kind"]
    if kind == "batch":
        return {"problems": _batch_problems(case, seed)}
    grid = _grid(case)
    C, spheres, vel = _flow(case, grid, seed)
    d = {"grid": grid, "C": C, "vel": vel}
    gen = _generator(seed + 1)
    if kind == "forced":
        d["kappa"] = _curvature(grid, spheres)
    if kind == "adjoint":  # an interface a few cells wide, and the gradient of a loss on the velocity
        d["C"] = sum(torch.roll(C, s, a) for a in range(3) for s in (-1, 1)) / 8 + C / 4
        d["grad"] = _noise(gen, grid)
    if kind == "viscous":  # four times the cell size squared over the largest viscosity
        d["tau"] = 4 * grid.h ** 2 / max(MU1 / 1000.0, MU2)
    if kind == "surface":
        d["theta"] = [_uniform(gen, grid.face_shape(a), 0.1, 1.0) for a in range(3)]
        d["kappa"] = _curvature(grid, spheres)
        d["p_gas"] = 1.0 + 0.1 * _uniform(gen, grid.shape)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    d["case"] = case
    if case["kind"] == "batch":
        pb = d.pop("problems")
        b = paris.Batch([q[0] for q in pb])
        d.update(batch=b, C=b.pack([q[1] for q in pb], "C"), rho1=[q[2] for q in pb],
                 vel=[b.pack([q[3][a] for q in pb], "uvw"[a]) for a in range(3)])
        d["work"] = [torch.empty_like(x) for x in d["vel"]] + [torch.empty_like(d["C"])]
        return d
    fp64 = bool(case.get("fp64", False))
    d["ctx"] = paris.Context(d["grid"], opts=paris.default_opts(precision=paris.FP64 if fp64 else paris.MIXED))
    if case["kind"] == "adjoint":
        d["C"].requires_grad_(True)
        for x in d["vel"]:
            x.requires_grad_(True)
        return d
    d["work"] = [torch.empty_like(x) for x in d["vel"]]
    d["cells"] = [torch.empty_like(d["C"]) for _ in range(2)]
    d["faces"] = [torch.empty_like(x) for x in d["vel"]]
    return d


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "adjoint":
        C, us = state["C"], state["vel"]
        u, v, w, p = paris.projection(C, *us, state["ctx"], case["ratio"], RHO2, DT)
        gC, gu, gv, gw = torch.autograd.grad((u, v, w), (C, *us), state["grad"])
        return {"u": u, "v": v, "w": w, "p": p, "gC": gC, "gu": gu, "gv": gv, "gw": gw}
    if kind == "viscous":
        ctx, out = state["ctx"], {}
        for a in range(3):
            nu = ctx.face_viscosity(a, state["C"], MU1, MU2, 1000.0, RHO2, out=state["faces"][a])
            ctx.viscous_solve(a, nu, state["tau"], state["vel"][a], us=state["work"][a], tol=1e-10,
                              multigrid=case["multigrid"])
            out["uvw"[a]] = state["work"][a]
        return out
    for x, y in zip(state["work"], state["vel"]):
        x.copy_(y)
    if kind == "batch":
        u, v, w, p = state["work"]
        n = case["count"]
        state["batch"].projection_step(state["C"], state["rho1"], [RHO2] * n, [1e-3] * n, u, v, w, p)
        return {"u": u, "v": v, "w": w, "p": p}
    ctx, C, (u, v, w) = state["ctx"], state["C"], state["work"]
    p, q = state["cells"]
    if kind == "fields":
        beta = ctx.face_coeffs(C, case["ratio"], RHO2, out=state["faces"])
        rhs, _ = ctx.divergence(u, v, w, DT, out=p, want_mean=False)
        ctx.project(*beta, C, DT, u, v, w)  # the fraction stands in for the caller's pressure
        return {"bx": beta[0], "by": beta[1], "bz": beta[2], "rhs": rhs, "u": u, "v": v, "w": w}
    p.zero_()
    if kind == "step":
        ctx.projection_step(C, case["ratio"], RHO2, DT, u, v, w, p)
    elif kind == "forced":
        ctx.projection_step_forced(C, state["kappa"], case["ratio"], RHO2, SIGMA, GRAVITY, DT, u, v, w, p)
    elif kind == "surface":
        ctx.free_surface_step(C, RHO_L, DT, u, v, w, p, p_gas=state["p_gas"], theta=state["theta"],
                              kappa=state["kappa"], sigma=SIGMA)
        q.zero_()
        ctx.phantom_projection(C, u, v, w, q)
        return {"u": u, "v": v, "w": w, "p": p, "phat": q}
    return {"u": u, "v": v, "w": w, "p": p}


def work(case):
    """Each input read once and each output written once; about 30 operations a cell and array set."""
    if case["kind"] == "batch":
        shapes = random.Random(case["count"])
        n = sum(math.prod(shapes.choice(BATCH_AXES) for _ in range(3)) for _ in range(case["count"]))
        return {"bytes": 8 * 8 * n, "flops": 30 * n}
    n = case["nx"] * case["ny"] * case["nz"]
    # doubles a cell: C, u*, p and the outputs; forcing reads kappa; the adjoint has a second set and dL/dC
    arrays = {"step": 8, "forced": 9, "adjoint": 15, "viscous": 7, "surface": 15, "fields": 11}[case["kind"]]
    return {"bytes": 8 * arrays * n, "flops": 30 * n}


# ------------------------------------------------- the same in plain torch ---

def _beta(grid, C, rho1):
    """2/(rho_L + rho_R) on the faces, 0 on wall faces."""
    rho = rho1 * C + RHO2 * (1.0 - C)
    out = []
    for a in range(3):
        out.append(_between(grid, a, rho, lambda lo, hi: 2.0 / (lo + hi)))
    return out


def _between(grid, a, x, fn):
    """fn(lower cell, upper cell) on the faces of axis a, 0 on wall faces."""
    d = 2 - a
    if grid.bc[a] == PERIODIC:
        return fn(torch.roll(x, 1, d), x)
    n = x.shape[d]
    f = torch.zeros(grid.face_shape(a), device=x.device, dtype=x.dtype)
    f.narrow(d, 1, n - 1).copy_(fn(x.narrow(d, 0, n - 1), x.narrow(d, 1, n - 1)))
    return f


def _closed(grid, a, f):
    """A face array with both ends of its axis: n + 1 entries, wall faces 0."""
    d = 2 - a
    if grid.bc[a] == PERIODIC:
        return torch.cat([f, f.narrow(d, 0, 1)], d)
    f = f.clone()
    f.select(d, 0).zero_()
    f.select(d, f.shape[d] - 1).zero_()
    return f


def _divergence(grid, vel):
    return sum(torch.diff(_closed(grid, a, vel[a]), dim=2 - a) for a in range(3)) / grid.h


def _gradient(grid, p):
    return [_between(grid, a, p, lambda lo, hi: hi - lo) / grid.h for a in range(3)]


class _Level:
    """A x = sum over a cell's faces of b (x - x_neighbour) + sig x, faces closed (n + 1 entries along their axis)."""

    def __init__(self, b, sig, width):
        self.b, self.sig, self.width = b, sig, width
        d = sig.clone()
        for a in range(3):
            n = sig.shape[2 - a]
            d += b[a].narrow(2 - a, 0, n) + b[a].narrow(2 - a, 1, n)
        self.inv = torch.where(d > 0, 1.0 / d, torch.zeros_like(d))

    def apply(self, x):
        y = self.sig * x
        for a in range(3):
            d, n = 2 - a, x.shape[2 - a]
            g = torch.diff(torch.cat([x.narrow(d, n - 1, 1), x, x.narrow(d, 0, 1)], d), dim=d) * self.b[a]
            y -= torch.diff(g, dim=d)
        return y

    def smooth(self, f, x, times=4, lo=0.25, hi=2.0):
        """Chebyshev steps on the diagonally scaled operator, its spectrum's part [lo, hi]."""
        mid, half = 0.5 * (hi + lo), 0.5 * (hi - lo)
        r = f if x is None else f - self.apply(x)
        d = self.inv * r / mid
        x = d if x is None else x + d
        s = half / mid
        rho = s
        for _ in range(times - 1):
            r = r - self.apply(d)
            new = 1.0 / (2.0 / s - rho)
            d = new * rho * d + (2.0 * new / half) * (self.inv * r)
            rho = new
            x = x + d
        return x


def _pairs(n):
    """Starts of the aggregates of n cells: pairs, the last one of three where n is odd."""
    return list(range(0, n - n % 2, 2)) if n >= 4 else list(range(n))


class _Solver:
    """Conjugate gradients in FP64 on the system of _Level, with a multigrid cycle over cell aggregates."""

    def __init__(self, b, sig):
        shape = sig.shape
        self.levels = [_Level(b, sig, [torch.ones(shape[2 - a], device=sig.device, dtype=F64) for a in range(3)])]
        while max(self.levels[-1].sig.shape) >= 4:
            self.levels.append(self._coarser(self.levels[-1]))
        c = self.levels[-1]
        m = c.sig.numel()
        dense = torch.stack([c.apply(e.view(c.sig.shape)).flatten() for e in torch.eye(m, device=sig.device, dtype=F64)])
        self.coarse = torch.linalg.pinv(dense, hermitian=True, rtol=1e-12)

    @staticmethod
    def _sum(x, d):
        """Sums over the aggregates along dimension d."""
        n = x.shape[d]
        starts = _pairs(n)
        if len(starts) == n:
            return x
        y = x.narrow(d, 0, 2 * len(starts)).unflatten(d, (len(starts), 2)).sum(d + 1)
        if n % 2:
            y.select(d, len(starts) - 1).add_(x.select(d, n - 1))
        return y

    def _coarser(self, L):
        sig, b, width = L.sig, [], []
        for a in range(3):
            sig = self._sum(sig, 2 - a)
            width.append(self._sum(L.width[a], 0))
        for a in range(3):
            d = 2 - a
            at = torch.tensor(_pairs(L.sig.shape[d]) + [L.sig.shape[d]], device=sig.device)
            w, wc = L.width[a], width[a]
            dist = 0.5 * (torch.cat([w[-1:], w]) + torch.cat([w, w[:1]]))[at]
            dist = dist / (0.5 * (torch.cat([wc[-1:], wc]) + torch.cat([wc, wc[:1]])))
            f = L.b[a].index_select(d, at) * dist.view([-1 if k == d else 1 for k in range(3)])
            for e in range(3):
                if e != d:
                    f = self._sum(f, e)
            b.append(f)
        return _Level(b, sig, width)

    def _cycle(self, f, k=0):
        L = self.levels[k]
        if k == len(self.levels) - 1:
            return (self.coarse @ f.flatten()).view(f.shape)
        x = L.smooth(f, None)
        r = f - L.apply(x)
        for d in range(3):
            r = self._sum(r, d)
        e = self._cycle(r, k + 1)
        for d in range(3):
            n = x.shape[d]
            if e.shape[d] != n:
                e = torch.repeat_interleave(e, 2, d)
                if n % 2:
                    e = torch.cat([e, e.narrow(d, e.shape[d] - 1, 1)], d)
        return L.smooth(f, x + e)

    def solve(self, f, gauge):
        """gauge: mean-free right-hand side and solution (no Dirichlet cell)."""
        if gauge:
            f = f - f.mean()
        x, b2 = torch.zeros_like(f), float((f * f).sum())
        best = math.inf
        for _ in range(8):  # restarts from the true residual
            r = f - self.levels[0].apply(x)
            if gauge:
                r = r - r.mean()
            rr = float((r * r).sum())
            if rr <= 1e-30 * b2 or rr > 0.25 * best:
                break
            best, goal, rho, d = rr, max(1e-16 * rr, 1e-30 * b2), None, None
            for _ in range(150):
                z = self._cycle(r)
                new = (r * z).sum()
                d = z if d is None else z + (new / rho) * d
                rho = new
                q = self.levels[0].apply(d)
                alpha = rho / (d * q).sum()
                x += alpha * d
                r = r - alpha * q
                if float((r * r).sum()) <= goal:
                    break
        return x - x.mean() if gauge else x


def _poisson(grid, beta, rhs):
    """p of div (beta grad p) = rhs, both mean-free."""
    b = [_closed(grid, a, beta[a]) for a in range(3)]
    return _Solver(b, torch.zeros_like(rhs)).solve(-rhs * grid.h ** 2, True)


def _project(grid, beta, vel, dt):
    p = _poisson(grid, beta, _divergence(grid, vel) / dt)
    g = _gradient(grid, p)
    return p, _zero_walls(grid, [x - dt * b * y for x, b, y in zip(vel, beta, g)])


def _named(vel, p):
    return {"u": vel[0], "v": vel[1], "w": vel[2], "p": p}


def _exact_adjoint(case, d):
    grid, C = d["grid"], d["C"]
    beta = _beta(grid, C, case["ratio"])
    p, vel = _project(grid, beta, d["vel"], DT)
    g = d["grad"]
    q = _poisson(grid, beta, _divergence(grid, [b * x for b, x in zip(beta, g)]))
    gp, gq = _gradient(grid, p), _gradient(grid, q)
    gus = _zero_walls(grid, [x - y for x, y in zip(g, gq)])
    gb = [DT * x * (y - z) * b * b for x, y, z, b in zip(gp, gq, g, beta)]
    gC = torch.zeros_like(C)
    for a in range(3):
        f, n = _closed(grid, a, gb[a]), C.shape[2 - a]
        gC += f.narrow(2 - a, 0, n) + f.narrow(2 - a, 1, n)
    gC *= -0.5 * (case["ratio"] - RHO2)
    return {**_named(vel, p), "gC": gC, "gu": gus[0], "gv": gus[1], "gw": gus[2]}


def _exact_viscous(case, d):
    grid, C, out = d["grid"], d["C"], {}
    mu, rho = MU1 * C + MU2 * (1.0 - C), 1000.0 * C + RHO2 * (1.0 - C)
    for a in range(3):
        nu = _between(grid, a, mu, torch.add) / _between(grid, a, rho, torch.add)
        un, own = d["vel"][a], grid.bc[a] == WALL
        if own:  # the unknowns: the faces between the component's wall faces
            nu, un = (x.narrow(2 - a, 1, x.shape[2 - a] - 2) for x in (nu, un))
        mass = grid.h ** 2 / (d["tau"] * nu)
        sig, b = mass.clone(), []
        for e in range(3):
            k, n = 2 - e, un.shape[2 - e]
            f = torch.ones([m + (i == k) for i, m in enumerate(un.shape)], device=C.device, dtype=F64)
            if grid.bc[e] == WALL:  # beyond the ends: 0 (the wall face) or minus the end value
                f.select(k, 0).zero_()
                f.select(k, n).zero_()
                sig.select(k, 0).add_(1.0 if e == a else 2.0)
                sig.select(k, n - 1).add_(1.0 if e == a else 2.0)
            b.append(f)
        x = _Solver(b, sig).solve(mass * un, False)
        full = torch.zeros(grid.face_shape(a), device=C.device, dtype=F64)
        (full.narrow(2 - a, 1, x.shape[2 - a]) if own else full).copy_(x)
        out["uvw"[a]] = full
    return out


def _pair(grid, a, x, y):
    """x of the lower cell times y of the upper one, on the faces of axis a (0 on wall faces)."""
    d, n = 2 - a, x.shape[2 - a]
    if grid.bc[a] == PERIODIC:
        return torch.roll(x, 1, d) * y
    f = torch.zeros(grid.face_shape(a), device=x.device, dtype=F64)
    f.narrow(d, 1, n - 1).copy_(x.narrow(d, 0, n - 1) * y.narrow(d, 1, n - 1))
    return f


def _surface_solve(grid, cls, beta, dt, vel, theta, value):
    """The projection on the cells of class 1, with Dirichlet values (one per face, theta h away) towards class 2."""
    one, two = (cls == 1).double(), (cls == 2).double()
    b, sig, rhs, links = [], torch.zeros_like(one), -_divergence(grid, vel) / dt * grid.h ** 2, []
    for a in range(3):
        d, n = 2 - a, cls.shape[2 - a]
        inner, up, down = (_pair(grid, a, x, y) for x, y in ((one, one), (one, two), (two, one)))
        links.append((inner, up, down))
        b.append(_closed(grid, a, beta * inner))
        for cut, at in ((up, 1), (down, 0)):
            s = beta * cut / theta[a]
            sig += _closed(grid, a, s).narrow(d, at, n)
            rhs += _closed(grid, a, s * value[a]).narrow(d, at, n)
    p = one * _Solver(b, sig).solve(rhs * one, False)
    out = []
    for a in range(3):
        inner, up, down = links[a]
        lo, hi = _between(grid, a, p, lambda x, y: x), _between(grid, a, p, lambda x, y: y)
        g = inner * (hi - lo) + up * (value[a] - lo) / theta[a] + down * (hi - value[a]) / theta[a]
        out.append(vel[a] - dt * beta * g / grid.h)
    return p, out


def _touching(grid, mask):
    t = torch.zeros_like(mask)
    for a in range(3):
        d, n = 2 - a, mask.shape[2 - a]
        if grid.bc[a] == PERIODIC:
            t |= torch.roll(mask, 1, d) | torch.roll(mask, -1, d)
        else:
            t.narrow(d, 1, n - 1).logical_or_(mask.narrow(d, 0, n - 1))
            t.narrow(d, 0, n - 1).logical_or_(mask.narrow(d, 1, n - 1))
    return t


def _exact_surface(case, d):
    grid, C = d["grid"], d["C"]
    liquid = C < 0.5
    cls = torch.where(liquid, 1, 2)
    liq = liquid.double()
    value = []
    for a in range(3):  # the interface pressure on the cut faces: the gas cell's, and the mean curvature's
        gas = _between(grid, a, d["p_gas"] * (1 - liq), torch.add)
        value.append(gas + SIGMA * 0.5 * _between(grid, a, d["kappa"], torch.add))
    vel = _zero_walls(grid, [x.clone() for x in d["vel"]])
    p, vel = _surface_solve(grid, cls, 1.0 / RHO_L, DT, vel, d["theta"], value)
    p = torch.where(liquid, p, d["p_gas"])
    first = _touching(grid, liquid) & ~liquid
    second = _touching(grid, first) & ~liquid & ~first
    cls = torch.where(liquid, 0, torch.where(first | second, 1, 2))
    ones = [torch.ones(grid.face_shape(a), device=C.device, dtype=F64) for a in range(3)]
    phat, vel = _surface_solve(grid, cls, 1.0, 1.0, vel, ones, [torch.zeros_like(x) for x in ones])
    return {**_named(vel, p), "phat": phat}


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    if kind == "batch":
        got = []
        for g, C, rho1, vel in d["problems"]:
            p, vel = _project(g, _beta(g, C, rho1), vel, 1e-3)
            got.append([*vel, p])
        return {k: torch.cat([x[i].flatten() for x in got]) for i, k in enumerate(("u", "v", "w", "p"))}
    grid, C, vel = d["grid"], d["C"], d["vel"]
    if kind == "adjoint":
        return _exact_adjoint(case, d)
    if kind == "viscous":
        return _exact_viscous(case, d)
    if kind == "surface":
        return _exact_surface(case, d)
    beta = _beta(grid, C, case["ratio"])
    if kind == "fields":
        rhs = _divergence(grid, vel) / DT
        u = _zero_walls(grid, [x - DT * b * y for x, b, y in zip(vel, beta, _gradient(grid, C))])
        return {"bx": beta[0], "by": beta[1], "bz": beta[2], "rhs": rhs - rhs.mean(),
                "u": u[0], "v": u[1], "w": u[2]}
    if kind == "forced":
        ks = d["kappa"]
        force = []
        for a in range(3):
            jump = _between(grid, a, C, lambda lo, hi: hi - lo) * 0.5 * _between(grid, a, ks, torch.add)
            force.append(vel[a] + DT * (GRAVITY[a] - (SIGMA / grid.h) * jump * beta[a]))
        vel = _zero_walls(grid, force)
    p, vel = _project(grid, beta, vel, DT)
    return _named(vel, p)
