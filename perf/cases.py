"""Performance cases of the PolyPIC transfers: what a user of this library has
it do, from a 16^3 APIC step to a 23-million-particle BF16 step.

Each case is a dict of plain values.  ``prepare`` makes a program's state on
the GPU from a seed (particles in the order the previous step left them, the
grids, the workspace), ``run`` makes one pass through the public entry points,
``work`` counts what a pass cannot do without and ``exact`` gives the pass's
outputs in 64 bits from plain torch.

Kinds:
  step     polypic_step: sort, P2G, grid update (optionally with the pressure
           projection, a fabric sheet coupled by drag, Eq 12's affine map), G2P
  project  polypic_grid_update with the projection on a sorted fluid
  adjoint  the three adjoints of one step, as a reverse pass calls them
  rollout  autograd.rollout forward and backward (a training step)
"""
import math

import numpy as np
import torch

from paper_2308_01060_gb300 import autograd
from paper_2308_01060_gb300 import polypic as pp

RHO = 1000.0
GRAVITY = (0.0, -9.81, 0.0)
PPC = 8  # particles per cell
DEV = "cuda"


def _case(kind, n, modes, per_m, fill, fmt="f32", spread=True, **more):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "modes": modes, "cells_per_m": per_m,
         "fill": fill, "format": fmt, "spread": spread, "affine": False, "sheet": 0,
         "project": False, "steps": 1}
    c.update(more)
    return c


def listed():
    L = []

    def add(name, *a, **k):
        L.append(dict(_case(*a, **k), name=name))

    # the smallest call: an APIC step of 7 thousand particles, all launches and latency
    add("step_apic_16", "step", (16, 16, 16), 4, 16.0, 0.5, spread=False)
    # a small full-PolyPIC step on a grid no tile size divides
    add("step_poly27_33x29x45", "step", (33, 29, 45), 27, 33.0, 0.5)
    # the flagship: the collapsed 128^3 dam break, full PolyPIC, FP32
    add("step_poly27_128", "step", (128, 128, 128), 27, 128.0, 0.25)
    # the same fluid with APIC, the transfer most programs run
    add("step_apic_128", "step", (128, 128, 128), 4, 128.0, 0.25)
    # the paper's 8-mode setting with half-precision coefficients, ragged grid
    add("step_poly8_f16_101x84x75", "step", (101, 84, 75), 8, 64.0, 0.6, fmt="f16")
    # the largest: 23 million particles, full PolyPIC, BF16 coefficients
    add("step_poly27_bf16_203x170x181", "step", (203, 170, 181), 27, 203.0, 0.5, fmt="bf16")
    # Eq 12's affine map with full PolyPIC (modes evaluated per stencil node)
    add("step_affine27_64", "step", (64, 64, 64), 27, 64.0, 0.5, affine=True)
    # liquid on fabric: a pool and a 256^2-vertex sheet coupled by drag
    add("splash_poly27_128", "step", (128, 128, 128), 27, 128.0, 0.02, sheet=256)
    # the grid update with the pressure projection, the longest part of a projected step
    add("project_128", "project", (128, 128, 128), 27, 128.0, 0.25, project=True)
    # a whole projected step of a mid-size simulation, 8 modes
    add("step_project8_72x56x64", "step", (72, 56, 64), 8, 64.0, 0.5, project=True)
    # reverse pass of one step of the differentiable transfer
    add("adjoint_poly27_64", "adjoint", (64, 64, 64), 27, 64.0, 0.5)
    # a training step: a differentiable 4-step rollout, forward and backward
    add("rollout_poly8_24", "rollout", (24, 24, 24), 8, 24.0, 0.5, spread=False, steps=4)
    return L


def draw(rng):
    def dims(lo, hi, cells):
        while True:
            n = [int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(3)]
            if n[0] * n[1] * n[2] <= cells:
                return n

    kind = rng.choice(["step", "step", "step", "step", "project", "adjoint", "rollout"])
    if kind == "step":
        n = dims(14, 150, 128 ** 3)
        modes, fmt = rng.choice([4, 8, 27]), rng.choice(["f32", "f32", "f32", "bf16", "f16"])
        what = rng.choice(["plain", "plain", "plain", "affine", "sheet", "project"])
        affine = what == "affine" and fmt == "f32" and max(n) <= 80
        sheet = rng.randrange(48, 256) if what == "sheet" and min(n) >= 24 else 0
        # 16-bit fits are compared code by code: their velocity is not solved for
        project = what == "project" and fmt == "f32"
        return _case(kind, n, modes, float(rng.choice([16, 32, 64, 128, n[0]])),
                     rng.uniform(0.1, 0.6), fmt, rng.random() < 0.7, affine=affine, sheet=sheet,
                     project=project)
    if kind == "project":
        n = dims(24, 140, 128 ** 3)
        return _case(kind, n, 27, float(rng.choice([32, 64, 128])), rng.uniform(0.1, 0.6),
                     project=True)
    if kind == "adjoint":
        n = dims(16, 80, 64 ** 3)
        return _case(kind, n, rng.choice([4, 8, 27]), float(rng.choice([16, 32, 64])),
                     rng.uniform(0.2, 0.6))
    n = dims(14, 30, 24 ** 3)
    return _case(kind, n, rng.choice([4, 8]), float(rng.choice([16, 32])), rng.uniform(0.3, 0.6),
                 "f32", False, steps=rng.randrange(2, 5))


# ------------------------------------------------------------------ geometry

def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _dx(case):
    return 1.0 / case["cells_per_m"]


def _dt(case):
    return 0.064 * _dx(case)  # about a fifteenth of a cell per step at 1 m/s


def _heights(case):
    """Cells of fluid in each column of the seeded interior (a 2-cell margin):
    a surface that slopes and undulates around the fill fraction.  (nz-4, nx-4)."""
    nx, ny, nz = _dims(case)
    i = (np.arange(nx - 4) + 0.5) / (nx - 4)
    k = (np.arange(nz - 4) + 0.5) / (nz - 4)
    h = case["fill"] * (1 + 0.5 * (0.5 - i)[None, :] + 0.2 * np.cos(5 * k)[:, None] * np.sin(7 * i)[None, :])
    return np.clip(np.round(h * (ny - 4)), 1, ny - 4).astype(np.int64)


def _count(case):
    return int(_heights(case).sum()) * PPC


def _sheet_count(case):
    m = case["sheet"]
    return m * m + 2 * (m - 1) ** 2 if m else 0


def _triples(modes):
    first = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1)]
    rest = [(a, b, c) for c in range(3) for b in range(3) for a in range(3) if 2 in (a, b, c)]
    return (first + rest)[:modes]


def work(case):
    R, f32 = case["modes"], case["format"] == "f32"
    cells = case["nx"] * case["ny"] * case["nz"]
    P, S = _count(case), _sheet_count(case)
    coeff = 12 * R if f32 else 12 * ((R + 1) // 2) + 4
    transfer = (81 * 3 * 3 * 2 if R == 27 else 3 * R * 27) * 2  # sum-factorised, P2G or G2P
    if case["kind"] == "project":  # m, mv in, v~ out, the cells' counts
        return {"bytes": 40.0 * cells, "flops": 30.0 * cells}
    # particles: x, m, c in and out, key and slot; grids: m, mv and v~ written, cell starts
    grids = (2 if S else 1) * 40.0 * cells
    one = {"bytes": (P + S) * (32.0 + 8 + 2 * coeff) + S * 8.0 + grids,
           "flops": (P + S) * 2.0 * transfer}
    if case["kind"] == "adjoint":
        # x, m, slot, c and the output adjoints in, three adjoints out; five grids in and out
        return {"bytes": P * (16 + 4 + coeff + 12 + coeff + 24 + coeff) + 60.0 * cells,
                "flops": P * 4.0 * transfer}
    if case["kind"] == "rollout":
        return {k: v * 3 * case["steps"] for k, v in one.items()}
    return one


# ------------------------------------------------------------------ particles

def _cells_of(x, n, dx):
    inv = torch.tensor(1.0 / dx, dtype=torch.float32, device=x.device)
    v = x.float() * inv
    c = torch.floor(v).long()
    return torch.stack([c[b].clamp(0, n[b] - 1) for b in range(3)])


def _slots(x, n, dx):
    """Key of every particle, the slot order and the cell starts, as documented
    for polypic_sort."""
    i, j, k = _cells_of(x, n, dx)
    tx, ty, tz = (n[0] + 7) // 8, (n[1] + 7) // 8, (n[2] + 3) // 4
    tile = ((k >> 2) * ty + (j >> 3)) * tx + (i >> 3)
    block = ((i >> 2) & 1) | (((j >> 2) & 1) << 1) | (((k >> 1) & 1) << 2)
    key = (tile << 8) | (block << 5) | (i & 3) | ((j & 3) << 2) | ((k & 1) << 4)
    count = torch.bincount(key, minlength=tx * ty * tz * 256)
    start = torch.zeros(count.numel() + 1, dtype=torch.int64, device=x.device)
    start[1:] = torch.cumsum(count, 0)
    order = torch.argsort(key, stable=True)
    ks = key[order]
    rank = torch.arange(order.numel(), device=x.device) - start[ks]
    dealt = torch.argsort(((ks >> 5) << 31) | (rank << 5) | (ks & 31))
    return key, order[dealt], start


def _field(x, seed):
    """A smooth velocity of about 1 m/s at positions x (3, N), double."""
    r = np.random.default_rng(seed)
    v = torch.zeros_like(x)
    for _ in range(3):
        q = r.integers(1, 4, size=3) * 2 * math.pi
        amp, ph = r.standard_normal(3) * 0.4, float(r.uniform(0, 2 * math.pi))
        wave = torch.sin(q[0] * x[0] + q[1] * x[1] + q[2] * x[2] + ph)
        for a in range(3):
            v[a] += float(amp[a]) * wave
    return v


def _fluid_positions(case, g):
    """Uniform in the fluid's cells: PPC in each (a scene as it is seeded), or
    the cell of each particle drawn as well (uneven cells, a flow that has moved)."""
    h = torch.as_tensor(_heights(case), device=DEV)
    top = torch.cumsum(h.reshape(-1), 0)
    cells = int(top[-1])
    P = cells * PPC
    if case["spread"]:
        cell = (torch.rand(P, generator=g, device=DEV, dtype=torch.float64) * cells).long().clamp(max=cells - 1)
    else:
        cell = torch.arange(P, device=DEV) // PPC
    col = torch.searchsorted(top, cell, right=True)
    j = cell - (top[col] - h.reshape(-1)[col])
    w = h.shape[1]
    c = torch.stack([col % w + 2, j + 2, col // w + 2])
    u = torch.rand((3, P), generator=g, device=DEV)
    # inside the cell also after rounding
    return ((c + u * 0.99998 + 1e-5) * _dx(case)).float()


def _sheet_positions(case, g):
    """A rippled sheet over the middle of the fluid: vertices, then the centroids
    of the two triangles of each quad; masses of 0.1 kg/m^2."""
    nx, ny, nz = _dims(case)
    m, dx = case["sheet"], _dx(case)
    u = torch.arange(m, device=DEV, dtype=torch.float64) / (m - 1) - 0.5
    side = [0.8 * nx * dx, 0.8 * nz * dx]
    xx = (0.5 * nx * dx + side[0] * u)[None, :].expand(m, m)
    zz = (0.5 * nz * dx + side[1] * u)[:, None].expand(m, m)
    ph = torch.rand(2, generator=g, device=DEV, dtype=torch.float64) * 6.28
    y0 = (2.0 + case["fill"] * (ny - 4)) * dx
    yy = y0 + 0.4 * dx * (torch.sin(9 * u + ph[0])[None, :] + torch.sin(7 * u + ph[1])[:, None]) + 0.5 * dx
    v = torch.stack([xx, yy.clamp(min=2.5 * dx, max=(ny - 2.5) * dx), zz])
    a, b, c, d = v[:, :-1, :-1], v[:, :-1, 1:], v[:, 1:, :-1], v[:, 1:, 1:]
    x = torch.cat([v.reshape(3, -1), ((a + b + d) / 3).reshape(3, -1), ((a + d + c) / 3).reshape(3, -1)], 1)
    tri = 0.1 * 0.5 * (side[0] / (m - 1)) * (side[1] / (m - 1))
    mass = torch.full((x.shape[1],), tri / 2, device=DEV)
    mass[: m * m] = tri
    return x.float(), mass


def _particles(case, seed, sheet=False):
    """x, mass, absorbed mass in the slot order of the step before, the generator."""
    g = torch.Generator(device=DEV).manual_seed(2 * seed + int(sheet))
    dx, n = _dx(case), _dims(case)
    if sheet:
        x, mass = _sheet_positions(case, g)
    else:
        x = _fluid_positions(case, g)
        mass = torch.full((x.shape[1],), RHO * dx ** 3 / PPC, device=DEV)
    before = x - _dt(case) * _field(x.double(), seed).float()
    order = _slots(before, n, dx)[1]
    x, mass = x[:, order].contiguous(), mass[order].contiguous()
    absorbed = mass * torch.rand(mass.shape, generator=g, device=DEV) * 0.5 if sheet else None
    return x, mass, absorbed, g


def _coefficients(case, x, seed, g, lo, hi):
    """FP32 coefficients (3, R, hi - lo) of particles lo..hi: the field, 2% of noise
    on it, higher modes of 0.1 m/s over a cell."""
    R, dx = case["modes"], _dx(case)
    c = torch.randn((3, R, hi - lo), generator=g, device=DEV) * 0.1
    deg = torch.tensor([sum(t) for t in _triples(R)], device=DEV, dtype=torch.float64)
    c *= (dx ** -deg).float()[None, :, None]
    c[:, 0] = _field(x[:, lo:hi].double(), seed).float() + 0.2 * c[:, 0]
    return c


def _fill_state(case, ctx, x, mass, absorbed, seed, g):
    P, R, dx = x.shape[1], case["modes"], _dx(case)
    s = ctx.new_particles(P, solid=absorbed is not None, device=DEV)
    s.x.copy_(x)
    s.mass.copy_(mass)
    if absorbed is not None:
        s.mass_abs.copy_(absorbed)
    deg = torch.tensor([sum(t) for t in _triples(R)], device=DEV, dtype=torch.float64)
    for lo in range(0, P, 1 << 21):
        hi = min(P, lo + (1 << 21))
        c = _coefficients(case, x, seed, g, lo, hi)
        if case["format"] == "f32":
            s.coeff[:, :, lo:hi] = c
            continue
        c *= (dx ** deg).float()[None, :, None]
        scale = c.abs().amax(dim=(0, 1))
        s.scale[lo:hi] = scale
        c = (c / scale).to(s.coeff.dtype)
        for r in range(R):
            s.coeff[:, r // 2, lo:hi, r % 2] = c[:, r]
    return s


# ------------------------------------------------------------------ prepare

def _context(case):
    return pp.Context(_dims(case), _dx(case), case["modes"], case["format"],
                      map_affine=case["affine"])


def _params(case):
    return pp.UpdateSettings(dt=_dt(case), gravity=GRAVITY, drag_k=5.0 * _dx(case) ** 2 * 1e3 if case["sheet"] else 0.0,
                             rho=RHO, project=case["project"], pcg_maxiter=2000, pcg_rtol=1e-6)


def _views(ctx, s_in, s_out, grid):
    """A step's outputs: the sort's, the new state (the modes in four groups of one
    magnitude each), the grids."""
    if ctx.coeff_format == "f32":
        cuts = [c for c in (0, 1, 4, 8, 27) if c <= ctx.num_modes]
        coeff = [s_out.coeff[:, a:b] for a, b in zip(cuts, cuts[1:])]
    else:
        coeff = [s_out.coeff, s_out.scale]
    out = {"key": s_in.key, "slot": s_in.perm, "start": s_in.cell_start, "x": s_out.x,
           "mass": s_out.mass, "coeff": coeff, "m": grid.mass, "mv": grid.mom, "v": grid.vel}
    if s_out.mass_abs is not None:
        out["absorbed"] = s_out.mass_abs
    return out


def prepare(case, seed):
    st = {"kind": case["kind"], "case": case}
    if case["kind"] == "rollout":
        x, mass, _, g = _particles(case, seed)
        c = _coefficients(case, x, seed, g, 0, x.shape[1])
        st.update(ctx=_context(case), x=x.requires_grad_(), mass=mass, c=c.requires_grad_(),
                  target=_face_field(case, seed + 7), full=RHO * _dx(case) ** 3)
        return st
    ctx = st["ctx"] = _context(case)
    st["params"] = _params(case)
    x, mass, _, g = _particles(case, seed)
    P = x.shape[1]
    if case["kind"] == "step":
        st["fluid"] = _fill_state(case, ctx, x, mass, None, seed, g)
        st["fluid_out"] = ctx.new_particles(P, device=DEV)
        st["grid"] = ctx.new_grid(device=DEV)
        st["out"] = {"fluid": _views(ctx, st["fluid"], st["fluid_out"], st["grid"])}
        S = _sheet_count(case)
        if S:
            xs, ms, ab, gs = _particles(case, seed, sheet=True)
            st["solid"] = _fill_state(case, ctx, xs, ms, ab, seed, gs)
            st["solid_out"] = ctx.new_particles(S, solid=True, device=DEV)
            st["solid_grid"] = ctx.new_grid(device=DEV)
            st["out"]["solid"] = _views(ctx, st["solid"], st["solid_out"], st["solid_grid"])
        st["ws"] = ctx.workspace(P, S, device=DEV)
        return st
    # the grids of a forward step: its mass, and momentum of a smooth field with noise
    st["ws"] = ctx.workspace(P, device=DEV)
    grid = st["grid"] = ctx.new_grid(device=DEV)
    m = _p2g_mass(x, mass, _dims(case), _dx(case))
    vel = _face_field(case, seed)
    for a in range(3):
        v = vel[a] + 0.1 * torch.randn(vel[a].shape, generator=g, device=DEV)
        grid.mass[a].copy_(m[a])
        grid.mom[a].copy_(grid.mass[a] * v)
    if case["kind"] == "project":
        s = ctx.new_particles(P, device=DEV)
        s.x.copy_(x)
        pp.polypic_sort(ctx, s, st["ws"])
        st["fluid"], st["out"] = s, grid.vel
        return st
    s = st["fluid"] = _fill_state(case, ctx, x, mass, None, seed, g)
    pp.polypic_sort(ctx, s, st["ws"])
    for a, v in enumerate(_update(case, [t.double() for t in grid.mass], [t.double() for t in grid.mom])):
        grid.vel[a].copy_(v)
    R, dx = case["modes"], _dx(case)
    deg = torch.tensor([sum(t) for t in _triples(R)], device=DEV, dtype=torch.float64)
    bar = st["bar"] = ctx.new_particles(P, device=DEV)
    bar.coeff.copy_(torch.randn(bar.coeff.shape, generator=g, device=DEV) * (dx ** deg).float()[None, :, None])
    bar.x.copy_(torch.randn(bar.x.shape, generator=g, device=DEV) / dx)
    st["bar_grid"] = ctx.new_grid(device=DEV)
    st["bar_g2p"] = pp.ParticleState(x=torch.empty_like(s.x), mass=s.mass, coeff=s.coeff, key=s.key,
                                     perm=s.perm, cell_start=s.cell_start)
    st["bar_p2g"] = ctx.new_particles(P, device=DEV)
    cuts = [c for c in (0, 1, 4, 8, 27) if c <= R]
    st["out"] = {"v": st["bar_grid"].vel, "m": st["bar_grid"].mass, "mv": st["bar_grid"].mom,
                 "x_g2p": st["bar_g2p"].x, "x_p2g": st["bar_p2g"].x,
                 "coeff": [st["bar_p2g"].coeff[:, a:b] for a, b in zip(cuts, cuts[1:])]}
    return st


def _face_field(case, seed):
    n, dx = _dims(case), _dx(case)
    out = []
    for a in range(3):
        ax = [(torch.arange(n[b] + (a == b), device=DEV, dtype=torch.float64) + (0.0 if a == b else 0.5)) * dx
              for b in range(3)]
        z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        out.append(_field(torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)]), seed)[a].reshape(x.shape).float())
    return out


# ------------------------------------------------------------------ run

def run(st):
    kind = st["kind"]
    if kind == "step":
        if "solid" in st:
            pp.polypic_step(st["ctx"], st["fluid"], st["fluid_out"], st["grid"], st["params"],
                            st["ws"], solid_in=st["solid"], solid_out=st["solid_out"],
                            gs=st["solid_grid"])
        else:
            pp.polypic_step(st["ctx"], st["fluid"], st["fluid_out"], st["grid"], st["params"],
                            st["ws"])
        return st["out"]
    if kind == "project":
        pp.polypic_grid_update(st["ctx"], st["grid"], st["params"], fluid_particles=st["fluid"],
                               ws=st["ws"])
        return st["out"]
    if kind == "adjoint":
        ctx, s, g, bg, ws = st["ctx"], st["fluid"], st["grid"], st["bar_grid"], st["ws"]
        pp.polypic_g2p_adjoint(ctx, g, s, st["params"].dt, st["bar"], bg, st["bar_g2p"], ws)
        pp.polypic_grid_update_adjoint(ctx, g, st["params"], bg, bg)
        pp.polypic_p2g_adjoint(ctx, s, bg, st["bar_p2g"], ws)
        return st["out"]
    case = st["case"]
    vel, m = autograd.rollout(st["ctx"], st["x"], st["mass"], st["c"], case["steps"], _dt(case),
                              gravity=GRAVITY, checkpoint_every=2)
    loss = sum((0.5 * (w / st["full"]) * (v - u) ** 2).sum() for v, w, u in zip(vel, m, st["target"]))
    gc, gx = torch.autograd.grad(loss, [st["c"], st["x"]])
    return {"v": [v.detach() for v in vel], "loss": loss.detach(), "c": gc, "x": gx}


# ------------------------------------------------------------------ 64-bit values

CHUNK = 1 << 18


def _axis(x, b, a, n, dx):
    """Lowest stencil node, offset t and quadratic-mode guard of positions x (N,)
    along axis b on face grid a: the integers from the FP32 position."""
    inv = torch.tensor(1.0 / dx, dtype=torch.float32, device=x.device)
    v = x.detach().float() * inv
    X = v if a == b else v - 0.5
    base = torch.floor(X - 0.5)
    t32 = X - (base + 1.0)
    guard = (1.0 - 2.0 * t32) * (1.0 + 2.0 * t32) < 2.0 ** -10
    base = base.double()
    t = x / dx - (0.0 if a == b else 0.5) - (base + 1.0)
    return base.long(), t, guard


def _weights(t):
    return torch.stack([0.5 * (0.5 - t) ** 2, 0.75 - t ** 2, 0.5 * (0.5 + t) ** 2], -1)


def _offsets(t, dx):
    return (torch.arange(-1, 2, device=t.device, dtype=torch.float64) - t[:, None]) * dx


def _basis(z, t, dx, D):
    """f_0 .. f_{D-1} at offsets z (N, ...) of particles with offset t."""
    t = t.reshape(t.shape + (1,) * (z.dim() - 1))
    f = [torch.ones_like(z), z, z * z - dx * t * (1 - 4 * t * t) * z - 0.25 * dx * dx]
    return torch.stack(f[:D], 1)


def _p2g_factors(t, dx, D):
    return _weights(t)[:, None, :] * _basis(_offsets(t, dx), t, dx, D)


def _g2p_factors(t, guard, dx, D):
    W = _weights(t)
    rows = [W, W * _offsets(t, dx) / (0.25 * dx * dx)]
    if D > 2:
        second = torch.tensor([0.5, -1.0, 0.5], device=t.device, dtype=torch.float64) / dx ** 2
        rows.append((~guard)[:, None] * second[None, :])
    return torch.stack(rows[:D], 1)


def _degrees(R):
    return 3 if R == 27 else 2


def _dense(c, R):
    """(R, N) modes -> (N, D, D, D) by per-axis degree."""
    D = _degrees(R)
    at = torch.tensor([(a * D + b) * D + e for a, b, e in _triples(R)], device=c.device)
    return torch.zeros((c.shape[1], D ** 3), dtype=c.dtype, device=c.device).index_copy(1, at, c.T).reshape(-1, D, D, D)


def _nodes(base, n, a):
    """Flat indices (N, 3, 3, 3) [kx][ky][kz] of the stencils on face grid a."""
    k = torch.arange(3, device=base[0].device)
    d = [n[b] + (a == b) for b in range(3)]
    ix, iy, iz = (base[b][:, None] + k for b in range(3))
    return (iz[:, None, None, :] * d[1] + iy[:, None, :, None]) * d[0] + ix[:, :, None, None]


def _empty_grids(n):
    return [torch.zeros((n[2] + (a == 2)) * (n[1] + (a == 1)) * (n[0] + (a == 0)), dtype=torch.float64,
                        device=DEV) for a in range(3)]


def _shape(grids, n):
    return [g.reshape(n[2] + (a == 2), n[1] + (a == 1), n[0] + (a == 0)) for a, g in enumerate(grids)]


def _p2g_mass(x, mass, n, dx):
    out = _empty_grids(n)
    for lo in range(0, x.shape[1], CHUNK):
        xs, m = x[:, lo:lo + CHUNK].double(), mass[lo:lo + CHUNK].double()
        for a in range(3):
            ax = [_axis(xs[b], b, a, n, dx) for b in range(3)]
            W = [_weights(t) for _, t, _ in ax]
            w = m[:, None, None, None] * W[0][:, :, None, None] * W[1][:, None, :, None] * W[2][:, None, None, :]
            out[a].index_add_(0, _nodes([b for b, _, _ in ax], n, a).reshape(-1), w.reshape(-1))
    return _shape(out, n)


def _p2g(x, mass, c, n, dx, R, map_dt=None):
    """m and mv on the three face grids; differentiable in x and c."""
    D = _degrees(R)
    m_out, v_out = _empty_grids(n), _empty_grids(n)
    for lo in range(0, x.shape[1], CHUNK):
        xs, m, cs = x[:, lo:lo + CHUNK].double(), mass[lo:lo + CHUNK].double(), c[:, :, lo:lo + CHUNK].double()
        if map_dt is not None:
            C = cs[:, 1:4].permute(2, 0, 1)
            M = torch.linalg.inv(torch.eye(3, dtype=torch.float64, device=DEV) + map_dt * C)
        for a in range(3):
            ax = [_axis(xs[b], b, a, n, dx) for b in range(3)]
            W = [_weights(t) for _, t, _ in ax]
            w = m[:, None, None, None] * W[0][:, :, None, None] * W[1][:, None, :, None] * W[2][:, None, None, :]
            T = _dense(cs[a], R)
            if map_dt is None:
                F = [_p2g_factors(t, dx, D) for _, t, _ in ax]
                T = torch.einsum("pabc,pck->pabk", T, F[2])
                T = torch.einsum("pabk,pbj->pajk", T, F[1])
                v = m[:, None, None, None] * torch.einsum("pajk,pai->pijk", T, F[0])
            else:
                z = [_offsets(t, dx) for _, t, _ in ax]
                N = z[0].shape[0]
                z = torch.stack([z[0][:, :, None, None].expand(N, 3, 3, 3), z[1][:, None, :, None].expand(N, 3, 3, 3),
                                 z[2][:, None, None, :].expand(N, 3, 3, 3)], 1).reshape(N, 3, 27)
                xi = torch.bmm(M, z)
                f = [_basis(xi[:, b], ax[b][1], dx, D) for b in range(3)]
                T = torch.einsum("pabc,pcn->pabn", T, f[2])
                T = (T * f[1][:, None]).sum(2)
                v = w * (T * f[0]).sum(1).reshape(N, 3, 3, 3)
            at = _nodes([b for b, _, _ in ax], n, a).reshape(-1)
            m_out[a] = m_out[a].index_add(0, at, w.reshape(-1)) if x.requires_grad else m_out[a].index_add_(0, at, w.reshape(-1))
            v_out[a] = v_out[a].index_add(0, at, v.reshape(-1)) if x.requires_grad else v_out[a].index_add_(0, at, v.reshape(-1))
    return _shape(m_out, n), _shape(v_out, n)


def _g2p(vel, x, n, dx, R, dt):
    """c (3, R, N) and the advected positions; differentiable in vel and x."""
    D = _degrees(R)
    at = torch.tensor([(a * D + b) * D + e for a, b, e in _triples(R)], device=DEV)
    parts = []
    for lo in range(0, x.shape[1], CHUNK):
        xs = x[:, lo:lo + CHUNK].double()
        c = []
        for a in range(3):
            ax = [_axis(xs[b], b, a, n, dx) for b in range(3)]
            G = [_g2p_factors(t, gd, dx, D) for _, t, gd in ax]
            v = vel[a].reshape(-1)[_nodes([b for b, _, _ in ax], n, a)]
            T = torch.einsum("pijk,pai->pajk", v, G[0])
            T = torch.einsum("pajk,pbj->pabk", T, G[1])
            T = torch.einsum("pabk,pck->pabc", T, G[2])
            c.append(T.reshape(-1, D ** 3)[:, at].T)
        parts.append(torch.stack(c))
    c = torch.cat(parts, 2) if len(parts) > 1 else parts[0]
    lo = 1.5 * dx
    xo = torch.stack([(x[b].double() + dt * c[b, 0]).clamp(lo, (n[b] - 1.5) * dx) for b in range(3)])
    return c, xo


def _update(case, m, mv, solid=None):
    """v~ of one phase, or of both with drag; walls; no projection."""
    dt, n = np.float32(_dt(case)).item(), _dims(case)
    K = np.float32(_params(case).drag_k).item()
    out, out_s = [], []
    for a in range(3):
        g = np.float32(GRAVITY[a]).item()
        v = torch.where(m[a] > 0, mv[a] / torch.where(m[a] > 0, m[a], 1.0), 0.0) + dt * g
        if solid is not None:
            ms, ps = solid[0][a], solid[1][a]
            vs = torch.where(ms > 0, ps / torch.where(ms > 0, ms, 1.0), 0.0) + dt * g
            both = (m[a] > 0) & (ms > 0)
            mf, mq = torch.where(both, m[a], 1.0), torch.where(both, ms, 1.0)
            mean = (mf * v + mq * vs) / (mf + mq)
            u = (v - vs) / (1 + dt * K * (1 / mf + 1 / mq))
            v, vs = (torch.where(both, mean + mq / (mf + mq) * u, v),
                     torch.where(both, mean - mf / (mf + mq) * u, vs))
        wall = torch.ones(n[a] + 1, dtype=torch.float64, device=DEV)
        wall[0] = wall[-1] = 0.0
        wall = wall.reshape([-1 if 2 - d == a else 1 for d in range(3)])
        out.append(v * wall)
        if solid is not None:
            out_s.append(vs * wall)
    return out if solid is None else (out, out_s)


def _projected(case, vel, cells):
    """vel made divergence free on the cells that hold particles (boolean
    (nz, ny, nx)), p = 0 elsewhere, no flow through walls: CG in 64 bits."""
    n = _dims(case)
    fl = cells.double()
    axis = {0: 2, 1: 1, 2: 0}
    deg = torch.full(cells.shape, 6.0, dtype=torch.float64, device=DEV)
    for a in range(3):
        for at in (0, n[a] - 1):
            deg.select(axis[a], at).sub_(1.0)
    rhs = 0.0
    for a in range(3):
        rhs = rhs - (vel[a].narrow(axis[a], 1, n[a]) - vel[a].narrow(axis[a], 0, n[a]))
    rhs = rhs * fl

    def lap(p):
        q = deg * p
        for a in range(3):
            d, m = axis[a], n[a] - 1
            q.narrow(d, 0, m).sub_(p.narrow(d, 1, m))
            q.narrow(d, 1, m).sub_(p.narrow(d, 0, m))
        return q * fl

    p, r = torch.zeros_like(rhs), rhs.clone()
    z = r / deg
    d, rz, b2 = z.clone(), (r * z).sum(), float((rhs * rhs).sum())
    for it in range(6000):
        q = lap(d)
        al = rz / (d * q).sum()
        p.add_(al * d)
        r.sub_(al * q)
        z = r / deg
        new = (r * z).sum()
        d = z + (new / rz) * d
        rz = new
        if it % 50 == 49 and float((r * r).sum()) <= 1e-24 * b2:
            break
    out = []
    for a in range(3):
        v, dd = vel[a].clone(), axis[a]
        v.narrow(dd, 1, n[a] - 1).sub_(p.narrow(dd, 1, n[a] - 1) - p.narrow(dd, 0, n[a] - 1))
        out.append(v)
    return out


def _occupied(x, n, dx):
    i, j, k = _cells_of(x, n, dx)
    return (torch.bincount((k * n[1] + j) * n[0] + i, minlength=n[0] * n[1] * n[2]) > 0).reshape(n[2], n[1], n[0])


def _decoded(case, s):
    """Coefficients (3, R, P) of a state, in 64 bits for the 16-bit formats."""
    if case["format"] == "f32":
        return s.coeff
    R = case["modes"]
    deg = torch.tensor([sum(t) for t in _triples(R)], device=DEV, dtype=torch.float64)
    c = s.coeff.permute(0, 1, 3, 2).reshape(3, -1, s.count)[:, :R].double()
    return c * s.scale.double() * (_dx(case) ** -deg)[None, :, None]


def _exact_phase(case, s, vel, grids):
    n, dx, R = _dims(case), _dx(case), case["modes"]
    slot = _slots(s.x, n, dx)[1]
    x, dt = s.x[:, slot], np.float32(_dt(case)).item()
    c, xo = _g2p(vel, x, n, dx, R, dt)
    if case["format"] == "f32":
        cuts = [k for k in (0, 1, 4, 8, 27) if k <= R]
        coeff = [c[:, a:b] for a, b in zip(cuts, cuts[1:])]
    else:
        deg = torch.tensor([sum(t) for t in _triples(R)], device=DEV, dtype=torch.float64)
        c = c * (dx ** deg)[None, :, None]
        scale = c.abs().amax(dim=(0, 1))
        H = (R + 1) // 2
        codes = torch.zeros((3, H, s.count, 2), dtype=torch.float64, device=DEV)
        for r in range(R):
            codes[:, r // 2, :, r % 2] = c[:, r] / scale
        coeff = [codes, scale]
    out = {"key": None, "slot": None, "start": None, "x": xo, "mass": s.mass[slot].double(),
           "coeff": coeff, "m": grids[0], "mv": grids[1], "v": vel}
    if s.mass_abs is not None:
        out["absorbed"] = s.mass_abs[slot].double()
    return out


def exact(case, seed):
    if _count(case) > 6_000_000:
        return None
    n, dx, R, dt = _dims(case), _dx(case), case["modes"], np.float32(_dt(case)).item()
    if case["kind"] == "rollout":
        return _exact_rollout(case, seed)
    st = prepare(case, seed)
    s = st["fluid"]
    if case["kind"] == "step":
        map_dt = dt if case["affine"] else None
        gf = _p2g(s.x, s.mass, _decoded(case, s), n, dx, R, map_dt)
        if "solid" not in st:
            vel = _update(case, *gf)
            if case["project"]:
                vel = _projected(case, vel, _occupied(s.x, n, dx))
            return {"fluid": _exact_phase(case, s, vel, gf)}
        q = st["solid"]
        gs = _p2g(q.x, q.mass.double() + q.mass_abs.double(), _decoded(case, q), n, dx, R, map_dt)
        vf, vs = _update(case, *gf, solid=gs)
        if case["project"]:
            vf = _projected(case, vf, _occupied(s.x, n, dx))
        return {"fluid": _exact_phase(case, s, vf, gf), "solid": _exact_phase(case, q, vs, gs)}
    g = st["grid"]
    m, mv = [t.double() for t in g.mass], [t.double() for t in g.mom]
    if case["kind"] == "project":
        return _projected(case, _update(case, m, mv), _occupied(s.x, n, dx))
    # adjoint: the gradients of <bar c, c'> + <bar x, x'>, chunk by chunk
    slot = _slots(s.x, n, dx)[1]
    vel = [v.double().requires_grad_() for v in g.vel]
    gx = torch.zeros((3, s.count), dtype=torch.float64, device=DEV)
    for lo in range(0, s.count, CHUNK):
        at = slot[lo:lo + CHUNK]
        x = s.x[:, at].double().requires_grad_()
        c, xo = _g2p(vel, x, n, dx, R, dt)
        loss = (c * st["bar"].coeff[:, :, lo:lo + CHUNK]).sum() + (xo * st["bar"].x[:, lo:lo + CHUNK]).sum()
        loss.backward()
        gx[:, at] = x.grad
    bar_v = [v.grad for v in vel]
    m, mv = [t.requires_grad_() for t in m], [t.requires_grad_() for t in mv]
    sum((v * w).sum() for v, w in zip(_update(case, m, mv), bar_v)).backward()
    bar_m, bar_mv = [t.grad for t in m], [t.grad for t in mv]
    px, pc = torch.zeros_like(gx), torch.zeros((3, R, s.count), dtype=torch.float64, device=DEV)
    for lo in range(0, s.count, CHUNK):
        at = slice(lo, min(s.count, lo + CHUNK))
        x, c = s.x[:, at].double().requires_grad_(), s.coeff[:, :, at].double().requires_grad_()
        a, b = _p2g(x, s.mass[at], c, n, dx, R)
        sum((u * w).sum() for u, w in zip(a + b, bar_m + bar_mv)).backward()
        px[:, at], pc[:, :, at] = x.grad, c.grad
    cuts = [k for k in (0, 1, 4, 8, 27) if k <= R]
    return {"v": bar_v, "m": bar_m, "mv": bar_mv, "x_g2p": gx, "x_p2g": px,
            "coeff": [pc[:, a:b] for a, b in zip(cuts, cuts[1:])]}


def _exact_rollout(case, seed):
    st = prepare(case, seed)
    n, dx, R, dt = _dims(case), _dx(case), case["modes"], np.float32(_dt(case)).item()
    x0, c0 = st["x"].detach().double().requires_grad_(), st["c"].detach().double().requires_grad_()
    x, c = x0, c0
    for k in range(case["steps"]):
        m, mv = _p2g(x, st["mass"], c, n, dx, R)
        vel = _update(case, m, mv)
        c, x = _g2p(vel, x, n, dx, R, dt)
    loss = sum((0.5 * (w.detach() / st["full"]) * (v - u.double()) ** 2).sum()
               for v, w, u in zip(vel, m, st["target"]))
    gc, gx = torch.autograd.grad(loss, [c0, x0])
    return {"v": [v.detach() for v in vel], "loss": loss.detach(), "c": gc, "x": gx}
