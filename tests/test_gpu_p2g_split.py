"""Both splits of the P2G chunk kernel (four block groups a tile below 152 * 4 *
2048 particles, two from there on) in every form it has: 27 modes in the three
coefficient formats, solid phases of 4, 8 and 27 modes, Eq 12's affine map of 8
and 27, and the G2P adjoint's scatter, each against the FP64 oracle on a grid no
tile divides, with uneven cells, one-layer blocks, a crowded cell, lone particles
and empty blocks.

Tolerances: 1e-5 for the sums, as in the tests of the single forms, and what the
rounding of a position costs beside it: v = fl(x fl(1/dx)) is off by up to 2 * 2^-24
of itself, 2^-23 max(n) cells, and a node's weight times a mode changes by no more
than that times the particle's own contribution; 1e-4 for the positions' adjoint."""
import os

import numpy as np
import pytest
import torch

import oracle
import slot_layout
from paper_2308_01060_gb300 import polypic as pp
from paper_2308_01060_gb300 import scenes
from gpu_util import (assert_close, decoded, grid_from_host, np_, random_grid_velocity, sorted_particles,
                      u32)

pytestmark = pytest.mark.gpu
SPLIT = 152 * 4 * 2048
GRIDS = {"wide": (29, 14, 23), "narrow": (61, 58, 63)}


def _tol(n):
    return 1e-5 + 2.0 ** -23 * max(n)


def _positions(split, seed):
    """(3, P) float32, dx = 1 / n[0], in shuffled order."""
    n = GRIDS[split]
    rng = np.random.default_rng(seed)
    hi = np.array(n) - 2
    many = 4000 if split == "wide" else SPLIT
    parts = [rng.integers([2, 2, 2], np.minimum(hi, 40), size=(many, 3)),     # uneven cells
             np.stack([rng.integers(2, hi[0], 1500), np.full(1500, hi[1] - 2),
                       rng.integers(2, hi[2], 1500)], 1),                     # a layer
             np.tile(hi - 1, (150, 1)),                                       # one crowded cell
             rng.integers([2, 2, 2], hi, size=(40, 3))]                       # lone particles
    cells = np.concatenate(parts)
    cells = cells[rng.permutation(len(cells))]
    assert (len(cells) < SPLIT) == (split == "wide")
    x = (cells + rng.random(cells.shape) * 0.999 + 5e-4) / n[0]
    return np.ascontiguousarray(x.T.astype(np.float32))


def _modes(R, P, dx, rng):
    """Random coefficients of one magnitude over a cell, (3, R, P) float32."""
    c = rng.standard_normal((3, R, P), dtype=np.float32)
    return c * (dx ** -scenes.mode_degrees(R)).astype(np.float32)[None, :, None]


def _with_oracle(fn, *args, **kw):
    oracle.set_threads(os.cpu_count() or 1)
    try:
        return fn(*args, **kw)
    finally:
        oracle.set_threads(1)


@pytest.mark.parametrize("split", GRIDS)
@pytest.mark.parametrize("R,fmt,solid,affine", [
    (27, "f32", False, False), (27, "f32", True, False), (8, "f32", True, False),
    (4, "f32", True, False), (8, "f32", False, True), (27, "f32", True, True),
    (27, "bf16", False, False), (27, "f16", True, False)])
def test_p2g_in_every_form(split, R, fmt, solid, affine):
    n = GRIDS[split]
    dx, dt = 1.0 / n[0], 1e-3
    x = _positions(split, R)
    P = x.shape[1]
    rng = np.random.default_rng(R + 1)
    mass = (1e-3 * (0.5 + rng.random(P))).astype(np.float32)
    ab = (5e-4 * rng.random(P)).astype(np.float32) if solid else None
    ctx = pp.Context(n, dx, R, coeff_format=fmt, map_affine=affine)
    ps = pp.upload_particles(ctx, x, mass, mass_abs=ab)
    if fmt == "f32":
        c = _modes(R, P, dx, rng)
        ps.coeff.copy_(torch.as_tensor(c))
    else:
        ps.coeff.copy_(torch.as_tensor(rng.uniform(-1, 1, ps.coeff.shape)).to(ps.coeff.dtype))
        ps.scale.copy_(torch.as_tensor(0.5 + rng.random(P), dtype=torch.float32))
        c = decoded(ps, R, dx)
    ws = ctx.workspace(P)
    pp.polypic_sort(ctx, ps, ws)
    g, again = ctx.new_grid(vel=False), ctx.new_grid(vel=False)
    pp.polypic_p2g_mapped(ctx, ps, g, dt, ws)
    pp.polypic_p2g_mapped(ctx, ps, again, dt, ws)
    assert pp.polypic_check_device_status(ctx) == 0
    assert all(np.array_equal(u32(p), u32(q)) for p, q in zip(g.mass + g.mom, again.mass + again.mom))
    m, mv = _with_oracle(oracle.p2g, x, mass, c, n, dx, mass_abs=ab, map_affine=affine, dt=dt)
    for a in range(3):
        assert_close(np_(g.mass[a]), m[a], _tol(n), f"mass {a}")
        assert_close(np_(g.mom[a]), mv[a], _tol(n), f"momentum {a}")


@pytest.mark.parametrize("split,accumulate", [("wide", False), ("wide", True), ("narrow", True)])
def test_the_scatter_of_the_g2p_adjoint(split, accumulate):
    R, n, dt = 27, GRIDS[split], 1e-3
    dx = 1.0 / n[0]
    x = _positions(split, 5)
    P = x.shape[1]
    ctx = pp.Context(n, dx, R)
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=np.ones(P, np.float32), coeff=None))
    rng = np.random.default_rng(6)
    gv = random_grid_velocity(n, dx, seed=7)
    lc = _modes(R, P, 1.0 / dx, rng)      # dx^degree: of one magnitude in the fit's units
    lx = rng.standard_normal((3, P), dtype=np.float32)
    perm = slot_layout.library_order(x, n, dx)[0]
    bar_out, bar = ctx.new_particles(P), ctx.new_particles(P)
    bar_out.coeff.copy_(torch.from_numpy(np.ascontiguousarray(lc[:, :, perm])))
    bar_out.x.copy_(torch.from_numpy(np.ascontiguousarray(lx[:, perm])))
    bar.x.zero_()
    v0 = [rng.standard_normal(oracle.face_shape(a, n)).astype(np.float32) for a in range(3)]
    bar_v = grid_from_host(ctx, vel=v0)
    pp.polypic_g2p_adjoint(ctx, grid_from_host(ctx, vel=gv), ps, dt, bar_out, bar_v, bar, ws,
                           accumulate=accumulate)
    assert pp.polypic_check_device_status(ctx) == 0
    lv, lx0 = _with_oracle(oracle.g2p_adjoint, x, gv, R, n, dx, dt, lc, lx)
    for a in range(3):
        assert_close(np_(bar_v.vel[a]), lv[a] + (v0[a] if accumulate else 0.0), _tol(n), f"grid {a}")
    assert_close(np_(bar.x), lx0, 1e-4, "positions")


@pytest.mark.parametrize("split", GRIDS)
@pytest.mark.parametrize("R,solid,affine", [(27, False, False), (4, True, False), (8, False, True)])
def test_a_stale_sort_inside_a_block_is_latched(split, R, solid, affine):
    """A particle that has moved to another cell of its own 4x4x2 block."""
    n = GRIDS[split]
    dx = 1.0 / n[0]
    x = _positions(split, 3)
    ctx = pp.Context(n, dx, R, map_affine=affine)
    ab = np.zeros(x.shape[1], np.float32) if solid else None
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=np.ones(x.shape[1], np.float32), coeff=None,
                                                      mass_abs=ab))
    g = ctx.new_grid(vel=False)
    pp.polypic_p2g_mapped(ctx, ps, g, 1e-3, ws)
    assert pp.polypic_check_device_status(ctx) == 0
    cell = np.floor(x[:, :200] * np.float32(n[0]))
    p = int(np.flatnonzero((cell[0] % 4 < 3) & (cell[0] < n[0] - 4))[0])
    ps.x[0, p] = float((cell[0, p] + 1.5) * dx)
    pp.polypic_p2g_mapped(ctx, ps, g, 1e-3, ws)
    assert pp.polypic_check_device_status(ctx) == 3
