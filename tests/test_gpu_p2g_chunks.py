"""The chunk kernel of P2G (27 modes, the node-by-node affine map, solid phases)
against the FP64 oracle where its shapes can go wrong: grids no tile divides,
blocks with few or one live cell, cells above 32 and 64 particles, runs of
empty blocks, solid phases of every mode count, the 16-bit formats' codes, and
both splits of a tile (the wide one below 152 * 4 * 2048 particles).

Tolerance 1e-5, as for every FP32 transfer of this suite: sums of at most a few
hundred terms of one magnitude, each rounded to 2^-24."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_01060_gb300 import polypic as pp
from paper_2308_01060_gb300 import scenes
from gpu_util import assert_close, decoded, np_, sorted_particles, u32

pytestmark = pytest.mark.gpu
TOL = 1e-5


def _points(kind, n, seed):
    """Positions (3, P) float32 in cells of a grid n with dx = 1 / n[0]."""
    dx = 1.0 / n[0]
    rng = np.random.default_rng(seed)
    lo, hi = np.array([2, 2, 2]), np.array(n) - 2
    if kind == "poisson":      # uneven cells, some empty
        P = int(np.prod(hi - lo)) * 3
        cells = rng.integers(lo, hi, size=(P, 3))
    elif kind == "one_cell":   # a single crowded cell, and a far lone particle
        cells = np.concatenate([np.tile(lo, (150, 1)), (hi - 1)[None, :]])
    elif kind == "layer":      # one layer of cells: blocks with 8 live cells
        cells = rng.integers(lo, hi, size=(4000, 3))
        cells[:, 1] = lo[1] + 1
    elif kind == "lines":      # blocks with a few cells of 33 and 65 particles
        cells = np.concatenate([np.tile(lo + [4 * i, 0, 2 * i], (33 + 32 * (i % 2), 1)) for i in range(4)])
    x = (cells + rng.random(cells.shape) * 0.999 + 5e-4) * dx
    return np.ascontiguousarray(x.T.astype(np.float32)), dx


def _check(n, dx, x, R, mass_abs=None, seed=0):
    rng = np.random.default_rng(seed + 100)
    P = x.shape[1]
    mass = (1e-3 * (0.5 + rng.random(P))).astype(np.float32)
    c = scenes.random_modes(R, P, dx, rng)
    c[:, 0] = rng.standard_normal((3, P))
    c = c.astype(np.float32)
    ctx = pp.Context(n, dx, R)
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=mass, coeff=c, mass_abs=mass_abs))
    g = ctx.new_grid(vel=False)
    pp.polypic_p2g(ctx, ps, g, ws)
    assert pp.polypic_check_device_status(ctx) == 0
    m, mv = oracle.p2g(x, mass, c, n, dx, mass_abs=mass_abs)
    for a in range(3):
        assert_close(np_(g.mass[a]), m[a], TOL, f"mass {a}")
        assert_close(np_(g.mom[a]), mv[a], TOL, f"momentum {a}")
    again = ctx.new_grid(vel=False)
    pp.polypic_p2g(ctx, ps, again, ws)
    assert all(np.array_equal(u32(p), u32(q)) for p, q in zip(g.mass + g.mom, again.mass + again.mom))


@pytest.mark.parametrize("n", [(12, 9, 7), (16, 16, 16), (29, 14, 23)])
@pytest.mark.parametrize("kind", ["poisson", "one_cell", "layer", "lines"])
@pytest.mark.parametrize("R,solid", [(27, False), (27, True), (8, True), (4, True)])
def test_chunks_against_oracle(n, kind, R, solid):
    if kind == "lines" and n[0] < 20:
        pytest.skip("needs four blocks along x")
    x, dx = _points(kind, n, seed=R)
    rng = np.random.default_rng(5)
    ab = (5e-4 * rng.random(x.shape[1])).astype(np.float32) if solid else None
    _check(n, dx, x, R, ab)


def test_narrow_split_on_a_large_fluid():
    sc = scenes.dam_break_scene(n=104, R=27)   # 2 million particles: two groups a tile
    f = sc.fluid
    assert f.n >= 152 * 4 * 2048
    _check(sc.n, sc.dx, f.x, 27)


@pytest.mark.parametrize("fmt", ["bf16", "f16"])
def test_chunks_decode_16bit_codes(fmt):
    """P2G of codes equals the oracle's P2G of the decoded coefficients."""
    n, R = (21, 18, 15), 27
    x, dx = _points("poisson", n, seed=3)
    rng = np.random.default_rng(4)
    P = x.shape[1]
    ctx = pp.Context(n, dx, R, coeff_format=fmt)
    mass = (1e-3 * (0.5 + rng.random(P))).astype(np.float32)
    ps = pp.upload_particles(ctx, x, mass)
    ps.coeff.copy_(torch.as_tensor(rng.uniform(-1, 1, ps.coeff.shape)).to(ps.coeff.dtype))
    ps.scale.copy_(torch.as_tensor(0.5 + rng.random(P), dtype=torch.float32))
    ws = ctx.workspace(P)
    g = ctx.new_grid(vel=False)
    pp.polypic_sort(ctx, ps, ws)
    pp.polypic_p2g(ctx, ps, g, ws)
    assert pp.polypic_check_device_status(ctx) == 0
    m, mv = oracle.p2g(x, mass, decoded(ps, R, dx), n, dx)
    for a in range(3):
        assert_close(np_(g.mass[a]), m[a], TOL)
        assert_close(np_(g.mom[a]), mv[a], TOL)


def test_a_stale_sort_is_latched():
    """Positions moved after the sort: the transfer reports it."""
    n = (16, 16, 16)
    x, dx = _points("poisson", n, seed=9)
    ctx = pp.Context(n, dx, 27)
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=np.ones(x.shape[1], np.float32), coeff=None))
    assert pp.polypic_check_device_status(ctx) == 0
    ps.x[0, 0] = (ps.x[0, 0] + 4 * dx) if float(ps.x[0, 0]) < 0.5 else (ps.x[0, 0] - 4 * dx)
    g = ctx.new_grid(vel=False)
    pp.polypic_p2g(ctx, ps, g, ws)
    assert pp.polypic_check_device_status(ctx) == 3
