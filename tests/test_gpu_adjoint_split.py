"""Both particle adjoints with two CTAs an SM (4, 8 and 27 modes above 152 * 2048
particles) and with three (one mode above twice as many), against the oracle;
the suite's other adjoint tests are below these lines.  Tolerances as there."""
import os

import numpy as np
import pytest
import torch

import oracle
import slot_layout
from paper_2308_01060_gb300 import polypic as pp
from paper_2308_01060_gb300 import scenes
from gpu_util import assert_close, grid_from_host, np_, random_grid_velocity, sorted_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,n", [(1, 60), (4, 48), (8, 48), (27, 48)])
def test_adjoints_of_large_phases(R, n):
    sc = scenes.random_velocity_scene(n=n, R=R, seed=R, sigma_v=0.3, dt=1e-3, steps=1)
    f, dx = sc.fluid, sc.dx
    assert f.n > 152 * 2048 * (2 if R == 1 else 1)
    ctx = pp.Context(sc.n, dx, R)
    ps, ws = sorted_particles(ctx, f)
    rng = np.random.default_rng(R)
    lm, lp = ([rng.standard_normal(oracle.face_shape(a, sc.n)).astype(np.float32) for a in range(3)]
              for _ in range(2))
    gv = random_grid_velocity(sc.n, dx, seed=R)
    deg = scenes.mode_degrees(R)
    lc_out = (rng.standard_normal((3, R, f.n)) * (dx ** deg)[None, :, None]).astype(np.float32)
    lx_out = rng.standard_normal((3, f.n)).astype(np.float32)
    perm = slot_layout.library_order(f.x, sc.n, dx)[0]
    bar_out = ctx.new_particles(f.n)
    bar_out.coeff.copy_(torch.from_numpy(np.ascontiguousarray(lc_out[:, :, perm])))
    bar_out.x.copy_(torch.from_numpy(np.ascontiguousarray(lx_out[:, perm])))
    bar, bar_v = ctx.new_particles(f.n), ctx.new_grid()
    bar.coeff.fill_(0.5)
    # the positions' adjoint: G2P's, with P2G's added; the coefficients': added to 0.5
    pp.polypic_g2p_adjoint(ctx, grid_from_host(ctx, vel=gv), ps, sc.dt, bar_out, bar_v, bar, ws)
    pp.polypic_p2g_adjoint(ctx, ps, grid_from_host(ctx, mass=lm, mom=lp), bar, ws, accumulate=True)
    assert pp.polypic_check_device_status(ctx) == 0
    oracle.set_threads(os.cpu_count() or 1)
    try:
        lc, lx = oracle.p2g_adjoint(f.x, f.mass, f.coeff, sc.n, dx, lm, lp)
        lv, lx2 = oracle.g2p_adjoint(f.x, gv, R, sc.n, dx, sc.dt, lc_out, lx_out)
    finally:
        oracle.set_threads(1)
    for a in range(3):
        assert_close(np_(bar_v.vel[a]), lv[a], 1e-5, f"grid {a}")
    assert_close(np_(bar.coeff), lc + 0.5, 1e-5, "coefficients")
    assert_close(np_(bar.x), lx + lx2, 1e-4, "positions")
