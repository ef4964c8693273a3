"""The projection's multigrid levels where their sizes can go wrong, against
the oracle's FP64 solve: a single level, a small level right below the finest
one, one and two listed levels, odd dimensions at every level, cells without
fluid neighbours, rows of fluid that end at the box's far faces, and batches
that are not a multiple of the residual checks.

Tolerance 1e-4, as for the suite's other projections: CG runs to a relative
residual of 1e-6 on systems whose smallest eigenvalue is a few 1e-3."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_01060_gb300 import polypic as pp
from gpu_util import assert_close, grid_from_host, np_, random_grid_velocity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(8, 8, 8), (9, 7, 8), (16, 16, 18), (17, 33, 15), (40, 36, 33),
                               (70, 21, 66), (5, 90, 61)])
@pytest.mark.parametrize("fill", [0.2, 0.9])
def test_projection_on_scattered_cells(n, fill):
    dx, dt = 1.0 / n[0], 1e-3
    rng = np.random.default_rng(int(100 * fill) + n[0])
    inner = np.stack(np.meshgrid(*[np.arange(1, m - 1) for m in n], indexing="ij"), -1).reshape(-1, 3)
    cells = inner[rng.random(len(inner)) < fill]
    x = ((cells + 0.5) * dx).T.astype(np.float32)
    ctx = pp.Context(n, dx, 4)
    ps = pp.upload_particles(ctx, np.ascontiguousarray(x), np.ones(x.shape[1], np.float32))
    ws = ctx.workspace(ps.count)
    pp.polypic_sort(ctx, ps, ws)
    v = random_grid_velocity(n, dx, seed=n[1])
    ones = [np.ones_like(a) for a in v]
    g = grid_from_host(ctx, mass=ones, mom=v)
    prm = pp.UpdateSettings(dt=dt, project=True, pcg_rtol=1e-6, pcg_maxiter=2000)
    pp.polypic_grid_update(ctx, g, prm, fluid_particles=ps, ws=ws)
    assert pp.polypic_check_device_status(ctx) == 0
    fluid = np.zeros((n[2], n[1], n[0]), bool)
    fluid[cells[:, 2], cells[:, 1], cells[:, 0]] = True
    fv = oracle.grid_update(n, dt, prm.gravity, ones, v)
    vp, _, _ = oracle.pcg_project(n, dx, dt, 1000.0, fluid, fv, rtol=1e-10, maxiter=5000)
    for a in range(3):
        assert_close(np_(g.vel[a]), vp[a], 1e-4, f"v {a}")
    again = ctx.new_grid()
    for a in range(3):
        again.mass[a].copy_(g.mass[a])
        again.mom[a].copy_(g.mom[a])
    pp.polypic_grid_update(ctx, again, prm, fluid_particles=ps, ws=ws)
    assert all(torch.equal(p, q) for p, q in zip(g.vel, again.vel))  # bit-identical
