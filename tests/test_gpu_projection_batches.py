"""The projection stopped after any number of iterations (also inside a batch of
8, whose launches are not the captured graph's), and with fluid cells on the
box's own faces, against the oracle's FP64 solve."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_01060_gb300 import polypic as pp
from gpu_util import assert_close, grid_from_host, np_, random_grid_velocity

pytestmark = pytest.mark.gpu
DT = 1e-3


def _problem(n, cells, seed):
    """Context, particles in the middle of `cells` and sorted, face velocities,
    the fluid mask and the exactly projected velocity."""
    dx = 1.0 / n[0]
    x = np.ascontiguousarray(((cells + 0.5) * dx).T.astype(np.float32))
    ctx = pp.Context(n, dx, 4)
    ps = pp.upload_particles(ctx, x, np.ones(x.shape[1], np.float32))
    ws = ctx.workspace(ps.count)
    pp.polypic_sort(ctx, ps, ws)
    pp.polypic_check_device_status(ctx)      # cells on the faces are outside the valid region
    v = random_grid_velocity(n, dx, seed=seed)
    ones = [np.ones_like(a) for a in v]
    fluid = np.zeros((n[2], n[1], n[0]), bool)
    fluid[cells[:, 2], cells[:, 1], cells[:, 0]] = True
    prm = pp.UpdateSettings(dt=DT, project=True)
    fv = oracle.grid_update(n, DT, prm.gravity, ones, v)
    vp = oracle.pcg_project(n, dx, DT, 1000.0, fluid, fv, rtol=1e-11, maxiter=8000)[0]

    def project(**settings):
        g = grid_from_host(ctx, mass=ones, mom=v)
        p = pp.UpdateSettings(dt=DT, project=True, **settings)
        try:
            pp.polypic_grid_update(ctx, g, p, fluid_particles=ps, ws=ws)
            converged = True
        except pp.PolyPICError as e:
            assert e.name == "NOT_CONVERGED"
            converged = False
        assert (pp.polypic_check_device_status(ctx) == 0) == converged
        return [np_(a) for a in g.vel], converged

    return project, vp


@pytest.mark.parametrize("n", [(8, 8, 8), (24, 20, 18), (40, 36, 33)])
def test_every_iteration_brings_the_velocity_closer(n):
    """Conjugate gradients minimise the pressure error's energy norm, which is the
    L2 norm of the velocity error, over spaces that grow with every iteration: it
    falls with each, whichever batch the iteration is in, down to FP32 rounding
    (1e-5 of the velocity, as for the suite's other FP32 sums)."""
    inner = np.stack(np.meshgrid(*[np.arange(1, m - 1) for m in n], indexing="ij"), -1).reshape(-1, 3)
    cells = inner[np.random.default_rng(n[0]).random(len(inner)) < 0.8]
    project, vp = _problem(n, cells, seed=3)
    size = np.sqrt(sum((a ** 2).sum() for a in vp))
    err = []
    for it in range(1, 22):
        v, converged = project(pcg_rtol=1e-12, pcg_maxiter=it)
        err.append(np.sqrt(sum(((a - b) ** 2).sum() for a, b in zip(v, vp))) / size)
    for a, b in zip(err, err[1:]):
        assert b < a or b < 1e-5, err
    assert err[12] < 0.1 * err[0]            # five iterations into the second batch


@pytest.mark.parametrize("n", [(9, 7, 8), (24, 20, 18), (33, 40, 21)])
def test_fluid_on_the_faces_of_the_box(n):
    every = np.stack(np.meshgrid(*[np.arange(m) for m in n], indexing="ij"), -1).reshape(-1, 3)
    cells = every[np.random.default_rng(n[1]).random(len(every)) < 0.7]
    project, vp = _problem(n, cells, seed=4)
    v, converged = project(pcg_rtol=1e-6, pcg_maxiter=2000)
    assert converged
    for a in range(3):
        assert_close(v[a], vp[a], 1e-4, f"v {a}")
