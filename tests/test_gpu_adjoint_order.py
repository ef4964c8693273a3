"""The P2G adjoint walks a tile's particles in memory order: inputs in random
order (indices far outside the tile's window), tiles above the listed size, and
both forms of the outputs, against the oracle.  Tolerances as for the suite's
other P2G adjoints (1e-5 for the coefficients, 1e-4 for the positions)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_01060_gb300 import polypic as pp
from paper_2308_01060_gb300 import scenes
from gpu_util import assert_close, grid_from_host, np_, sorted_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 4, 8, 27])
@pytest.mark.parametrize("kind", ["shuffled", "crowded", "lone"])
@pytest.mark.parametrize("accumulate", [False, True])
def test_p2g_adjoint_in_any_input_order(R, kind, accumulate):
    n, dx = (17, 15, 22), 1.0 / 17
    rng = np.random.default_rng(R)
    lo, hi = np.array([2, 2, 2]), np.array(n) - 2
    if kind == "shuffled":     # 9 thousand particles in no order
        cells = rng.integers(lo, hi, size=(9000, 3))
    elif kind == "crowded":    # one tile with 3500 particles, among others
        cells = np.concatenate([rng.integers([9, 9, 5], [12, 12, 8], size=(3500, 3)),
                                rng.integers(lo, hi, size=(700, 3))])
    else:                      # tiles of one particle
        cells = np.array([[2, 2, 2], [14, 12, 19], [9, 3, 11]])
    P = len(cells)
    x = np.ascontiguousarray(((cells + 0.02 + 0.96 * rng.random((P, 3))) * dx).T.astype(np.float32))
    mass = (0.5 + rng.random(P)).astype(np.float32)
    c = scenes.random_modes(R, P, dx, rng)
    c[:, 0] = rng.standard_normal((3, P))
    c = c.astype(np.float32)
    ctx = pp.Context(n, dx, R)
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=mass, coeff=c))
    lm, lp = ([rng.standard_normal(oracle.face_shape(a, n)).astype(np.float32) for a in range(3)]
              for _ in range(2))
    bar = ctx.new_particles(P)
    c0 = rng.standard_normal(bar.coeff.shape).astype(np.float32)
    x0 = rng.standard_normal((3, P)).astype(np.float32)
    bar.coeff.copy_(torch.from_numpy(c0))
    bar.x.copy_(torch.from_numpy(x0))
    pp.polypic_p2g_adjoint(ctx, ps, grid_from_host(ctx, mass=lm, mom=lp), bar, ws, accumulate=accumulate)
    assert pp.polypic_check_device_status(ctx) == 0
    lc, lx = oracle.p2g_adjoint(x, mass, c, n, dx, lm, lp)
    if accumulate:
        lc, lx = lc + c0, lx + x0
    assert_close(np_(bar.coeff), lc, 1e-5)
    assert_close(np_(bar.x), lx, 1e-4)
