"""The P2G adjoint reads and writes the particles that `perm` names and no
others, also where the caller's perm names a particle twice (and so leaves
another one out): every named particle gets its gradient, one that is not named
keeps what its outputs held.  Tolerances as for the suite's other P2G adjoints."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_01060_gb300 import polypic as pp
from paper_2308_01060_gb300 import scenes
from gpu_util import assert_close, grid_from_host, np_, sorted_particles, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 4, 8, 27])
def test_only_named_particles(R):
    n, dx, P = (16, 13, 11), 1.0 / 16, 1500
    rng = np.random.default_rng(R)
    cells = rng.integers([2, 2, 2], np.array(n) - 2, size=(P, 3))
    x = np.ascontiguousarray(((cells + 0.02 + 0.96 * rng.random((P, 3))) * dx).T.astype(np.float32))
    mass = (0.5 + rng.random(P)).astype(np.float32)
    c = scenes.random_modes(R, P, dx, rng).astype(np.float32)
    ctx = pp.Context(n, dx, R)
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=mass, coeff=c))
    # every fourth slot of a tile names its predecessor's particle
    perm, start = u32(ps.perm).copy(), u32(ps.cell_start)
    for t in range(ctx.num_keys // 256):
        j = np.arange(start[256 * t], start[256 * t + 256])[3::4]
        perm[j] = perm[j - 1]
    ps.perm.copy_(torch.from_numpy(perm.view(np.int32)))
    named = np.zeros(P, bool)
    named[perm] = True
    assert 0.7 < named.mean() < 0.8
    lm, lp = ([rng.standard_normal(oracle.face_shape(a, n)).astype(np.float32) for a in range(3)]
              for _ in range(2))
    bar = ctx.new_particles(P)
    bar.coeff.fill_(7.0)
    bar.x.fill_(7.0)
    pp.polypic_p2g_adjoint(ctx, ps, grid_from_host(ctx, mass=lm, mom=lp), bar, ws)
    assert pp.polypic_check_device_status(ctx) == 0
    lc, lx = oracle.p2g_adjoint(x, mass, c, n, dx, lm, lp)
    assert_close(np_(bar.coeff)[..., named], lc[..., named], 1e-5)
    assert_close(np_(bar.x)[:, named], lx[:, named], 1e-4)
    assert (np_(bar.coeff)[..., ~named] == 7.0).all() and (np_(bar.x)[:, ~named] == 7.0).all()
