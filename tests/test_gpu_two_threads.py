"""Two host threads, each with a context, a stream and a workspace of its own:
every call succeeds and leaves the bits that it leaves alone.  The kernels'
shared-memory limits are state of the library, not of a call, so calls that
need different amounts of it must not lower one another's limit."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_2308_01060_gb300 import polypic as pp
from paper_2308_01060_gb300 import scenes
from gpu_util import grid_from_host, random_grid_velocity, sorted_particles

pytestmark = pytest.mark.gpu


def _positions(n, seed, per_cell=3):
    rng = np.random.default_rng(seed)
    lo, hi = np.array([2, 2, 2]), np.array(n) - 2
    cells = rng.integers(lo, hi, size=(int(np.prod(hi - lo)) * per_cell, 3))
    return np.ascontiguousarray(((cells + rng.random(cells.shape) * 0.999 + 5e-4) / n[0]).T.astype(np.float32))


def _run_both(calls, outputs, repeats):
    """Each call alone, then `repeats` times beside the other one's."""
    for call in calls:
        assert call() == pp.POLYPIC_OK
    torch.cuda.synchronize()
    alone = [[t.clone() for t in out()] for out in outputs]
    failed = [0, 0]
    start = threading.Barrier(2)

    def loop(i):
        start.wait()
        for _ in range(repeats):
            failed[i] += calls[i]() != pp.POLYPIC_OK

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0, 0]
    for out, want in zip(outputs, alone):
        assert all(torch.equal(a, b) for a, b in zip(out(), want))


def _p2g_call(n, seed, solid, **ctx_args):
    R = ctx_args.pop("R", 27)
    ctx = pp.Context(n, 1.0 / n[0], R, **ctx_args)
    x = _positions(n, seed)
    rng = np.random.default_rng(seed)
    mass = (0.5 + rng.random(x.shape[1])).astype(np.float32)
    ab = (0.1 * rng.random(x.shape[1])).astype(np.float32) if solid else None
    ps, ws = sorted_particles(ctx, scenes.ParticleSet(x=x, mass=mass, coeff=None, mass_abs=ab))
    ps.coeff.copy_(torch.as_tensor(rng.standard_normal(ps.coeff.shape)))
    if ps.scale is not None:
        ps.scale.fill_(1.0)
    g = ctx.new_grid(vel=False)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    cp, cg = ps.c_struct(), g.c_struct()
    wp, wb = pp._ws(ws)
    L, sp = pp.load_library(), ctypes.c_void_p(stream.cuda_stream)

    def call():
        return L.polypic_p2g_mapped(ctx.handle, ctypes.byref(cp), ctypes.byref(cg), 1e-3, wp, wb, sp)

    return call, (lambda: g.mass + g.mom), (ctx, ps, ws, g, stream)


@pytest.mark.parametrize("kind", [{}, {"coeff_format": "f16"}, {"map_affine": True},
                                  {"map_affine": True, "R": 8}, {"R": 8}])
def test_a_solid_phase_beside_a_fluid(kind):
    a, out_a, keep_a = _p2g_call((16, 16, 16), 1, True, **kind)
    b, out_b, keep_b = _p2g_call((12, 9, 14), 2, False, **kind)
    _run_both([a, b], [out_a, out_b], 5000)


def _projection_call(n, seed, **settings):
    ctx = pp.Context(n, 1.0 / n[0], 4)
    x = _positions(n, seed, per_cell=1)
    ps = pp.upload_particles(ctx, x, np.ones(x.shape[1], np.float32))
    ws = ctx.workspace(ps.count)
    pp.polypic_sort(ctx, ps, ws)
    v = random_grid_velocity(n, 1.0 / n[0], seed=seed)
    g = grid_from_host(ctx, mass=[np.ones_like(c) for c in v], mom=v)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    cp, cg = ps.c_struct(), g.c_struct()
    up = pp.UpdateSettings(dt=1e-3, project=True, **settings).c_struct()
    wp, wb = pp._ws(ws)
    L, sp = pp.load_library(), ctypes.c_void_p(stream.cuda_stream)

    def call():
        return L.polypic_grid_update(ctx.handle, ctypes.byref(cg), None, ctypes.byref(cp),
                                     ctypes.byref(up), wp, wb, sp)

    return call, (lambda: g.vel), (ctx, ps, ws, g, stream)


@pytest.mark.parametrize("settings", [dict(pcg_rtol=0.2, pcg_maxiter=7), dict(pcg_rtol=1e-6)],
                         ids=["launched", "replayed"])
def test_projections_of_two_grids(settings):
    a, out_a, keep_a = _projection_call((72, 56, 64), 3, **settings)
    b, out_b, keep_b = _projection_call((16, 16, 18), 4, **settings)
    _run_both([a, b], [out_a, out_b], 400)
