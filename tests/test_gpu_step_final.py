"""A step without statistics has its state in place when it returns: a stream
that is not ordered behind the step's may read it at once."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev

pytestmark = pytest.mark.gpu


def _problem(geom, shape):
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    r = np.sqrt((x - 0.5 * nx * g.h) ** 2 + (y - 0.5 * ny * g.h) ** 2 + (z - 0.5 * nz * g.h) ** 2)
    p = W.Params(ka=2.0, kd=0.7, gamma_inf=1.0, Df=4e-3, DF=1e-2, eps=0.75 * g.h)
    phi = 0.5 * (1 - np.tanh(np.clip(0.3 - r, -9 * g.h, 9 * g.h) / (2 * p.eps)))
    rng = np.random.default_rng(7)
    F = 1 + 0.2 * rng.uniform(-1, 1, shape)
    f = 0.2 * (1 + 0.3 * rng.uniform(-1, 1, shape)) * phi * (1 - phi) / p.eps
    dt = 0.3 * g.h * g.h / p.DF
    u = [dev(rng.uniform(-0.3, 0.3, s) * g.h / dt) for s in
         [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)][:g.ndim]]
    return g, p, dev(phi), dev(f), dev(F), dt, u + [None] * (3 - len(u))


# FP64: the Newton solve with its sweeps as tiles (2D) and colour by colour
# (3D); FP32: the solvers whose state may end in the second buffer, and a step
# that passes its first test, whose answer is the advected state itself
@pytest.mark.parametrize("geom,shape,prec,solver,tol", [
    (W.AXI, (1, 500, 301), 0, 1, 1e-10), (W.PLANAR, (1, 512, 500), 0, 1, 1e-10),
    (W.CART3D, (90, 96, 100), 0, 1, 1e-10), (W.CART3D, (90, 96, 100), 1, 0, 1e-6),
    (W.CART3D, (90, 96, 100), 1, 2, 1e-6), (W.CART3D, (90, 96, 100), 1, 1, 10.0)])
def test_state_is_final_on_return(geom, shape, prec, solver, tol):
    import paper_2605_27534_gb300 as sfx
    import torch
    g, p, phi, f0, F0, dt, u = _problem(geom, shape)
    if geom == W.PLANAR:
        u = [None] * 3
    opts = sfx.default_opts(tol=tol)
    ctx = sfx.Context.for_grid(g, prec)
    if prec:
        u = [None if a is None else a.float() for a in u]
        f0, F0 = sfx.sfx_df_pack(f0), sfx.sfx_df_pack(F0)
        ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_SOLVER, solver)
        ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_PREDICT, 0)
        ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_FAST_RESID, 0)
    step, other = torch.cuda.Stream(), torch.cuda.Stream()

    def once(stats):
        f, F = f0.clone(), F0.clone()
        torch.cuda.synchronize()
        with torch.cuda.stream(step):
            ctx.sfx_surfactant_step(p, phi, f, F, dt, *u, opts=opts, stats=stats)
        with torch.cuda.stream(other):
            got = f.clone(), F.clone()
        torch.cuda.synchronize()
        return got

    want = once(True)
    for _ in range(20):
        got = once(False)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
