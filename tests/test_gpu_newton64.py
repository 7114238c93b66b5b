"""The coupled Newton solve of FP64 contexts: the three geometries at odd and
tiny extents against the oracle, and the calls it hands to the Picard
solver (too few iterations allowed, scales outside the FP32 correction's
range, a given number of multigrid levels, diffusion-dominated steps)."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu
# both sides solve to |r| <= TOL |b|; the inverse Jacobian is bounded by dt
# (its columns are dominated by 1/dt), so each is within dt TOL |b| of the
# solution, |b| the App. C right-hand side
PARITY, TOL = 1e-12, 1e-13


def _bound(g, p, phi, f, F, fs, Fs, dt):
    """10 TOL dt |b|/|x| of the worse field, at least PARITY."""
    c1 = p.ka / (phi + p.eta)
    bf = fs / dt + c1 * F * p.gamma_inf * phi * (1 - phi) / p.eps
    bF = Fs / dt + p.kd * f
    return PARITY * max(1.0, *(dt * np.abs(b).max() / np.abs(x).max() for b, x in ((bf, f), (bF, F))))


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


def _problem(geom, shape, literal=0, scale=1.0, dnum=0.3):
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    c = [0.45 * n * g.h for n in (nx, ny, nz)]
    r = np.sqrt((x - c[0]) ** 2 * (geom != W.AXI) + x ** 2 * (geom == W.AXI) + (y - c[1]) ** 2
                + (z - c[2]) ** 2 * (geom == W.CART3D))
    p = W.Params(ka=2.0 / scale, kd=0.7, gamma_inf=scale, Df=4e-3, DF=1e-2, eps=0.75 * g.h,
                 literal_upwind=literal)
    phi = 0.5 * (1 - np.tanh(np.clip(0.3 - r, -9 * g.h, 9 * g.h) / (2 * p.eps)))
    rng = np.random.default_rng(7)
    F = scale * (1 + 0.2 * rng.uniform(-1, 1, shape))
    f = 0.2 * scale * (1 + 0.3 * rng.uniform(-1, 1, shape)) * phi * (1 - phi) / p.eps
    return g, p, phi, f, F, dnum * g.h * g.h / p.DF


def _both(sfx, g, p, phi, f, F, dt, opts, tol=TOL, flow=False):
    u = [None] * 3
    if flow:
        rng = np.random.default_rng(9)
        nz, ny, nx = g.shape
        shapes = [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)]
        u = [rng.uniform(-0.3, 0.3, s) * g.h / dt for s in shapes]
        if g.geom != W.CART3D:
            u[2] = None
    fo, Fo, st = oracle.surfactant_step(g, p, phi, f, F, dt, tol, *u)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    fd, Fd = dev(f), dev(F)
    s = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, dt, *[None if v is None else dev(v) for v in u],
                                opts=opts)
    fs = f if not flow else oracle.advect_bcg(g, *u, dt, f, p.bc_f)
    Fs = F if not flow else oracle.advect_bcg(g, *u, dt, F, p.bc_F)
    return (s, rel_err(host(fd), fo), rel_err(host(Fd), Fo),
            _bound(g, p, phi, fo, Fo, fs, Fs, dt))


@pytest.mark.parametrize("literal", [0, 1])
@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 37, 61)), (W.PLANAR, (1, 1, 1)),
                                        (W.PLANAR, (1, 300, 3)), (W.AXI, (1, 50, 33)),
                                        (W.AXI, (1, 7, 259)), (W.CART3D, (9, 14, 35)),
                                        (W.CART3D, (1, 2, 3)), (W.CART3D, (6, 5, 258))])
def test_newton_against_the_oracle(sfx, geom, shape, flow, literal):
    q = _problem(geom, shape, literal)
    s, ef, eF, tol = _both(sfx, *q, sfx.default_opts(tol=TOL), flow=flow)
    assert s.converged and s.res_f <= TOL and s.res_F <= TOL
    assert ef < tol and eF < tol


@pytest.mark.parametrize("kw", [dict(nu1=1, nu2=0), dict(nu1=0, nu2=7), dict(mg_levels=1),
                                dict(mg_levels=2), dict(max_cycles=400, check_every=3)])
def test_options_reach_the_same_solution(sfx, kw):
    q = _problem(W.PLANAR, (1, 36, 60))
    s, ef, eF, tol = _both(sfx, *q, sfx.default_opts(tol=TOL, **kw))
    assert s.converged and ef < tol and eF < tol


@pytest.mark.parametrize("scale", [1e-40, 1e-21, 1e35])
def test_scales_outside_the_float_range(sfx, scale):
    q = _problem(W.PLANAR, (1, 24, 40), scale=scale)
    s, ef, eF, tol = _both(sfx, *q, sfx.default_opts(tol=TOL))
    assert s.converged and ef < tol and eF < tol


def test_diffusion_dominated_step_takes_the_multigrid(sfx):
    q = _problem(W.PLANAR, (1, 32, 32), dnum=6.0)
    s, ef, eF, tol = _both(sfx, *q, sfx.default_opts(tol=TOL))
    assert s.converged and ef < tol and eF < tol


def test_not_converged_reports_the_allowed_iterations(sfx):
    g, p, phi, f, F, dt = _problem(W.PLANAR, (1, 24, 40))
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    fd, Fd = dev(f), dev(F)
    s = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, dt, opts=sfx.default_opts(tol=1e-15, max_cycles=1),
                                allow_not_converged=True)
    assert not s.converged and s.picard == 1 and np.isfinite(host(fd)).all()
    bad = F.copy()
    bad[0, 3, 5] = np.nan
    with pytest.raises(sfx.SfxError) as e:
        ctx.sfx_surfactant_step(p, dev(phi), dev(f), dev(bad), dt)
    assert e.value.status == sfx._lib.SFX_ERR_NONFINITE
