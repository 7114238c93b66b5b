"""Grids with more rows than a launch has blocks in y, of few cells each: the
advection and the drift faces take them as any other."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


def _column(nx, ny):
    rng = np.random.default_rng(6)
    g = W.Grid(W.PLANAR, nx, ny, 1, 1.0)
    y = np.arange(ny)[:, None] + 0 * np.arange(nx)
    phi = (0.5 * (1 - np.tanh(np.clip(30.0 - (y % 100), -9, 9) / 1.5)))[None]
    return g, phi, rng.uniform(0.5, 1, phi.shape), rng.uniform(0.5, 1, phi.shape), rng


def test_advection_of_a_tall_grid():
    import paper_2605_27534_gb300 as sfx
    import torch
    g, _, x, _, rng = _column(2, 393300)
    u = [rng.uniform(-0.3, 0.3, s) for s in ((1, g.ny, g.nx + 1), (1, g.ny + 1, g.nx))]
    want = oracle.advect_bcg(g, *u, None, 1.0, x, 0.7)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    out = dev(np.zeros(g.shape))
    ctx.sfx_advect(dev(u[0]), dev(u[1]), None, 1.0, dev(x), 0.7, out)
    assert rel_err(host(out), want) < 1e-14


def test_adjoint_operator_of_a_tall_grid():
    """Against the operator on its first and last 4000 rows (a row depends on
    four rows around it)."""
    import paper_2605_27534_gb300 as sfx
    g, phi, f, F, rng = _column(1, 262200)
    p = W.Params(ka=0.2, kd=0.1, Df=0.1, DF=0.2, eps=0.75)
    v = rng.uniform(-1, 1, g.shape), rng.uniform(-1, 1, g.shape)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    got = ctx.sfx_adjoint_apply(p, dev(phi), dev(f), dev(F), 0.5, dev(v[0]), dev(v[1]))
    n = 4000
    small = sfx.Context.for_grid(W.Grid(W.PLANAR, 1, n, 1, 1.0), sfx.SFX_F64)
    for rows, inner in ((slice(0, n), slice(0, n - 4)), (slice(g.ny - n, g.ny), slice(4, n))):
        cut = [dev(a[:, rows]) for a in (phi, f, F, *v)]
        want = small.sfx_adjoint_apply(p, cut[0], cut[1], cut[2], 0.5, cut[3], cut[4])
        for a, b in zip(got, want):
            assert (host(a)[:, rows][:, inner] == host(b)[:, inner]).all()


def test_fp32_picard_sweeps_of_a_tall_grid():
    """The solver of nonlinear sweeps (tiles of 16 rows) takes more rows than
    the drift faces' blocks of four: rows repeat, so do their results."""
    import paper_2605_27534_gb300 as sfx
    nx, ny = 1, 262300
    g, phi, _, _, _ = _column(nx, ny)
    p = W.Params(ka=0.2, kd=0.1, Df=0.1, DF=0.2, eps=0.75)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
    ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_SOLVER, 0)
    f, F = (sfx.sfx_df_pack(dev(a)) for a in (0.1 * phi, 1 + 0 * phi))
    st = ctx.sfx_surfactant_step(p, dev(phi), f, F, 0.5, opts=sfx.default_opts(tol=1e-6))
    assert st.converged
    F = host(sfx.sfx_df_unpack(F)).reshape(-1)
    assert abs(F[262235] - F[35]) < 1e-5 and abs(F[35] - 1) > 1e-4
