"""The 2D adjoint solve (table of weights, relaxation in tiles of 28 x 20
cells, ten half-sweeps per launch) at sizes around its tiles."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu
EPS = 2.3e-16


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("geom", [W.PLANAR, W.AXI])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 37), (45, 2), (28, 20), (29, 21), (57, 39), (133, 250)])
@pytest.mark.parametrize("sweeps", [1, 5, 6, 16])
def test_adjoint_2d_solves_the_transposed_system(sfx, geom, nx, ny, sweeps):
    """nu = dt lam0 satisfies (-J)^T nu = lam1 as sfx_adjoint_apply evaluates
    it, within the tolerance of the solve and the rounding of either form
    (10 products per field, each below |diagonal| |nu|), and the parameter
    terms are the sums of App. C with N^ f = (out(D) - out(2 D))/D."""
    rng = np.random.default_rng(nx + 7 * ny)
    g = W.Grid(geom, nx, ny, 1, 1.0 / max(nx, ny))
    h, dt = g.h, 2e-3
    p = W.Params(ka=2.0, kd=0.3, gamma_inf=1.0, Df=0.1 * h * h / dt, DF=0.2 * h * h / dt,
                 eps=0.75 * h, literal_upwind=sweeps == 6)
    x, y = (np.arange(nx) + 0.5) * h, (np.arange(ny)[:, None] + 0.5) * h
    chi = 0.3 - np.hypot(x - 0.4, y - 0.5)
    phi = 0.5 * (1 - np.tanh(np.clip(chi, -9 * h, 9 * h) / (2 * p.eps)))
    f = rng.uniform(0.1, 0.5, (ny, nx)) * phi * (1 - phi) / p.eps
    F = rng.uniform(0.5, 1.0, (ny, nx))
    lf, lF = rng.standard_normal((ny, nx)), rng.standard_normal((ny, nx))
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    d = [dev(a) for a in (phi, f, F)]
    a, b, dp = dev(lf), dev(lF), [0.0] * 4
    tol = 1e-12
    st = ctx.sfx_adjoint_step(p, *d, dt, a, b, dp,
                              sfx.default_opts(tol=tol, max_cycles=500, nu1=sweeps, nu2=0))
    assert st.converged
    nf, nF = dt * host(a), dt * host(b)
    big = max(np.abs(lf).max(), np.abs(lF).max())
    got = ctx.sfx_adjoint_apply(p, *d, dt, dev(nf), dev(nF), transpose=True)
    pe = phi + p.eta
    bh = (p.gamma_inf * phi * (1 - phi) / p.eps - f) / pe
    diag = 2 * (1 / dt + p.kd + p.ka * (F + np.abs(bh) * pe) / pe + 16 * (p.Df + p.DF) / h ** 2)
    vol = 4.0 if geom == W.AXI else 1.0      # neighbouring volumes differ by up to 3
    room = tol * big + 20 * EPS * vol * np.max(diag) * max(np.abs(nf).max(), np.abs(nF).max())
    assert np.abs(host(got[0]) - lf).max() <= room
    assert np.abs(host(got[1]) - lF).max() <= room

    zero = dev(np.zeros((ny, nx)))
    def unit(k, v):                          # N^ v of field k
        args = [dev(v), zero] if k == 0 else [zero, dev(v)]
        name, D = ("Df", p.Df) if k == 0 else ("DF", p.DF)
        o = []
        for m in (1, 2):
            q = W.Params(**dict(p.__dict__, **{name: m * D}))
            o.append(host(ctx.sfx_adjoint_apply(q, *d, dt, *args)[k]))
        return (o[0] - o[1]) / D, 20 * EPS * vol * diag * np.abs(v) / D
    Nf, ef = unit(0, f)
    NF, eF = unit(1, F)
    dv = nf - nF
    want = [(dv * F * bh).sum(), -(dv * f).sum(), (nf * Nf).sum(), (nF * NF).sum()]
    room = [20 * EPS * np.abs(dv * F * bh).sum(), 20 * EPS * np.abs(dv * f).sum(),
            (np.abs(nf) * np.max(ef)).sum(), (np.abs(nF) * np.max(eF)).sum()]
    slack = 20 * EPS * max(np.abs(nf).sum(), np.abs(nF).sum())   # nu = dt (nu/dt) rounds twice
    for k in range(4):
        assert abs(dp[k] - want[k]) <= room[k] + slack * (1 + np.abs([F * bh, f, Nf, NF][k]).max()), k
