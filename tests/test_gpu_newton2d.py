"""The 2D FP32 Newton iteration whose residual pass chooses its kind and
tests convergence itself, against the oracle's step."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("geom", [W.PLANAR, W.AXI])
@pytest.mark.parametrize("nx,ny", [(1, 5), (33, 2), (64, 64), (257, 40), (300, 131)])
@pytest.mark.parametrize("fast", [0, 1, 2])
def test_2d_newton_reaches_the_oracle_state(sfx, geom, nx, ny, fast):
    """Three steps (the second from the predicted increment, the third with a
    new dt, which has no prediction) against the oracle's step from the same
    state.  The form's float coefficients (D, drifts, phi, exchange) are off
    by 2^-24 each in about eight terms of up to 0.3 of the state, which the
    implicit solve does not amplify: 4 x 8 x 0.3 x 2^-24 = 6e-7 of the state,
    and the solve's tolerance."""
    g = W.Grid(geom, nx, ny, 1, 1.0 / max(nx, ny))
    h = g.h
    p = W.Params(ka=1.0, kd=0.2, Df=0.2 * h * h / 2e-3, DF=0.3 * h * h / 2e-3, eps=0.75 * h)
    x, y = (np.arange(nx) + 0.5) * h, (np.arange(ny)[:, None] + 0.5) * h
    chi = 0.3 - np.hypot(x - 0.4, y - 0.45)
    phi = 0.5 * (1 - np.tanh(np.clip(chi, -9 * h, 9 * h) / (2 * p.eps)))
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
    ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_FAST_RESID, fast)
    f = ctx.sfx_df_pack(dev(0.2 * phi * (1 - phi) / p.eps))
    F = ctx.sfx_df_pack(dev(1.0 - 0.5 * phi))
    d = dev(phi)
    tol = 1e-10
    for dt in (2e-3, 2e-3, 1e-3):
        f0, F0 = host(ctx.sfx_df_unpack(f)), host(ctx.sfx_df_unpack(F))
        st = ctx.sfx_surfactant_step(p, d, f, F, dt, opts=sfx.default_opts(tol=tol, max_cycles=60))
        assert st.converged and st.res_f <= tol and st.res_F <= tol
        f1, F1 = host(ctx.sfx_df_unpack(f)), host(ctx.sfx_df_unpack(F))
        ref = oracle.surfactant_step(g, p, phi, f0, F0, dt, 1e-13)
        for got, want in ((f1, ref[0]), (F1, ref[1])):
            assert np.abs(got - want).max() <= (1e-6 + 10 * tol) * np.abs(want).max()
