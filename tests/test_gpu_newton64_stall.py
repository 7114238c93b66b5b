"""FP64 steps that the Newton solve cannot take to the tolerance: it hands them
to the Picard solver once its residual has stalled, and takes what converges
slowly to its end."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


def _problem(geom, shape, dnum):
    g = W.Grid(geom, shape[2], shape[1], shape[0], 1.0 / max(shape))
    p = W.Params(ka=2.0, kd=0.7, Df=4e-3, DF=1e-2, eps=0.75 * g.h)
    rng = np.random.default_rng(3)
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    phi = 0.5 * (1 - np.tanh(np.clip(0.3 - x - 0.2 * y - 0.1 * z, -9 * g.h, 9 * g.h) / (2 * p.eps)))
    F = 1 + 0.2 * rng.uniform(-1, 1, shape)
    f = 0.2 * (1 + 0.3 * rng.uniform(-1, 1, shape)) * phi * (1 - phi) / p.eps
    return g, p, phi, f, F, dnum * g.h ** 2 / p.DF


@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 40, 60)), (W.AXI, (1, 40, 60)),
                                        (W.CART3D, (9, 14, 35))])
def test_a_tolerance_below_rounding(geom, shape):
    import paper_2605_27534_gb300 as sfx
    g, p, phi, f, F, dt = _problem(geom, shape, 0.3)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    ctx.sfx_profile(True)
    st = ctx.sfx_surfactant_step(p, dev(phi), dev(f), dev(F), dt,
                                 opts=sfx.default_opts(tol=1e-18, max_cycles=35), allow_not_converged=True)
    assert not st.converged and st.picard == 35
    # 35 of Picard's; Newton's falls a decade or more per iteration to 1e-16
    assert ctx.sfx_profile_read()["residual"][0] <= 35 + 22


@pytest.mark.parametrize("nu", [(1, 0), (1, 1), (4, 4)])
def test_slow_convergence_is_taken_to_its_end(nu):
    """One sweep per iteration near the largest diffusion number: the Newton
    solve still converges (its count of cycles is 2 (nu1 + nu2) an iteration)."""
    import paper_2605_27534_gb300 as sfx
    g, p, phi, f, F, dt = _problem(W.PLANAR, (1, 40, 60), 0.95)
    fo, Fo, _ = oracle.surfactant_step(g, p, phi, f, F, dt, 1e-13)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    fd, Fd = dev(f), dev(F)
    st = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, dt,
                                 opts=sfx.default_opts(tol=1e-12, nu1=nu[0], nu2=nu[1]))
    assert st.converged and st.vcycles == 2 * st.picard * sum(nu)
    assert rel_err(host(fd), fo) < 1e-11 and rel_err(host(Fd), Fo) < 1e-11
