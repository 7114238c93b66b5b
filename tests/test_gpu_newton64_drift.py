"""FP64 steps whose drift velocities D/eps exceed half precision, in which the
Newton solve's sweeps hold them: no surfactant, a state that is steady away
from the interface, and an ordinary one, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["clean", "at rest", "general"])
@pytest.mark.parametrize("ratio", [5e4, 7e4, 4e6])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 20, 33)), (W.AXI, (1, 20, 33)),
                                        (W.CART3D, (8, 14, 35))])
def test_large_drifts(geom, shape, ratio, kind):
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    eps = 0.75 * g.h
    D = ratio * eps
    dt = 0.2 * g.h * g.h / D
    p = W.Params(ka=0.02 / dt, kd=0.01 / dt, Df=D, DF=0.3 * D, eps=eps)
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    phi = 0.5 * (1 - np.tanh(np.clip(0.3 - x - 0.2 * y - 0.1 * z, -9 * g.h, 9 * g.h) / (2 * eps)))
    rng = np.random.default_rng(3)
    F = 1 + 0.2 * rng.uniform(-1, 1, shape)
    f = 0.2 * (1 + 0.3 * rng.uniform(-1, 1, shape)) * phi * (1 - phi) / eps
    if kind == "clean":
        f, F = 0 * f, 0 * F
    if kind == "at rest":     # in one phase, without exchange
        phi, f, F = 0 * phi + 1, 0 * f, 0 * F + 0.7
        p.kd = 0.0
    fo, Fo, _ = oracle.surfactant_step(g, p, phi, f, F, dt, 1e-13)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    fd, Fd = dev(f), dev(F)
    st = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, dt, opts=sfx.default_opts(tol=1e-13))
    assert st.converged
    # both solve to 1e-13 of the right-hand side, which exceeds x/dt by the
    # exchange: ka dt F Gamma_inf delta is 2 % of f's scale here
    assert rel_err(host(fd), fo) < 1e-11 and rel_err(host(Fd), Fo) < 1e-11


@pytest.mark.parametrize("shape", [(1, 20, 33), (8, 14, 35)])
def test_a_correction_beyond_the_float_range_is_not_added(shape):
    """1/dt = 1e20: the products of the sweeps' 2x2 blocks overflow, and the
    first residual passes (desorption takes 1e-10 of f in the step)."""
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0)
    p = W.Params(ka=0.0, kd=1e10, Df=1.0, DF=1.0, eps=0.75)
    phi = np.full(shape, 0.5)
    f, F = np.full(shape, 1e9), np.full(shape, 2e9)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    fd, Fd = dev(f), dev(F)
    st = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, 1e-20, opts=sfx.default_opts(tol=1e-9))
    # the residual is 1e-10 of f/dt: so is the change it stands for
    assert st.converged and rel_err(host(fd), f) < 2e-10 and rel_err(host(Fd), F) < 2e-10
