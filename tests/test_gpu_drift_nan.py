"""The FP64 face drifts at cells of phi that are not finite (their faces are not
a number) and at phi = -0."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


def _problem(geom, shape):
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(ka=0.0, kd=0.0, Df=1e-2, DF=2e-2, eps=0.75 * g.h)
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    phi = 0.5 * (1 - np.tanh((0.3 - x - 0.2 * y - 0.1 * z) / (2 * p.eps)))
    rng = np.random.default_rng(3)
    return g, p, phi, rng.uniform(0.5, 1, shape), rng.uniform(0.5, 1, shape), 0.2 * g.h ** 2 / p.DF


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 20, 33)), (W.AXI, (1, 20, 33)),
                                        (W.CART3D, (9, 14, 35))])
def test_faces_of_a_bad_cell_are_not_a_number(geom, shape, bad, prec):
    import paper_2605_27534_gb300 as sfx
    g, p, phi, f, F, dt = _problem(geom, shape)
    nz, ny, nx = shape
    k, j, i = nz // 2, ny // 2, nx // 2
    for at in ((k, j, i), (k, j, i + 2)):       # and between them a flat cell
        phi[at] = bad
    ctx = sfx.Context.for_grid(g, prec)
    out = ctx.sfx_adjoint_apply(p, dev(phi), dev(f), dev(F), dt, dev(f), dev(F))
    want = np.zeros(shape, bool)
    for a in (i, i + 2):
        want[k, j, a - 1:a + 2] = want[k, j - 1:j + 2, a] = True
        if nz > 1:
            want[k - 1:k + 2, j, a] = True
    for v in out:      # (next to an infinity the normal is inf/inf as well)
        got = np.isnan(host(v))
        assert got[want].all() and (np.isinf(bad) or (got == want).all())


@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 20, 33)), (W.CART3D, (9, 14, 35))])
def test_phi_of_minus_zero_has_no_normal(geom, shape):
    """phi (1 - phi) = -0 there: |grad phi| over it is below any threshold (as
    the oracle's normals and those of the forces have it)."""
    import paper_2605_27534_gb300 as sfx
    g, p, phi, f, F, dt = _problem(geom, shape)
    phi[:, ::3, ::2] = -0.0
    fo, Fo, _ = oracle.surfactant_step(g, p, phi, f, F, dt, 1e-13)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    fd, Fd = dev(f), dev(F)
    st = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, dt, opts=sfx.default_opts(tol=1e-13))
    # both solve to 1e-13 of a right-hand side that is x/dt here (no exchange)
    assert st.converged and rel_err(host(fd), fo) < 1e-12 and rel_err(host(Fd), Fo) < 1e-12
