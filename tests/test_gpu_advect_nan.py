"""BCG advection of fields and by velocities that are not finite, and of values
at the ends of the double range: as the definition (the oracle) has them."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu
GRIDS = [(W.PLANAR, (1, 37, 61)), (W.AXI, (1, 50, 33)), (W.CART3D, (9, 14, 35)), (W.CART3D, (30, 34, 40))]


def _problem(geom, shape):
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0)
    rng = np.random.default_rng(4)
    u = [rng.uniform(-0.3, 0.3, s) for s in [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)][:g.ndim]]
    return g, rng, u + [None] * (3 - len(u))


def _advect(g, u, x):
    import paper_2605_27534_gb300 as sfx
    out = dev(np.zeros(g.shape))
    sfx.Context.for_grid(g, sfx.SFX_F64).sfx_advect(*[None if a is None else dev(a) for a in u], 0.5,
                                                    dev(x), 0.7, out)
    with np.errstate(all="ignore"):
        return host(out), oracle.advect_bcg(g, *u, 0.5, x, 0.7)


@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("geom,shape", GRIDS)
def test_a_bad_velocity_in_a_uniform_field(geom, shape, value):
    """Its transverse terms, 0 times it, are not a number either."""
    g, rng, u = _problem(geom, shape)
    x = np.full(shape, 0.4)
    for d in range(g.ndim):
        u[d][tuple(n // 2 for n in shape)] = value
    got, want = _advect(g, u, x)
    assert np.isnan(want).sum() > 4 and (np.isfinite(got) == np.isfinite(want)).all()
