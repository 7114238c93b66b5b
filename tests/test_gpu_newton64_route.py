"""Which solver takes an FP64 step, told by its counts: 2 (nu1 + nu2) sweeps per
Newton iteration, 2 vcycles V-cycles per Picard iteration."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev

pytestmark = pytest.mark.gpu
NEWTON, PICARD = "newton", "picard"
SHAPES = {W.PLANAR: (1, 37, 61), W.AXI: (1, 50, 33), W.CART3D: (9, 14, 35)}


def _route(geom, shape, flow=False, dnum=0.3, literal=0, **kw):
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(ka=2.0, kd=0.7, Df=4e-3, DF=1e-2, eps=0.75 * g.h, literal_upwind=literal)
    rng = np.random.default_rng(3)
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    phi = 0.5 * (1 - np.tanh(np.clip(0.3 - x - 0.2 * y - 0.1 * z, -9 * g.h, 9 * g.h) / (2 * p.eps)))
    F = 1 + 0.2 * rng.uniform(-1, 1, shape)
    f = 0.2 * (1 + 0.3 * rng.uniform(-1, 1, shape)) * phi * (1 - phi) / p.eps
    dt = dnum * g.h ** 2 / p.DF
    # a uniform flow along y: F* stays positive (where F* < 0 and phi is small
    # the Newton solve leaves the step to Picard)
    u = [dev((0.2 if d == 1 else 0.0) * g.h / dt * np.ones(s)) for d, s in enumerate(
        [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)][:g.ndim])] if flow else []
    o = sfx.default_opts(tol=1e-10, **kw)
    st = sfx.Context.for_grid(g, sfx.SFX_F64).sfx_surfactant_step(p, dev(phi), dev(f), dev(F), dt, *u, opts=o)
    assert st.converged
    if st.vcycles == 2 * st.picard * (o.nu1 + o.nu2):
        return NEWTON
    assert st.vcycles == 2 * st.picard * o.vcycles
    return PICARD


@pytest.mark.parametrize("literal", [0, 1])
@pytest.mark.parametrize("geom", sorted(SHAPES))
@pytest.mark.parametrize("flow", [False, True])
def test_default_options(geom, flow, literal):
    # planar steps with a flow stay with the Picard solver
    want = PICARD if flow and geom == W.PLANAR else NEWTON
    assert _route(geom, SHAPES[geom], flow, literal=literal) == want


# the extents of the residual's launch shapes (cells in turn, 128 or 256 threads)
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 300, 3)), (W.PLANAR, (1, 700, 650)),
                                        (W.AXI, (1, 7, 259)), (W.CART3D, (1, 2, 3)),
                                        (W.CART3D, (6, 5, 258)), (W.CART3D, (70, 65, 80))])
def test_extents(geom, shape):
    assert _route(geom, shape) == NEWTON


@pytest.mark.parametrize("kw,want", [(dict(nu1=1, nu2=1), NEWTON), (dict(nu1=0, nu2=7), NEWTON),
                                     (dict(mg_levels=1), PICARD), (dict(mg_levels=2), PICARD),
                                     (dict(dnum=0.99), NEWTON), (dict(dnum=1.01), PICARD)])
def test_options(kw, want):
    assert _route(W.PLANAR, (1, 36, 60), **kw) == want
