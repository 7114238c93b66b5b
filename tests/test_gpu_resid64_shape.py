"""The FP64 residual takes cells in turn, in blocks of 128 or 256 threads by
the size of the grid: rows that are no multiple of a warp, fewer cells than a
block, and grids on either side of the line; the converged step does not
depend on it."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,nx,ny,nz", [(W.PLANAR, 1, 1, 1), (W.PLANAR, 5, 7, 1), (W.AXI, 33, 1, 1),
                                           (W.AXI, 129, 65, 1), (W.CART3D, 33, 5, 3),
                                           (W.PLANAR, 641, 487, 1), (W.CART3D, 65, 70, 70)])
def test_step_against_the_picard_solver(geom, nx, ny, nz):
    """Both solvers at tol 1e-12 (residuals relative to |b|, and the diagonal
    dominates by 1/dt): 1e-10."""
    import paper_2605_27534_gb300 as sfx
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(nx, ny, nz))
    h = g.h
    p = W.Params(ka=2.0, kd=0.3, Df=0.1 * h * h / 1e-3, DF=0.2 * h * h / 1e-3, eps=0.75 * h)
    rng = np.random.default_rng(nx + ny)
    z, y, x = np.meshgrid(*((np.arange(n) + 0.5) * h for n in (nz, ny, nx)), indexing="ij")
    chi = np.clip(0.3 - np.sqrt((x - 0.4) ** 2 + (y - 0.4) ** 2 + (z - 0.4) ** 2 * (nz > 1)), -9 * h, 9 * h)
    phi = 0.5 * (1 - np.tanh(chi / (2 * p.eps)))
    f = rng.uniform(0.1, 0.3, phi.shape) * phi * (1 - phi) / p.eps
    F = rng.uniform(0.8, 1.0, phi.shape)
    out = []
    for levels in (0, 1):              # naming the levels takes the Picard solver
        ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
        fd, Fd = dev(f), dev(F)
        o = sfx.default_opts(tol=1e-12, max_cycles=400)
        o.mg_levels = levels
        st = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, 1e-3, opts=o)
        assert st.converged
        out.append((host(fd), host(Fd)))
    assert rel_err(out[0][0], out[1][0]) < 1e-10 and rel_err(out[0][1], out[1][1]) < 1e-10
