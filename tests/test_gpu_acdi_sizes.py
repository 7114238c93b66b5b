"""ACDI steps around the grid size from which cells are marked: every cell below
it, marked cells above, against the oracle; and the launches either takes."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu
# phi is of order 1 and moves by at most zeta dt/h (1/2 here) times a flux of
# about twenty roundings
TOL = 1e-14


@pytest.mark.parametrize("clip", [False, True])
@pytest.mark.parametrize("kind", ["noise", "circle", "wide"])
@pytest.mark.parametrize("geom,shape,launches", [
    (W.PLANAR, (1, 511, 256), 3), (W.PLANAR, (1, 512, 256), 5), (W.PLANAR, (1, 300, 450), 5),
    (W.AXI, (1, 513, 260), 5), (W.AXI, (1, 257, 131), 3), (W.CART3D, (50, 50, 52), 3),
    (W.CART3D, (52, 50, 53), 5)])
def test_every_cell_and_marked_cells(geom, shape, launches, kind, clip):
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    eps = 0.75 * g.h
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    r = np.sqrt((x - 0.4 * nx * g.h) ** 2 + (y - 0.5 * ny * g.h) ** 2 + (z - 0.5 * nz * g.h) ** 2)
    if kind == "noise":
        phi = np.random.default_rng(5).uniform(0, 1, shape)
    else:
        phi = 0.5 * (1 - np.tanh((0.25 * min(n for n in shape if n > 1) * g.h - r) /
                                 (2 * eps * (8 if kind == "wide" else 1))))
    dt = 0.4 * g.h * g.h / (2 * g.ndim * eps)
    want = oracle.acdi_step(g, phi, dt, 1.0, eps, clip=clip)
    for prec in (sfx.SFX_F64, sfx.SFX_F32):      # FP64 arithmetic in both
        ctx = sfx.Context.for_grid(g, prec)
        p = dev(phi)
        ctx.sfx_profile(True)
        ctx.sfx_acdi_step(p, dt, 1.0, eps, clip=clip)
        assert ctx.sfx_profile_read()["phase"][0] == launches
        assert rel_err(host(p), want) < TOL
