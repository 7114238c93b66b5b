"""The ACDI update evaluates each face of a block of cells once: faces at the
edges of blocks, of ragged last blocks and of the grid, next to cells that are
not marked, and values that are clipped or NaN."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,shape", [(W.CART3D, (4, 4, 32)), (W.CART3D, (5, 5, 33)),
                                        (W.CART3D, (9, 7, 65)), (W.CART3D, (1, 8, 31)),
                                        (W.PLANAR, (1, 16, 32)), (W.AXI, (1, 17, 33)),
                                        (W.AXI, (1, 32, 64)), (W.PLANAR, (1, 1, 40))])
@pytest.mark.parametrize("kind", ["noise", "patches"])
def test_faces_of_blocks_against_the_oracle(geom, shape, kind):
    """Tolerance: as the marked cells' test, phi moves by at most zeta dt/h
    times a flux of some twenty roundings."""
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    eps, zeta = 0.75 * g.h, 1.0
    rng = np.random.default_rng(nx + ny)
    phi = rng.uniform(0, 1, shape)
    if kind == "patches":      # marked cells among saturated ones
        phi = np.where(rng.uniform(0, 1, shape) < 0.15, phi, (phi > 0.5) * 1.0)
        phi[..., nx // 2:] = 1.0
    dt = 0.4 * g.h * g.h / (2 * g.ndim * zeta * eps)
    for clip in (False, True):
        want = oracle.acdi_step(g, phi, dt, zeta, eps, clip=clip)
        got = []
        for prec in (sfx.SFX_F64, sfx.SFX_F32):
            p = dev(phi)
            sfx.Context.for_grid(g, prec).sfx_acdi_step(p, dt, zeta, eps, clip=clip)
            got.append(host(p))
            assert rel_err(got[-1], want) < 1e-14
        if clip:
            assert all(v.min() >= 0 and v.max() <= 1 for v in got)
    # a NaN is clipped to 0 in its cell and its neighbours, as fmin(fmax(v, 0), 1)
    phi[nz // 2, ny // 2, nx // 2] = np.nan
    for prec in (sfx.SFX_F64, sfx.SFX_F32):
        p = dev(phi)
        sfx.Context.for_grid(g, prec).sfx_acdi_step(p, dt, zeta, eps, clip=True)
        v = host(p)
        assert v[nz // 2, ny // 2, nx // 2] == 0 and np.isfinite(v).all()
