"""The FP64 advection of 3D grids takes 16 or 8 rows and a number of planes per
block by the size of the grid: grids that lead to either, chunks of one plane
and with a remainder, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (3, 2, 9), (31, 6, 5), (29, 15, 40), (40, 33, 50),
                                      (61, 70, 23), (64, 64, 64)])
@pytest.mark.parametrize("f64", [True, False])
def test_tilings_against_the_oracle(nx, ny, nz, f64):
    """Tolerance of the tiled advection: some fifty roundings of values of
    order 1."""
    import paper_2605_27534_gb300 as sfx
    import torch
    g = W.Grid(W.CART3D, nx, ny, nz, 1.0 / max(nx, ny, nz))
    rng = np.random.default_rng(nx + 3 * nz)
    xi = rng.uniform(0, 1, (nz, ny, nx))
    u = [rng.standard_normal((nz + (d == 2), ny + (d == 1), nx + (d == 0))) for d in range(3)]
    for a in u:
        a[rng.uniform(0, 1, a.shape) < 0.1] = 0.0
    if not f64:
        u = [a.astype(np.float32).astype(float) for a in u]
    dt = 0.1 * g.h
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64 if f64 else sfx.SFX_F32)
    ud = [dev(a, torch.float64 if f64 else torch.float32) for a in u]
    if f64:
        out = torch.empty((nz, ny, nx), dtype=torch.float64, device="cuda")
        ctx.sfx_advect(*ud, dt, dev(xi), 0.7, out)
        want = oracle.advect_bcg(g, *u, dt, xi, 0.7)
    else:            # float velocities: phi of an ACDI step, its regularisation off
        out = dev(xi)
        ctx.sfx_acdi_step(out, dt, 0.0, 0.75 * g.h, *ud)
        want = oracle.advect_bcg(g, *u, dt, xi, 1.0)
    assert rel_err(host(out), want) < 50 * 2.3e-16
