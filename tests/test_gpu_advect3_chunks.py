"""The 3D FP32 advection takes 16, 8 or 4 planes per block by the size of the
grid: grids on either side of those lines, chunks with a remainder, tiles with
one column or row, against the gathering tiles (the same bits)."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (31, 7, 5), (33, 8, 19), (64, 64, 64), (40, 33, 50),
                                      (100, 50, 70), (95, 64, 85), (100, 90, 120), (32, 15, 3)])
def test_staged_advection_is_the_gathered_one(nx, ny, nz):
    import paper_2605_27534_gb300 as sfx
    rng = np.random.default_rng(nx + ny + nz)
    g = W.Grid(W.CART3D, nx, ny, nz, 1.0 / max(nx, ny, nz))
    p = W.Params(ka=1.0, kd=0.1, Df=1e-4, DF=1e-4, eps=0.75 * g.h, bc_F=0.7, bc_f=0.1)
    shape = (nz, ny, nx)
    phi, f, F = rng.uniform(0.2, 0.8, shape), rng.uniform(0, 1, shape), rng.uniform(0, 1, shape)
    u = [rng.standard_normal((nz + (d == 2), ny + (d == 1), nx + (d == 0))) for d in range(3)]
    for a in u:
        a[rng.uniform(0, 1, a.shape) < 0.1] = 0.0
    out = []
    for staged in (1, 0):
        ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
        ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_ADVECT_STAGED, staged)
        fd, Fd = sfx.sfx_df_pack(dev(f)), sfx.sfx_df_pack(dev(F))
        ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, 0.02 * g.h, *[dev(a).float() for a in u],
                                allow_not_converged=True)
        out.append((host(fd), host(Fd)))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
