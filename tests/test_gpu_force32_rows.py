"""FP32 forces around the grid size from which interface cells are listed:
every cell in rows below it, a list above, against the oracle; and the
launches a small grid takes."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,shape,launches", [
    (W.PLANAR, (1, 1023, 512), 2), (W.PLANAR, (1, 1024, 512), 3), (W.PLANAR, (1, 1025, 512), 3),
    (W.CART3D, (64, 64, 127), 2), (W.CART3D, (64, 64, 129), 3), (W.AXI, (1, 33, 31), 2)])
def test_forces_in_rows_and_listed(geom, shape, launches):
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    rng = np.random.default_rng(2)
    p = W.Params(eps=0.75 * g.h)
    phi = rng.uniform(0.02, 0.98, shape)
    f = 0.4 * rng.uniform(0, 1, shape) * phi * (1 - phi) / p.eps
    C = np.where(rng.uniform(size=shape) < 0.1, rng.uniform(0.01, 0.99, shape), 0.0).astype(np.float32)
    _, want = oracle.marangoni(g, p, f, phi, C.astype(float), 1)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
    F = dev(np.full((g.ndim,) + shape, np.nan), torch.float32)
    args = (p, ctx.sfx_df_pack(dev(f)), dev(phi), dev(C), None, F)
    ctx.sfx_marangoni_force(*args)
    ctx.sfx_profile(True)
    ctx.sfx_marangoni_force(*args)
    assert ctx.sfx_profile_read()["forces"][0] == launches
    # C, its plane and the gradient of sigma in float
    assert np.abs(host(F) - want.reshape(F.shape)).max() < 1e-4 * np.abs(want).max()
