"""The FP32 normal between two cells of phi that are not finite alike: their
difference is not a number, and the normal is zero (not that of the other
directions)."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("shape", [(7, 9, 12), (1, 9, 12)])
def test_no_normal_between_equal_bad_cells(shape, bad):
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0)
    phi = np.broadcast_to(0.3 + 0.02 * np.arange(ny)[:, None] + 0 * np.arange(nx), shape).copy()
    k, j, i = nz // 2, ny // 2, nx // 2
    phi[k, j, i - 1] = phi[k, j, i + 1] = bad
    C = np.broadcast_to(0.05 * np.arange(ny)[:, None] + 0 * np.arange(nx), shape).copy()
    p = W.Params(eps=0.75, eos=W.EOS_LINEAR)
    delta = phi * (1 - phi) / p.eps
    f = 0.1 * (1 + np.broadcast_to(np.arange(ny)[:, None] + 0 * np.arange(nx), shape)) * np.where(
        np.isfinite(delta), delta, 0.2)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
    F = torch.zeros((g.ndim,) + shape, device="cuda")
    ctx.sfx_marangoni_force(p, sfx.sfx_df_pack(dev(f)), dev(phi), dev(C, torch.float32), None, F, 0)
    # delta_m (I - n n) grad sigma: grad sigma is along y as the gradient of phi
    # is, so that the force vanishes with n = e_y (three cells on) and is
    # |grad C| times grad sigma = -sigma0 E 0.1/Gamma_inf with n = 0
    F = host(F)
    assert abs(F[1, k, j, i] + 0.05 * p.E * 0.1) < 1e-5 * 0.05 * p.E and abs(F[1, k, j, i + 3]) < 1e-8
