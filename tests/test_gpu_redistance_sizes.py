"""Redistancing around the number of blocks from which only active ones iterate:
every block below it, listed blocks above, against the oracle; and the launches
either takes."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu
# a few roundings per step (about 4 ulp each, a contraction), far below this
TOL = 1e-12


def _field(shape, kind):
    nz, ny, nx = shape
    z, y, x = np.meshgrid(*(np.arange(n) + 0.5 for n in shape), indexing="ij", sparse=True)
    if kind == "uniform":
        return np.full(shape, 0.3)
    r = np.sqrt((x - 32) ** 2 + y ** 2 + (z - 4) ** 2 * (nz > 1))     # cut by walls and block edges
    q = np.sqrt((x - nx + 7) ** 2 + (y - ny + 6) ** 2 + (z - nz + 5) ** 2 * (nz > 1))
    return np.clip(np.maximum(9.0 - r, 3.1 - q) + 0.5, 0, 1)


# three blocks of 512 cells resident on an SM (in quarters): 456 on 152 SMs
@pytest.mark.parametrize("kind", ["uniform", "drops"])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 304, 768)), (W.PLANAR, (1, 305, 769)),
                                        (W.AXI, (1, 400, 900)), (W.CART3D, (32, 31, 110)),
                                        (W.CART3D, (45, 42, 131))])
def test_every_block_and_listed_blocks(geom, shape, kind):
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    blocks = -(-nx // 32) * (-(-ny // 4) * -(-nz // 4) if nz > 1 else -(-ny // 16))
    every = blocks <= 3 * torch.cuda.get_device_properties(0).multi_processor_count
    C = _field(shape, kind)
    dtau, eps = W.redist_dtau(g), 0.75 * g.h
    Cd = dev(C)
    for f32 in (0, 1):
        ctx = sfx.Context.for_grid(g, f32)
        if f32:
            ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_REDIST, 1)
        for iters in (0, 3, 24):
            chi_o, phi_o, _ = oracle.phase_field_build(g, C, iters, dtau, eps)
            chi, phi = torch.empty_like(Cd), torch.empty_like(Cd)
            ctx.sfx_profile(True)
            ctx.sfx_phase_field_build(Cd, chi, phi, None, iters=iters, dtau=dtau, eps=eps)
            if nz > 1 or not f32:           # (2D FP32: eight steps per launch)
                assert ctx.sfx_profile_read()["phase"][0] == iters + 2 + (0 if every else g.ndim + 1)
            assert rel_err(host(chi), chi_o) < (1e-5 if f32 else TOL)
            if not f32:
                assert rel_err(host(phi), phi_o) < TOL
            same = Cd.clone()               # chi in place of C
            ctx.sfx_phase_field_build(same, same, phi, None, iters=iters, dtau=dtau, eps=eps)
            assert np.array_equal(host(same), host(chi))
