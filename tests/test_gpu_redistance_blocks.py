"""The redistancing iterates only the blocks that the interface can reach:
grids with inactive blocks, ragged last blocks, interfaces at walls and at
block edges, uniform fields and step counts around the block extents,
against the oracle, which steps every cell."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


# chi and phi in units of h and 1: the two sides differ by roundings of the
# step (about 4 ulp each, a contraction), far below this
TOL = 1e-12


def _field(shape, kind):
    nz, ny, nx = shape
    z, y, x = np.meshgrid(*(np.arange(n) + 0.5 for n in shape), indexing="ij")
    if kind == "uniform":
        return np.full(shape, 0.3)
    if kind == "corner":          # cut by walls and by block edges
        r = np.sqrt((x - 32) ** 2 + y ** 2 + (z - 4) ** 2 * (nz > 1))
        return np.clip(9.0 - r + 0.5, 0, 1)
    if kind == "two":
        a = np.sqrt((x - 10) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2 * (nz > 1))
        b = np.sqrt((x - nx + 7) ** 2 + (y - 6) ** 2 + (z - nz + 5) ** 2 * (nz > 1))
        return np.clip(np.maximum(5.3 - a, 3.1 - b) + 0.5, 0, 1)
    return np.random.default_rng(3).uniform(0, 1, shape)


@pytest.mark.parametrize("kind", ["uniform", "corner", "two", "random"])
@pytest.mark.parametrize("geom,shape", [(W.CART3D, (9, 21, 131)), (W.CART3D, (40, 17, 33)),
                                        (W.PLANAR, (1, 70, 165)), (W.AXI, (1, 33, 31)),
                                        (W.PLANAR, (1, 1, 1))])
def test_redistance_blocks_against_the_oracle(sfx, geom, shape, kind):
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    C = _field(shape, kind)
    dtau, eps = W.redist_dtau(g), 0.75 * g.h
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    Cd = dev(C)
    for iters in (0, 1, 4, 24, 37):
        chi_o, phi_o, del_o = oracle.phase_field_build(g, C, iters, dtau, eps)
        chi, phi, dl = (torch.empty_like(Cd) for _ in range(3))
        ctx.sfx_phase_field_build(Cd, chi, phi, dl, iters=iters, dtau=dtau, eps=eps)
        assert rel_err(host(chi), chi_o) < TOL
        assert rel_err(host(phi), phi_o) < TOL
        # delta = phi (1 - phi)/eps moves by |1 - 2 phi|/eps times phi's error
        # (where phi is within 1e-8 of 1, one ulp of phi is 1e-8 of delta)
        assert np.abs(host(dl) - del_o).max() < TOL / eps
        assert np.array_equal(host(Cd), C)
        same = Cd.clone()               # chi in place of C
        ctx.sfx_phase_field_build(same, same, phi, None, iters=iters, dtau=dtau, eps=eps)
        assert np.array_equal(host(same), host(chi))
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)     # the float iterate
    ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_REDIST, 1)
    for iters in (0, 3, 24):
        chi_o, phi_o, _ = oracle.phase_field_build(g, C, iters, dtau, eps)
        ctx.sfx_phase_field_build(Cd, chi, phi, None, iters=iters, dtau=dtau, eps=eps)
        assert rel_err(host(chi), chi_o) < 1e-5
        same = Cd.clone()
        ctx.sfx_phase_field_build(same, same, phi, None, iters=iters, dtau=dtau, eps=eps)
        assert np.array_equal(host(same), host(chi))
