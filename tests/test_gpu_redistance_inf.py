"""Redistancing next to an infinite fraction: its neighbours across the
interface have the sub-cell distance 0 and relax towards it as defined."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f32", [0, 1])
@pytest.mark.parametrize("bad", [np.inf, -np.inf])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 37, 61)), (W.AXI, (1, 50, 33)),
                                        (W.CART3D, (9, 14, 35))])
def test_an_infinite_fraction(geom, shape, bad, f32):
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    z, y, x = np.meshgrid(*(np.arange(n) + 0.5 for n in shape), indexing="ij", sparse=True)
    C = np.clip(nx / 3.0 - x + 0.2 * np.sin(y) + 0.1 * np.cos(z) + 0.5, 0, 1)
    C[nz // 2, ny // 2, nx // 3] = bad
    eps, dtau = 0.75 * g.h, 0.3 * g.h
    with np.errstate(invalid="ignore"):
        chi_o, phi_o, _ = oracle.phase_field_build(g, C, 9, dtau, eps)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32 if f32 else sfx.SFX_F64)
    if f32:
        ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_REDIST, 1)
    chi, phi = dev(np.zeros(shape)), dev(np.zeros(shape))
    ctx.sfx_phase_field_build(dev(C), chi, phi, None, iters=9, dtau=dtau, eps=eps)
    chi, phi = host(chi), host(phi)
    ok = np.isfinite(chi_o)
    assert (~ok).any() and (np.isfinite(chi) == ok).all()
    # nine steps of a few roundings each, on distances up to some 10 h
    tol = 9 * 10 * g.h * (1e-6 if f32 else 1e-15)
    assert np.abs(chi - chi_o)[ok].max() < tol
    assert np.abs(phi - phi_o)[ok].max() < tol / (4 * eps) + 1e-15
