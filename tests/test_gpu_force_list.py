"""The Marangoni force takes its interface cells from a list: fields with none,
few and only interface cells, fractions at the thresholds of the interface
and of the plane offset (near 0, 1/2 and 1), and tiny and ragged grids,
against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


def _fraction(shape, kind):
    rng = np.random.default_rng(8)
    if kind == "none":
        return np.ones(shape)
    if kind == "all":
        return rng.uniform(0.01, 0.99, shape)
    C = (rng.uniform(size=shape) < 0.5).astype(float)
    edge = rng.uniform(size=shape) < 0.4
    C[edge] = rng.choice([0.0, 1e-7, 2e-6, 1e-4, 0.4999999, 0.5, 0.5000001, 1 - 1e-4, 1 - 2e-6,
                          1 - 1e-7, 1.0], edge.sum())
    return C


@pytest.mark.parametrize("kind", ["none", "all", "edges"])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 1, 1)), (W.PLANAR, (1, 37, 70)),
                                        (W.AXI, (1, 33, 31)), (W.CART3D, (9, 14, 35)),
                                        (W.CART3D, (8, 16, 64))])
@pytest.mark.parametrize("dm_mode", [0, 1])
def test_force_from_the_list_against_the_oracle(sfx, geom, shape, kind, dm_mode):
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    rng = np.random.default_rng(2)
    p = W.Params(eps=0.75 * g.h)
    phi = rng.uniform(0.02, 0.98, shape)
    f = 0.4 * rng.uniform(0, 1, shape) * phi * (1 - phi) / p.eps
    C = _fraction(shape, kind)
    n = (g.ndim,) + shape
    # every factor is good to a few ulp; sigma differences lose up to
    # sigma0/|sigma - sigma0| (50 here) of it
    s_o, F_o = oracle.marangoni(g, p, f, phi, C, dm_mode)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    s, F = dev(np.full(shape, np.nan)), dev(np.full(n, np.nan))
    ctx.sfx_marangoni_force(p, dev(f), dev(phi), dev(C), s, F, dm_mode)
    scale = max(np.abs(F_o).max(), 1e-300)
    assert np.abs(host(s) - s_o).max() < 1e-14
    # ... and the area of a nearly empty or full cell moves by dC/min(C, 1 - C)
    # of itself, dC the few ulp of 1 that either side's volume carries
    F_o = F_o.reshape(n)
    cond = 4e-16 / np.maximum(np.minimum(C, 1 - C), 1e-7)
    assert (np.abs(host(F) - F_o) <= 1e-12 * scale + cond * np.abs(F_o)).all()
    # float: C, its plane and the gradient rounded to float
    C32 = C.astype(np.float32)
    s_o, F_o = oracle.marangoni(g, p, f, phi, C32.astype(float), dm_mode)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
    s, F = dev(np.full(shape, np.nan), torch.float32), dev(np.full(n, np.nan), torch.float32)
    ctx.sfx_marangoni_force(p, ctx.sfx_df_pack(dev(f)), dev(phi), dev(C32), s, F, dm_mode)
    out = host(F)
    assert np.isfinite(out).all()
    if dm_mode:
        assert (out[:, (C32 <= 1e-6) | (C32 >= 1 - 1e-6)] == 0).all()
    if kind != "edges":     # there a float Youngs normal may cancel to nothing
        assert np.abs(out - F_o.reshape(n)).max() < 1e-4 * max(np.abs(F_o).max(), 1e-300)


def test_eos_of_large_float_grids_takes_the_band(sfx):
    """2^20 cells and more: the cells with Gamma = 0 and the band around the
    interface in two launches; an odd count of cells, Gamma up to and past
    saturation, phi at both ends of the threshold."""
    import torch
    g = W.Grid(W.PLANAR, 1031, 1025, 1, 1.0 / 1031)
    p = W.Params(eps=0.75 * g.h)
    rng = np.random.default_rng(6)
    phi = rng.choice([0.0, 1e-4, 5e-4, 9.9e-4, 1.01e-3, 0.1, 0.5, 0.9, 1 - 1.01e-3, 1 - 9.9e-4,
                      0.9995, 1.0], g.shape)
    f = rng.choice([0.0, 0.3, 0.499, 0.501, 0.9, 0.999999, 1.0, 1.3], g.shape) * phi * (1 - phi) / p.eps
    C = np.zeros(g.shape)
    want, _ = oracle.marangoni(g, p, f, phi, C, 1)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F32)
    s = dev(np.full(g.shape, np.nan), torch.float32)
    F = torch.empty((2,) + g.shape, device="cuda")
    ctx.sfx_marangoni_force(p, ctx.sfx_df_pack(dev(f)), dev(phi), dev(C, torch.float32), s, F)
    # the logarithm of 1 - x at x = 0.999999 from a pair of 48 bits: 1e-8;
    # sigma in float (values down to sigma0 (1 + E ln 1e-12) = -4.5)
    assert np.abs(host(s) - want).max() < 1e-6 and (host(F) == 0).all()
