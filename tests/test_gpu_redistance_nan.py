"""A fraction that is NaN stays in its cell: its neighbours step as if it lay
past a wall, as the maxima of the definition do with a NaN."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _definition(C, h, iters, dtau):
    """Redistancing as defined, every cell stepped; fmax and fmin drop NaN."""
    def nb(a, ax, s):
        p = np.pad(a, [(1, 1) if d == ax else (0, 0) for d in range(3)], mode="edge")
        return np.take(p, np.arange(a.shape[ax]) + 1 + s, axis=ax)

    axes = [d for d in range(3) if C.shape[d] > 1]
    s0 = 2 * h * (C - 0.5)
    sg = np.where(s0 > 0, 1.0, np.where(s0 < 0, -1.0, 0.0))
    cut, dsum = np.zeros(C.shape, bool), np.zeros(C.shape)
    for d in axes:
        m, p = nb(s0, d, -1), nb(s0, d, 1)
        cut |= (s0 * m < 0) | (s0 * p < 0)
        q = np.fmax(np.fmax(np.abs(p - m) / 2, np.abs(p - s0)), np.abs(s0 - m))
        dsum += q * q
    dist = h * s0 / np.fmax(np.sqrt(dsum), 1e-300)
    x = s0.copy()
    for _ in range(iters):
        g = np.zeros(C.shape)
        for d in axes:
            b, f = (x - nb(x, d, -1)) / h * sg, (nb(x, d, 1) - x) / h * sg
            g += np.fmax(np.fmax(b, 0) ** 2, np.fmin(f, 0) ** 2)
        x = np.where(cut, x - dtau / h * (sg * np.abs(x) - dist), x - dtau * sg * (np.sqrt(g) - 1))
    return x


@pytest.mark.parametrize("shape", [(12, 20, 50), (1, 40, 70)])
@pytest.mark.parametrize("payload", [0x7ff8000000000000, 0xfff8000000000001])
def test_a_nan_fraction_stays_in_its_cell(shape, payload):
    """1e-12 h: 24 steps of some ten roundings of values below 24 h."""
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0 / nx)
    z, y, x = np.meshgrid(*(np.arange(n) + 0.5 for n in shape), indexing="ij")
    r = np.sqrt((x - 25) ** 2 + (y - 11) ** 2 + (z - 6) ** 2 * (nz > 1))
    C = np.clip(6.2 - r + 0.5, 0, 1)
    bad = np.array([payload], dtype=np.uint64).view(np.float64)[0]
    for at in ((nz // 2, 11, 25), (nz // 2, 11, 35), (nz - 1, 3, 0), (0, ny - 1, nx - 1)):
        C[at] = bad
    dtau = W.redist_dtau(g)
    with np.errstate(all="ignore"):
        want = _definition(C, g.h, 24, dtau)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    Cd = dev(C)
    chi, phi = torch.empty_like(Cd), torch.empty_like(Cd)
    ctx.sfx_phase_field_build(Cd, chi, phi, None, iters=24, dtau=dtau, eps=0.75 * g.h)
    got = host(chi)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.isnan(got).sum() == 4
    ok = ~np.isnan(want)
    assert np.abs(got[ok] - want[ok]).max() < 1e-12 * g.h * 24
