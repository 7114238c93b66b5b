"""VoF advection of fields that hold a value that is not finite: the cells that
are not a number afterwards are those of the definition (the oracle's), on
grids below and above the size from which blocks are listed."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu
SHAPES = [(16, 60, 100), (1, 61, 99), (104, 100, 110), (1, 1030, 1025)]


def _run(shape, change, prec):
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0 / max(shape))
    z, y, x = np.meshgrid(*(np.arange(n) + 0.5 for n in shape), indexing="ij", sparse=True)
    r = np.sqrt((x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2 * (nz > 1))
    C = np.clip(0.3 * min(n for n in shape if n > 1) - r + 0.5, 0, 1)
    rng = np.random.default_rng(4)
    dt = 0.1 * g.h
    u = [np.sign(rng.uniform(-1, 1)) * rng.uniform(0.5, 1, s) for s in
         [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)][:g.ndim]]
    change(C, u)
    u3 = u + [None] * (3 - len(u))
    want = np.isnan(oracle.vof_advect(g, *u3, dt, C, 0))
    ctx = sfx.Context.for_grid(g, prec)
    real = torch.float32 if prec else torch.float64
    Cd = dev(C)
    ctx.sfx_vof_advect(*[None if a is None else dev(a, real) for a in u3], dt, Cd, 0)
    return np.isnan(host(Cd)), want


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("where", ["dry", "full"])
@pytest.mark.parametrize("shape", SHAPES)
def test_a_nan_fraction_counts_by_value(shape, where, prec):
    """Whatever its sign.  (Next to full cells it enters planes, whose offsets
    the oracle finds by another iteration.)"""
    nz, ny, nx = shape
    got = []
    for sign in (1, -1):
        def change(C, u):
            C[nz // 2, ny // 2, nx // 2 if where == "full" else 3] = np.copysign(np.nan, sign)
        g, want = _run(shape, change, prec)
        assert g.sum() > 1 and (where == "full" or (g == want).all())
        got.append(g)
    assert (got[0] == got[1]).all()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["dry", "wall"])
@pytest.mark.parametrize("shape", SHAPES)
def test_a_velocity_that_is_not_finite_reaches_empty_cells(shape, where, value, prec):
    """H (c_+ - c_-) is not a number with H = 0 either."""
    nz, ny, nx = shape

    def change(C, u):
        for d, a in enumerate(u):
            at = [nz // 3, 3, 2]
            if where == "wall":
                at[2 - d] = a.shape[2 - d] - 1
            a[tuple(at)] = value
    got, want = _run(shape, change, prec)
    assert want.sum() > 1 and (got == want).all()
