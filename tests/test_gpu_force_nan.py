"""A surface tension that is not finite reaches the FP64 force of its
neighbours, in cells without interface too: delta_m = 0 times a gradient that
is not finite is not a number."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dm_mode", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf])
@pytest.mark.parametrize("shape", [(9, 14, 35), (1, 20, 40), (1, 1, 1)])
def test_a_bad_sigma_shows_in_the_force(shape, bad, dm_mode):
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(eps=0.75 * g.h, eos=W.EOS_LINEAR)
    phi = np.full(shape, 0.5)
    f = np.full(shape, 0.1)
    at = (nz // 2, ny // 2, nx - 3 if nx > 3 else 0)
    f[at] = bad
    C = np.zeros(shape)
    C[:, :, :nx // 4] = 0.5 * (nx > 1)     # interface cells, far from the bad one
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    s, F = dev(np.zeros(shape)), dev(np.zeros((g.ndim,) + shape))
    ctx.sfx_marangoni_force(p, dev(f), dev(phi), dev(C), s, F, dm_mode)
    s, F = host(s), host(F)
    assert (~np.isfinite(s)).sum() == 1 and not np.isfinite(s[at])
    want = np.zeros(shape, bool)
    for ax, n in ((0, nz), (1, ny), (2, nx)):
        if ax == 0 and nz == 1:
            continue
        for d in (-1, 1):
            q = list(at)
            q[ax] = min(max(q[ax] + d, 0), n - 1)   # a wall cell stands in for its ghost
            want[tuple(q)] = True
    assert (np.isnan(F) == want).all()


@pytest.mark.parametrize("bad", [np.inf, -np.inf])
@pytest.mark.parametrize("shape", [(9, 14, 35), (1, 20, 40)])
def test_an_infinite_phi_shows_in_the_force(shape, bad):
    """The normal next to an infinite phi is not a number (inf/inf)."""
    import oracle
    import paper_2605_27534_gb300 as sfx
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(eps=0.75 * g.h, eos=W.EOS_LINEAR)
    rng = np.random.default_rng(1)
    phi, f = rng.uniform(0.3, 0.7, shape), rng.uniform(0.1, 0.2, shape)
    phi[nz // 2, ny // 2, nx - 3] = bad
    C = np.zeros(shape)
    C[:, :, :nx // 4] = 0.5
    _, want = oracle.marangoni(g, p, f, phi, C, 1)
    want = np.isnan(want.reshape((g.ndim,) + shape))
    assert want.any()
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    s, F = dev(np.zeros(shape)), dev(np.zeros((g.ndim,) + shape))
    ctx.sfx_marangoni_force(p, dev(f), dev(phi), dev(C), s, F, 1)
    assert (np.isnan(host(F)) == want).all()
