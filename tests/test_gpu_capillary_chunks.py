"""The capillary kernel takes 16, 8 or 4 planes per block by the size of the
grid: grids on either side of those lines, chunks with a remainder and tiles of
one cell, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (33, 9, 5), (34, 8, 17), (64, 64, 18), (65, 72, 37),
                                      (96, 100, 33)])
@pytest.mark.parametrize("f64", [True, False])
def test_chunks_against_the_oracle(nx, ny, nz, f64):
    """Per cell, kappa sums six face terms of unit normals over h and the
    force is sigma kappa |grad C| n: some forty roundings of terms below
    6/h (and 18 sigma/h^2), 3e-16 or 1.2e-7 each; phi in [0.2, 0.8] with steps
    that are far from flat, so no normal is near its threshold."""
    import paper_2605_27534_gb300 as sfx
    import torch
    g = W.Grid(W.CART3D, nx, ny, nz, 1.0 / max(nx, ny, nz))
    rng = np.random.default_rng(nx + nz)
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    phi = 0.5 + 0.1 * np.sin(0.7 * x) * np.cos(0.5 * y) + 0.1 * np.cos(0.6 * z + 0.3 * x) + \
        rng.uniform(-0.05, 0.05, (nz, ny, nx))
    C = rng.uniform(0, 1, (nz, ny, nx))
    sigma = rng.uniform(0.5, 1, (nz, ny, nx))
    p = W.Params(ka=1.0, kd=0.1, Df=1e-2, DF=1e-2, eps=0.75 * g.h)
    dt = torch.float64 if f64 else torch.float32
    if not f64:
        C, sigma = C.astype(np.float32).astype(float), sigma.astype(np.float32).astype(float)
    kap_o, force_o = oracle.capillary(g, phi, C, sigma, p.eps)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64 if f64 else sfx.SFX_F32)
    force = torch.empty((3, nz, ny, nx), dtype=dt, device="cuda")
    kappa = torch.empty((nz, ny, nx), dtype=dt, device="cuda")
    ctx.sfx_capillary_force(p, dev(phi), dev(C, dt), dev(sigma, dt), force, kappa)
    u = 40 * (3e-16 if f64 else 1.2e-7) * (1 if f64 else 10)   # a float normal of nearly flat phi
    assert np.abs(host(kappa) - kap_o).max() <= u * 6 / g.h
    assert np.abs(host(force) - np.asarray(force_o).reshape(3, nz, ny, nx)).max() <= u * 18 / g.h ** 2
