"""The FP64 BCG step from marched tiles (30 cells by 6 or 14 and chunks of
planes) against the oracle: extents at, below and past the tile edges, flow
through every wall, still faces, flat and rough fields, double velocities
and (through the ACDI step) float ones."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu
# a face value is about ten roundings of values of order max|x|, and a cell
# adds 2d fluxes of Courant number below 1/2
TOL = 1e-14


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


def _faces(shape, geom, seed):
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    u = [rng.uniform(-1, 1, s) for s in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))]
    for a in u:
        a[rng.uniform(size=a.shape) < 0.1] = 0.0
    return u if geom == W.CART3D else u[:2] + [None]


@pytest.mark.parametrize("field", ["rough", "front", "flat"])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 1, 1)), (W.PLANAR, (1, 6, 30)),
                                        (W.PLANAR, (1, 13, 61)), (W.AXI, (1, 7, 31)),
                                        (W.AXI, (1, 29, 29)), (W.CART3D, (1, 1, 1)),
                                        (W.CART3D, (8, 14, 30)), (W.CART3D, (17, 29, 33)),
                                        (W.CART3D, (33, 15, 2))])
def test_advect_tiles_against_the_oracle(sfx, geom, shape, field):
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    rng = np.random.default_rng(1)
    x = {"rough": rng.uniform(-1, 1, shape), "flat": np.full(shape, 0.7),
         "front": (np.arange(nx)[None, None] > nx // 2) * np.ones(shape)}[field]
    u, dt = _faces(shape, geom, 2), 0.15 * g.h
    want = oracle.advect_bcg(g, *u, dt, x, -0.4)
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    out = torch.full(shape, np.nan, dtype=torch.float64, device="cuda")
    ctx.sfx_advect(*[None if a is None else dev(a) for a in u], dt, dev(x), -0.4, out)
    assert rel_err(host(out), want) < TOL
    # both fields of a step in one launch: with no kinetics, diffusion or
    # drift the step is its advection
    p = W.Params(ka=0.0, kd=0.0, Df=0.0, DF=0.0, eps=0.75 * g.h, bc_F=-0.4, bc_f=0.2)
    f, F = dev(x + 1.0), dev(x)
    ctx.sfx_surfactant_step(p, dev(np.full(shape, 0.5)), f, F, dt,
                            *[None if a is None else dev(a) for a in u],
                            opts=sfx.default_opts(tol=1e-14))
    assert rel_err(host(F), want) < 2 * TOL
    assert rel_err(host(f), oracle.advect_bcg(g, *u, dt, x + 1.0, 0.2)) < 2 * TOL
