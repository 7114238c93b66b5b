"""VoF advection over active blocks (grids of 2^20 cells and more) and over
every block (below), against the oracle: fluid at block edges and corners and
at walls moving into blocks that held none, empty and full domains."""
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


def _drops(shape, kind):
    C = np.zeros(shape)
    if kind == "full":
        return C + 1.0
    if kind == "empty":
        return C
    nz, ny, nx = shape
    z, y, x = np.meshgrid(*(np.arange(n) + 0.5 for n in shape), indexing="ij", sparse=True)
    three = nz > 1
    # a drop across a corner of blocks, one on a corner of the grid, and a
    # single cell of fluid in the last cell of a block
    for cx, cy, cz, r in ((64, 32, 8, 3.7), (0, 0, 0, 5.2), (nx - 1, ny - 2, nz - 1, 2.9)):
        d = np.sqrt((x - cx) ** 2 + (y - cy) ** 2 + three * (z - cz) ** 2)
        C = np.maximum(C, np.clip(r - d + 0.5, 0, 1))
    C[min(15, nz - 1), 47, 31 + 32] = 0.3
    return C


@pytest.mark.parametrize("kind", ["drops", "full", "empty"])
@pytest.mark.parametrize("shape", [(90, 96, 130), (1, 1030, 1025), (16, 60, 100), (1, 61, 99)])
def test_vof_blocks_against_the_oracle(sfx, shape, kind):
    nz, ny, nx = shape
    geom = W.CART3D if nz > 1 else W.PLANAR
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    C = _drops(shape, kind)
    rng = np.random.default_rng(4)
    dt = 0.1 * g.h
    faces = [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)][:g.ndim]
    u = [np.sign(rng.uniform(-1, 1)) * rng.uniform(0.5, 1, s) for s in faces]
    for d, a in enumerate(u):                    # closed walls
        ax = 2 - d
        a[(slice(None),) * ax + (0,)] = 0
        a[(slice(None),) * ax + (-1,)] = 0
    u += [None] * (3 - len(u))
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    ctx32 = sfx.Context.for_grid(g, sfx.SFX_F32)
    ud = [None if a is None else dev(a) for a in u]
    u32 = [None if a is None else a.float() for a in ud]
    Cd, C32 = dev(C), dev(C)
    for step in range(2):
        C = oracle.vof_advect(g, *u, dt, C, step)
        ctx.sfx_vof_advect(*ud, dt, Cd, step)
        ctx32.sfx_vof_advect(*u32, dt, C32, step)
        # plane offsets are found to 1e-16 by other iterations on each side,
        # and a flux moves by dV/dalpha <= 1/max(m) of that
        assert np.abs(host(Cd) - C).max() < 1e-12
        # float geometry: a few float roundings per flux
        assert np.abs(host(C32) - C).max() < 1e-5
