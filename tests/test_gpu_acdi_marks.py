"""The ACDI step computes psi and its normal only near the interface: fields
whose |grad psi| lies on either side of the threshold of the normal, flat and
saturated fields, steep noise everywhere and tiny grids, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu
# phi is of order 1 and moves by at most zeta dt/h (1/2 here) times a flux of
# about twenty roundings
TOL = 1e-14


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


def _phi(shape, h, eps, kind, ndim):
    nz, ny, nx = shape
    z, y, x = np.meshgrid(*((np.arange(n) + 0.5) * h for n in shape), indexing="ij")
    if kind == "noise":
        return np.random.default_rng(5).uniform(0, 1, shape)
    if kind == "saturated":
        return (x > 0.5 * nx * h).astype(float)
    # psi = s x: |grad psi| = s, at and around the threshold 0.1
    s = {"below": 0.099, "at": 0.1, "above": 0.101, "wide": 0.35}[kind]
    r = np.exp(s * (x + 0.3 * y - 0.5 * nx * h) / eps)
    return r / (1 + r)


@pytest.mark.parametrize("clip", [False, True])
@pytest.mark.parametrize("kind", ["noise", "saturated", "below", "at", "above", "wide"])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 1, 1)), (W.PLANAR, (1, 19, 300)),
                                        (W.AXI, (1, 33, 17)), (W.CART3D, (7, 9, 35)),
                                        (W.CART3D, (1, 3, 2))])
@pytest.mark.parametrize("ratio", [0.75, 40.0])
def test_marked_cells_against_the_oracle(sfx, geom, shape, kind, clip, ratio):
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    eps = ratio * g.h
    phi = _phi(shape, g.h, eps, kind, g.ndim)
    zeta = 1.0
    dt = 0.4 * g.h * g.h / (2 * g.ndim * zeta * eps)
    want = oracle.acdi_step(g, phi, dt, zeta, eps, clip=clip)
    for prec in (sfx.SFX_F64, sfx.SFX_F32):      # FP64 arithmetic in both
        ctx = sfx.Context.for_grid(g, prec)
        p = dev(phi)
        ctx.sfx_acdi_step(p, dt, zeta, eps, clip=clip)
        assert rel_err(host(p), want) < TOL
