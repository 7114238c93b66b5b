"""Different calls of one context on streams that are not ordered against each
other: each gives what it gives alone, bit for bit."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev

pytestmark = pytest.mark.gpu


# above 2^20 cells (block and face lists) and below
@pytest.mark.parametrize("geom,shape", [(W.CART3D, (104, 100, 110)), (W.PLANAR, (1, 1030, 1025)),
                                        (W.CART3D, (40, 44, 50))])
@pytest.mark.parametrize("prec", [0, 1])
def test_calls_of_one_context_overlap(geom, shape, prec):
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(eps=0.75 * g.h)
    z, y, x = np.meshgrid(*((np.arange(n) + 0.5) for n in shape), indexing="ij", sparse=True)
    r = np.sqrt((x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2 * (nz > 1))
    rng = np.random.default_rng(5)
    ball = np.clip(0.3 * min(n for n in shape if n > 1) - r + 0.5, 0, 1)
    speck = np.where(rng.uniform(size=shape) < 0.05, rng.uniform(0.1, 0.9, shape), 0.0)
    real = torch.float32 if prec else torch.float64
    u = [dev(rng.uniform(-0.3, 0.3, s), real) for s in
         [(nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)][:g.ndim]]
    u += [None] * (3 - len(u))
    phi = dev(rng.uniform(0.02, 0.98, shape))
    f = dev(0.4 * rng.uniform(0, 1, shape) * 0.2 / p.eps)
    f = sfx.sfx_df_pack(f) if prec else f
    fractions = [dev(np.maximum(ball, speck)), dev(speck)]
    Cf = fractions[1].to(real)
    ctx = sfx.Context.for_grid(g, prec)
    C = fractions[0].clone()
    force = torch.empty((g.ndim,) + shape, dtype=real, device="cuda")
    sigma = torch.empty(shape, dtype=real, device="cuda")
    chi, phi2 = torch.empty_like(phi), torch.empty_like(phi)

    def vof():
        C.copy_(fractions[0])
        ctx.sfx_vof_advect(*u, 0.5 * g.h, C)

    def marangoni():
        ctx.sfx_marangoni_force(p, f, phi, Cf, sigma, force)

    def phase():
        ctx.sfx_phase_field_build(fractions[0], chi, phi2, None, iters=24, eps=p.eps)

    calls = [vof, marangoni, phase]
    streams = [torch.cuda.Stream() for _ in calls]
    outs = [[C], [sigma, force], [chi, phi2]]
    for k in calls:
        k()
    torch.cuda.synchronize()
    want = [[t.clone() for t in o] for o in outs]
    torch.cuda.synchronize()
    for _ in range(20):
        for k, s in zip(calls, streams):
            with torch.cuda.stream(s):
                for _ in range(3):
                    k()
        torch.cuda.synchronize()
        for o, w in zip(outs, want):
            assert all(torch.equal(a, b) for a, b in zip(o, w))


@pytest.mark.parametrize("shape", [(40, 44, 50), (1, 300, 310)])
def test_fp64_forces_of_one_context_overlap(shape):
    """The FP64 force has no scratch: two of them, of different fractions."""
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(W.CART3D if nz > 1 else W.PLANAR, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(eps=0.75 * g.h)
    rng = np.random.default_rng(5)
    phi = dev(rng.uniform(0.02, 0.98, shape))
    f = dev(0.4 * rng.uniform(0, 1, shape) * 0.2 / p.eps)
    C = [dev(np.where(rng.uniform(size=shape) < w, rng.uniform(0.1, 0.9, shape), 0.0)) for w in (0.02, 0.4)]
    ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
    sigma = [torch.empty_like(phi) for _ in C]
    force = [torch.empty((g.ndim,) + shape, dtype=torch.float64, device="cuda") for _ in C]
    streams = [torch.cuda.Stream() for _ in C]

    def call(k):
        ctx.sfx_marangoni_force(p, f, phi, C[k], sigma[k], force[k])

    for k in (0, 1):
        call(k)
    torch.cuda.synchronize()
    want = [t.clone() for t in force]
    torch.cuda.synchronize()
    for _ in range(40):
        for _ in range(4):
            for k in (0, 1):
                with torch.cuda.stream(streams[k]):
                    call(k)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(force, want))
