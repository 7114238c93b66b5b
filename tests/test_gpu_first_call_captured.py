"""The forces and the phase field of a new context can be captured into a
graph by their first call (they allocate nothing then) and give what an
ordinary call gives."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 40, 36)), (W.CART3D, (20, 24, 28)),
                                        (W.CART3D, (64, 64, 70))])
@pytest.mark.parametrize("prec", [0, 1])
def test_first_calls_within_a_capture(geom, shape, prec):
    import paper_2605_27534_gb300 as sfx
    import torch
    nz, ny, nx = shape
    g = W.Grid(geom, nx, ny, nz, 1.0 / max(shape))
    p = W.Params(ka=1.0, kd=0.1, Df=1e-2, DF=1e-2, eps=0.75 * g.h, sigma0=1.0, E=0.2)
    z, y, x = np.meshgrid(*((np.arange(n) + 0.5) for n in shape), indexing="ij")
    r = np.sqrt((x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2 * (nz > 1))
    C = dev(np.clip(0.3 * min(n for n in shape if n > 1) - r + 0.5, 0, 1))
    dt = torch.float32 if prec else torch.float64

    def calls(ctx):
        out = dict(chi=torch.empty_like(C), phi=torch.empty_like(C),
                   sigma=torch.zeros(shape, dtype=dt, device="cuda"),
                   force=torch.zeros((g.ndim,) + shape, dtype=dt, device="cuda"))
        f = torch.full(shape, 0.2, dtype=torch.float64, device="cuda")
        f, Cc = sfx.sfx_df_pack(f) if prec else f, C.to(dt)

        def run():
            ctx.sfx_phase_field_build(C, out["chi"], out["phi"], None, iters=24,
                                      dtau=W.redist_dtau(g), eps=p.eps)
            ctx.sfx_marangoni_force(p, f, out["phi"], Cc, out["sigma"], out["force"])
        return run, out, (f, Cc)

    run, want, keep = calls(sfx.Context.for_grid(g, prec))
    run()
    run2, got, keep2 = calls(sfx.Context.for_grid(g, prec))
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        run2()
    for _ in range(2):
        graph.replay()
    for k in want:
        a, b = host(got[k]), host(want[k])
        assert np.abs(a - b).max() <= 1e-12 * max(1.0, np.abs(b).max()) * (1 if prec == 0 else 1e6), k
