"""FP64 steps of fields that vanish in float: solved as any other (the system is
linear without adsorption, so the scale drops out)."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fields", ["both", "f", "F"])
@pytest.mark.parametrize("scale", [1e-60, 1e-200])
@pytest.mark.parametrize("geom,shape", [(W.PLANAR, (1, 20, 33)), (W.CART3D, (9, 14, 35))])
def test_scale_drops_out(geom, shape, scale, fields):
    import paper_2605_27534_gb300 as sfx
    g = W.Grid(geom, shape[2], shape[1], shape[0], 1.0 / max(shape))
    p = W.Params(ka=0.0, kd=0.0, Df=1e-2, DF=2e-2, eps=0.75 * g.h)
    rng = np.random.default_rng(3)
    x, y, z = W.cell_centre_offsets(shape, g.h, (0, 0, 0))
    phi = 0.5 * (1 - np.tanh((0.3 - x - 0.2 * y - 0.1 * z) / (2 * p.eps)))
    f, F = rng.uniform(0.5, 1, shape), rng.uniform(0.5, 1, shape)
    dt = 0.2 * g.h ** 2 / p.DF
    out = []
    for s in (1.0, scale):
        ctx = sfx.Context.for_grid(g, sfx.SFX_F64)
        fd = dev(f * (s if fields in ("both", "f") else 1.0))
        Fd = dev(F * (s if fields in ("both", "F") else 1.0))
        st = ctx.sfx_surfactant_step(p, dev(phi), fd, Fd, dt, opts=sfx.default_opts(tol=1e-13))
        assert st.converged
        out.append((host(fd), host(Fd)))
    (f1, F1), (f2, F2) = out
    # both solve to 1e-13 of x/dt
    assert rel_err(f2 / (scale if fields in ("both", "f") else 1.0), f1) < 1e-12
    assert rel_err(F2 / (scale if fields in ("both", "F") else 1.0), F1) < 1e-12
