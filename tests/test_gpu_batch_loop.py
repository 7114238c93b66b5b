"""The batched step decides about another iteration in its last instance: with
many instances of one block each, which finish together and converge after
different numbers of iterations, every repetition takes the same iterations
to the same state."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom", [W.PLANAR, W.AXI])
def test_the_loop_ends_when_every_instance_has_converged(geom):
    import paper_2605_27534_gb300 as sfx
    import torch
    rng = np.random.default_rng(11)
    n, inst, phi, f, F = 1500, [], [], [], []
    for k in range(n):
        nx, ny = (int(v) for v in rng.integers(2, 13, 2))
        h, dt = 1.0 / max(nx, ny), 1e-3
        D = 10 ** rng.uniform(-4, -0.3) * h * h / dt
        p = W.Params(ka=10 ** rng.uniform(-3, 3), kd=10 ** rng.uniform(-3, 2), Df=D, DF=D, eps=0.75 * h)
        inst.append((nx, ny, h, dt, p))
        a = 0.5 * (1 - np.tanh(np.linspace(-3, 3, ny)[:, None] + 0 * np.arange(nx)))
        phi.append(a.ravel())
        f.append((rng.uniform(0.1, 0.4, a.shape) * a * (1 - a) / p.eps).ravel())
        F.append(rng.uniform(0.4, 0.9, a.shape).ravel())
    B = sfx.Batch(inst, geom=sfx.SFX_AXISYM if geom == W.AXI else sfx.SFX_PLANAR2D)
    B.sfx_batch_set_schedule(128, 2, 60)
    phi, f0, F0 = dev(np.concatenate(phi)), *(sfx.sfx_df_pack(dev(np.concatenate(v))) for v in (f, F))
    fb, Fb = f0.clone(), F0.clone()
    want = None
    for _ in range(100):
        fb.copy_(f0), Fb.copy_(F0)
        B.sfx_batch_step(phi, fb, Fb, 1e-9)
        st = B.sfx_batch_stats()
        assert all(st["converged"])
        got = (st["iters"], fb.clone(), Fb.clone())
        want = want or got
        assert got[0] == want[0] and torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    assert len(set(want[0])) > 3
