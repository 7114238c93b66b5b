"""The gradient of a rollout does not depend on where its segments end, and a
graph that is kept gives it twice (the states of the last segment come from
the forward)."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_rollout_gradient_over_segment_lengths(precision):
    """Tolerance: six steps solved to 1e-12 and adjoint solves to 1e-13, with
    amplification of the order of the condition 1 + dt (k_a F + ...) ~ 10."""
    import paper_2605_27534_gb300 as sfx
    import torch
    n = 24
    g = W.Grid(W.PLANAR, n, n + 5, 1, 1.0 / n)
    p = W.Params(ka=2.0, kd=0.3, gamma_inf=1.0, Df=0.02, DF=0.05, eps=0.75 * g.h)
    y, x = np.meshgrid((np.arange(n + 5) + 0.5) * g.h, (np.arange(n) + 0.5) * g.h, indexing="ij")
    chi = 0.3 - np.hypot(x - 0.5, y - 0.6)
    phi = (0.5 * (1 - np.tanh(chi / (2 * p.eps))))[None]
    Cf = np.clip(chi / g.h + 0.5, 0, 1)[None]
    rng = np.random.default_rng(2)
    gam = 0.1 * (1 + 0.3 * rng.uniform(-1, 1, phi.shape))
    ctx = sfx.Context.for_grid(g, precision)
    ref = None
    for K in (20, 6, 4, 1):
        setup = sfx.RolloutSetup(context=ctx, params=p, phi=dev(phi), C=dev(Cf), F0=dev(1 - Cf),
                                 dt=1e-3, nsteps=6, K=K)
        theta = torch.tensor([p.ka, p.kd, p.Df, p.DF], dtype=torch.float64, requires_grad=True)
        g0 = dev(gam).requires_grad_(True)
        L = sfx.SurfactantRollout.apply(g0, theta, setup)
        a = torch.autograd.grad(L, (g0, theta), retain_graph=True)
        b = torch.autograd.grad(L, (g0, theta))
        with torch.no_grad():
            assert abs(sfx.SurfactantRollout.apply(g0, theta, setup).item() - L.item()) <= 1e-11 * L.item()
        got = [host(v) for v in a]
        assert all(rel_err(host(v), w) < 1e-10 for v, w in zip(b, got))
        if ref is None:
            ref = got
        assert all(rel_err(w, v) < 1e-10 for w, v in zip(got, ref)), K
    setup = sfx.RolloutSetup(context=ctx, params=p, phi=dev(phi), C=dev(Cf), F0=dev(1 - Cf),
                             dt=1e-3, nsteps=0)
    g0 = dev(gam).requires_grad_(True)
    theta = torch.tensor([p.ka, p.kd, p.Df, p.DF], dtype=torch.float64, requires_grad=True)
    sfx.SurfactantRollout.apply(g0, theta, setup).backward()
    assert bool(torch.isfinite(g0.grad).all()) and float(theta.grad.abs().max()) == 0.0
