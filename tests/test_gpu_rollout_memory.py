"""The backward of a rollout holds the states of one segment at a time."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_backward_memory(precision):
    import paper_2605_27534_gb300 as sfx
    import torch
    n, K = 512, 8
    g = W.Grid(W.PLANAR, n, n, 1, 1.0 / n)
    p = W.Params(ka=2.0, kd=0.3, gamma_inf=1.0, Df=1e-4, DF=1e-4, eps=0.75 * g.h)
    y, x = np.meshgrid((np.arange(n) + 0.5) * g.h, (np.arange(n) + 0.5) * g.h, indexing="ij")
    chi = 0.3 - np.hypot(x - 0.5, y - 0.5)
    phi = (0.5 * (1 - np.tanh(np.clip(chi, -9 * g.h, 9 * g.h) / (2 * p.eps))))[None]
    Cf = np.clip(chi / g.h + 0.5, 0, 1)[None]
    setup = sfx.RolloutSetup(context=sfx.Context.for_grid(g, precision), params=p, phi=dev(phi),
                             C=dev(Cf), F0=dev(1 - Cf), dt=1e-3, nsteps=3 * K, K=K)
    theta = torch.tensor([p.ka, p.kd, p.Df, p.DF], dtype=torch.float64, requires_grad=True)
    g0 = dev(0.1 * np.ones(phi.shape)).requires_grad_(True)
    pair = 2 * 8 * n * n                       # bytes of a state (f, F)
    before = torch.cuda.memory_allocated()
    L = sfx.SurfactantRollout.apply(g0, theta, setup)
    held = torch.cuda.memory_allocated() - before
    assert held <= (K + 3 + 1) * pair          # the last segment, three checkpoints
    torch.cuda.reset_peak_memory_stats()
    torch.autograd.grad(L, (g0, theta))
    # never more states than the forward left, besides the state in work, the
    # adjoint's and the doubles of the state it is at (six pairs at most)
    assert torch.cuda.max_memory_allocated() - before <= held + 6 * pair
