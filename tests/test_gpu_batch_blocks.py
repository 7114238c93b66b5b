"""The batched step's block tables, cells per thread and advection tiles:
instances of uneven sizes against single-grid steps, bit for bit."""
import numpy as np
import pytest

import workloads as W
from gpu_util import dev

pytestmark = pytest.mark.gpu

SMALL = [(1, 1), (2, 300), (31, 9), (32, 8), (33, 7), (62, 17), (257, 3)]
LARGE = SMALL + [(300, 700), (64, 4000), (31, 3000), (255, 600), (128, 1500)]   # 8 cells per thread
MIDDLE = SMALL + [(200, 800), (63, 1200)]                                       # 2


@pytest.fixture(scope="module")
def sfx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2605_27534_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("geom", [W.PLANAR, W.AXI])
@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("sizes,block", [(SMALL, 256), (MIDDLE, 128), (LARGE, 256), (LARGE, 512)])
@pytest.mark.parametrize("fast", [0, 2])
def test_uneven_batch_bitwise_equals_single_grid_steps(sfx, geom, flow, sizes, block, fast):
    """One converging step; the last instance is uniform, at rest and far from
    any interface: it converges at its first pair residual."""
    import torch
    rng = np.random.default_rng(3)
    inst, phi, f, F, ur, uz = [], [], [], [], [], []
    for k, (nx, ny) in enumerate(sizes + [(40, 50)]):
        rest = k == len(sizes)
        h, dt = 1.0 / max(nx, ny), 1e-3
        p = W.Params(ka=2.0, kd=0.2, Df=0.1 * h * h / dt, DF=0.2 * h * h / dt, eps=0.75 * h,
                     bc_F=0.7)
        inst.append((nx, ny, h, dt, p))
        x, y = (np.arange(nx) + 0.5) * h, (np.arange(ny)[:, None] + 0.5) * h
        a = 0.5 * (1 - np.tanh(np.clip(0.3 - np.hypot(x - 0.4, y - 0.5), -9 * h, 9 * h) / (1.5 * h)))
        phi.append(np.zeros((ny, nx)) if rest else a)
        f.append(0.0 * a if rest else rng.uniform(0.1, 0.4, a.shape) * a * (1 - a) / p.eps)
        F.append(np.full(a.shape, 0.7) if rest else rng.uniform(0.4, 0.9, a.shape))
        s = 0.0 if rest else 0.2 * h / dt
        ur.append(s * rng.uniform(-1, 1, (ny, nx + 1)))
        uz.append(s * rng.uniform(-1, 1, (ny + 1, nx)))
    cat = lambda v: np.concatenate([a.ravel() for a in v])
    B = sfx.Batch(inst, geom=sfx.SFX_AXISYM if geom == W.AXI else sfx.SFX_PLANAR2D)
    B.sfx_batch_set_schedule(block, 3, 40)
    B.sfx_batch_set_tuning(sfx._lib.SFX_TUNE_F32_FAST_RESID, fast)
    fb, Fb = sfx.sfx_df_pack(dev(cat(f))), sfx.sfx_df_pack(dev(cat(F)))
    u = (dev(cat(ur), torch.float32), dev(cat(uz), torch.float32)) if flow else (None, None)
    B.sfx_batch_step(dev(cat(phi)), fb, Fb, 1e-10, ur=u[0], uz=u[1])
    st = B.sfx_batch_stats()
    assert all(st["converged"])
    if fast == 0:
        assert st["iters"][-1] == 1
    o = sfx.default_opts(tol=1e-10, max_cycles=40, nu1=3, nu2=0)
    off = 0
    for k, (nx, ny, h, dt, p) in enumerate(inst):
        ctx = sfx.Context.for_grid(W.Grid(geom, nx, ny, 1, h), sfx.SFX_F32)
        ctx.sfx_set_tuning(sfx._lib.SFX_TUNE_F32_FAST_RESID, fast)
        f1, F1 = sfx.sfx_df_pack(dev(f[k])), sfx.sfx_df_pack(dev(F[k]))
        v = [dev(ur[k], torch.float32), dev(uz[k], torch.float32), None] if flow else []
        s1 = ctx.sfx_surfactant_step(p, dev(phi[k]), f1, F1, dt, *v, opts=o)
        assert s1.picard == st["iters"][k], k
        n = nx * ny
        assert torch.equal(f1.reshape(-1), fb.reshape(-1)[2 * off:2 * (off + n)]), k
        assert torch.equal(F1.reshape(-1), Fb.reshape(-1)[2 * off:2 * (off + n)]), k
        V = (2 * np.arange(nx) + 1) * np.pi * h ** 3 if geom == W.AXI else h * h
        for m, q in ((st["mass_f"][k], f1), (st["mass_F"][k], F1)):
            w = V * q.cpu().numpy().astype(np.float64).reshape(ny, nx, 2).sum(-1)
            assert abs(m - w.sum()) <= 1e-12 * max(np.abs(w).sum(), 1e-300)
        off += n
