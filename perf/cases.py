"""The work that the performance of this framework is judged on.

Each case is one pass through the public entry points, as a program that
marches a soluble surfactant in time calls them: the coupled step on planar,
axisymmetric and 3D blocks in both precisions, the batched step, the gradient
of a rollout, and the interface work around the step (VoF advection, phase
field, ACDI, forces).  Sizes and physics follow the repository's workloads
(128^2 adsorption, 256^2 gradient, 512^2 vortex, 256^3 Hadamard-Rybczynski
bubble, 64 axisymmetric instances, 512 flat-interface columns).

A pass is one time step: the state moves on in place from pass to pass, as in
a user's time loop.  `exact` evaluates the same formulas in 64-bit torch.
"""
import math

import numpy as np
import torch

import paper_2605_27534_gb300 as sfx

PLANAR, AXI, CART = sfx.SFX_PLANAR2D, sfx.SFX_AXISYM, sfx.SFX_CART3D
TOL = 1e-10


def listed():
    return [
        # the smallest call: 2D no-flow adsorption in FP64, default options
        dict(name="step_planar_128_f64", kind="step", geom=PLANAR, nx=128, ny=128, nz=1, f64=True,
             flow=False, tuned=False),
        # a single rising bubble on an axisymmetric block of odd size, FP64
        dict(name="step_axi_131x257_f64", kind="step", geom=AXI, nx=131, ny=257, nz=1, f64=True,
             flow=True, tuned=False),
        # a 3D bubble in FP64 (the reference precision of a resolution study)
        dict(name="step_3d_96_f64", kind="step", geom=CART, nx=96, ny=96, nz=96, f64=True,
             flow=True, tuned=False),
        # the largest: the 256^3 bubble, FP32 form, static interface, the tuned schedule
        dict(name="step_3d_256_f32", kind="step", geom=CART, nx=256, ny=256, nz=256, f64=False,
             flow=True, tuned=True),
        # a 3D block of odd, ragged size, FP32 form, default options
        dict(name="step_3d_ragged_f32", kind="step", geom=CART, nx=157, ny=131, nz=117, f64=False,
             flow=True, tuned=False),
        # a whole moving-interface step: VoF, phase field, coupled step, Marangoni force
        dict(name="moving_2d_512_f32", kind="moving", nx=512, ny=512),
        # a parameter study: many axisymmetric instances in one batch
        dict(name="batch_axi_64", kind="batch", geom=AXI, instances=64, nr=256, pattern=3),
        # the flat-interface kinetics sweep: many small planar columns
        dict(name="batch_columns_512", kind="batch", geom=PLANAR, instances=512, nr=8, pattern=256),
        # the gradient workload: forward steps, loss and discrete adjoint
        dict(name="rollout_256", kind="rollout", nx=256, ny=256, steps=8, f64=False),
        # geometric VoF advection of a 3D bubble
        dict(name="vof_3d_256_f32", kind="vof", nx=256, ny=256, nz=256),
        # the 3D phase field of a new interface (FP64 redistancing)
        dict(name="phase_3d_192", kind="phase", nx=192, ny=192, nz=192, f64=True),
        # phase-field transport and both interface forces in 3D
        dict(name="interface_3d_160_f32", kind="interface", nx=160, ny=160, nz=160, f64=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "moving", "batch", "rollout", "vof", "phase",
                       "interface"])
    f64 = rng.random() < 0.5
    if kind == "step":
        geom = rng.choice([PLANAR, AXI, CART, CART])
        if geom == CART:
            lo, hi = (24, 96) if f64 else (32, 232)
            n = [_log(rng, lo, hi) for _ in range(3)]
        else:
            n = [_log(rng, 48, 320), _log(rng, 48, 512), 1]
        return dict(kind=kind, geom=geom, nx=n[0], ny=n[1], nz=n[2], f64=f64,
                    flow=geom != PLANAR or rng.random() < 0.5, tuned=not f64 and rng.random() < 0.5)
    if kind == "moving":
        return dict(kind=kind, nx=_log(rng, 64, 640), ny=_log(rng, 64, 640))
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind=kind, geom=AXI, instances=_log(rng, 4, 64), nr=_log(rng, 48, 256),
                        pattern=rng.randrange(1000))
        return dict(kind=kind, geom=PLANAR, instances=_log(rng, 16, 512), nr=rng.randrange(4, 17),
                    pattern=_log(rng, 64, 320))
    if kind == "rollout":
        return dict(kind=kind, nx=_log(rng, 40, 256), ny=_log(rng, 40, 256),
                    steps=rng.randrange(2, 9), f64=f64)
    lo, hi = dict(vof=(32, 240), phase=(32, 192), interface=(32, 176))[kind]
    c = dict(kind=kind, nx=_log(rng, lo, hi), ny=_log(rng, lo, hi), nz=_log(rng, lo, hi))
    return c if kind == "vof" else dict(c, f64=f64)


# ------------------------------------------------------------------ inputs
class _Params:
    """The fields of sfx_params (numbers, or tensors that broadcast)."""

    def __init__(self, **kw):
        d = dict(ka=1.0, kd=0.1, gamma_inf=1.0, Df=1e-2, DF=1e-2, eps=0.0, eta=1e-6, sigma0=1.0,
                 E=0.2, eos=0, literal_upwind=0, bc_F=1.0, bc_f=0.0)
        d.update(kw)
        self.__dict__.update(d)


def _rand(seed, n):
    return torch.rand(n, generator=torch.Generator().manual_seed(int(seed)), dtype=torch.float64)


def _centres(geom, shape, h):
    """Cell-centre coordinates (x, y[, z]) that broadcast to the cell shape."""
    nz, ny, nx = shape
    ax = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h for n in (nx, ny, nz)]
    x, y, z = ax[0].view(1, 1, -1), ax[1].view(1, -1, 1), ax[2].view(-1, 1, 1)
    return [x, y, z] if geom == CART else [x, y]


def _noise(seed, geom, shape, h):
    """Smooth seeded field with values within [-1, 1]: five cosine modes."""
    r = _rand(seed, 40).view(5, 8)
    x = _centres(geom, shape, h)
    L = max(shape) * h
    out = torch.zeros(shape, device="cuda", dtype=torch.float64)
    for m in r.tolist():
        t = 2 * math.pi * m[0]
        for a, q in zip(x, m[1:]):
            t = t + 2 * math.pi * (1 + 3 * q) / L * a
        out += torch.cos(t) / 5
    return out


def _distance(geom, shape, h, centre, R):
    """Signed distance of the circle or sphere, positive inside."""
    r2 = 0
    for a, c in zip(_centres(geom, shape, h), centre):
        r2 = r2 + (a - c) ** 2
    return (R - torch.sqrt(r2)).expand(shape)


def _phi(chi, h, eps):
    """The tanh profile of a distance known in the band that redistancing
    reaches (nine cells either side)."""
    return (0.5 * (1 - torch.tanh(torch.clamp(chi, -9 * h, 9 * h) / (2 * eps)))).contiguous()


def _fraction(geom, shape, h, centre, R, k=8):
    """Volume fraction of the circle, sphere or sphere on the axis: exact
    along x, k (k^2 in 3D) midpoints across the cut cells."""
    chi = _distance(geom, shape, h, centre, R)
    C = (chi > 0).double()
    cut = torch.nonzero(chi.abs() < (1.0 if geom == CART else 0.75) * h)
    x0 = cut[:, 2] * h
    q = (torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) / k
    y = (cut[:, 1, None] + q) * h - centre[1]
    s2 = R * R - y * y
    if geom == CART:
        z = (cut[:, 0, None] + q) * h - centre[2]
        s2 = (s2[:, :, None] - (z * z)[:, None, :]).flatten(1)
    if geom == AXI:
        a, b = (x0 ** 2)[:, None], ((x0 + h) ** 2)[:, None]
        v = ((torch.minimum(b, s2) - a).clamp(min=0) / (b - a)).mean(1)
    else:
        s, a = torch.sqrt(s2.clamp(min=0)), x0[:, None] - centre[0]
        v = ((torch.minimum(a + h, s) - torch.maximum(a, -s)).clamp(min=0) / h).mean(1)
    C[cut[:, 0], cut[:, 1], cut[:, 2]] = v.clamp(0, 1)
    return C


def _hr(r, R, lam=0.01):
    """Hadamard-Rybczynski stream function over (r sin theta)^2, unit far field."""
    A, B = (2 + 3 * lam) / (2 * (1 + lam)), lam / (2 * (1 + lam))
    r = r.clamp(min=1e-30)
    return torch.where(r >= R, 0.5 * (1 - A * R / r + B * R ** 3 / r ** 3),
                       (r * r / (R * R) - 1) / (4 * (1 + lam)))


def _hr_faces(geom, shape, h, centre, R):
    """Divergence-free face velocities of the Hadamard-Rybczynski flow."""
    nz, ny, nx = shape

    def grid(n, c, half):
        return (torch.arange(n + (not half), device="cuda", dtype=torch.float64) + 0.5 * half) * h - c
    if geom == AXI:
        r = grid(nx, 0.0, False)
        z = grid(ny, centre[1], False)[:, None]
        psi = r * r * _hr(torch.sqrt(r * r + z * z), R)
        ur = torch.zeros(ny, nx + 1, device="cuda", dtype=torch.float64)
        ur[:, 1:] = -(psi[1:, 1:] - psi[:-1, 1:]) / (r[1:] * h)
        uz = 2 * (psi[:, 1:] - psi[:, :-1]) / (r[1:] ** 2 - r[:-1] ** 2)
        return [ur[None].contiguous(), uz[None].contiguous()]
    v = [grid(n, c, False) for n, c in zip((nx, ny, nz), centre)]
    m = [grid(n, c, True) for n, c in zip((nx, ny, nz), centre)]
    z = v[2].view(-1, 1, 1)

    def pot(x, y):
        return _hr(torch.sqrt(x * x + y * y + z * z), R)
    ay = pot(v[0], m[1][:, None]) * v[0]
    ax = -pot(m[0], v[1][:, None]) * v[1][:, None]
    return [((ay[:-1] - ay[1:]) / h).contiguous(), ((ax[1:] - ax[:-1]) / h).contiguous(),
            ((ax[:, :-1] + ay[:, :, 1:] - ax[:, 1:] - ay[:, :, :-1]) / h).contiguous()]


def _stream_faces(psi, h):
    return [((psi[1:] - psi[:-1]) / h)[None].contiguous(),
            (-(psi[:, 1:] - psi[:, :-1]) / h)[None].contiguous()]


def _vortex_faces(nx, ny, h):
    """The single vortex: stream function sin^2 sin^2 / pi on the box."""
    x = torch.arange(nx + 1, device="cuda", dtype=torch.float64) / nx
    y = torch.arange(ny + 1, device="cuda", dtype=torch.float64)[:, None] / ny
    return _stream_faces(torch.sin(math.pi * x) ** 2 * torch.sin(math.pi * y) ** 2 / math.pi, h)


def _bubble(geom, shape, seed, flow=True, scale=0.2):
    """A bubble near the middle of the block, its fraction, profile and flow."""
    nz, ny, nx = shape
    h = 1.0 / (nx if geom == AXI else max(nx, ny, nz))
    ext = min(2 * nx, ny) if geom == AXI else min(n for n in (nx, ny, nz) if n > 1)
    j = _rand(seed, 3).tolist()
    centre = [(0.5 * n + q - 0.5) * h for n, q in zip((nx, ny, nz), j)]
    if geom == AXI:
        centre[0] = 0.0
    R = scale * ext * h
    eps = 0.75 * h
    chi = _distance(geom, shape, h, centre, R)
    return dict(h=h, eps=eps, centre=centre, R=R, chi=chi, phi=_phi(chi, h, eps),
                C=_fraction(geom, shape, h, centre, R),
                u=_hr_faces(geom, shape, h, centre, R) if flow else None)


def _step_problem(case, seed):
    """Inputs of a `step` case in 64 bits, rounded to what the context takes."""
    geom, shape = case["geom"], (case["nz"], case["ny"], case["nx"])
    flow, fl = case["flow"], torch.float64 if case["f64"] else torch.float32
    b = _bubble(geom, shape, seed, flow and geom != PLANAR, 0.25 if geom == PLANAR else 0.2)
    h = b["h"]
    if geom == PLANAR and flow:           # the rotating circle
        x, y = ((torch.arange(n + 1, device="cuda", dtype=torch.float64) * h - c)
                for n, c in zip((case["nx"], case["ny"]), b["centre"]))
        psi = -0.5 * (x * x + y[:, None] ** 2)
        b["u"] = _stream_faces(psi, h)
    if geom == CART:                      # Pe_F = 10, Pe_f = 100, d = 0.25
        p = _Params(ka=4.0, kd=4.0, Df=2.5e-3, DF=2.5e-2, eps=b["eps"])
        dt = 3.2 * h * h
    elif geom == AXI:                     # Pe = 100, d = 0.4
        p = _Params(ka=2.5, kd=2.5, Df=4e-3, DF=4e-3, eps=b["eps"])
        dt = 0.1 * h
    elif flow:
        p = _Params(ka=1 / 0.3, kd=1 / 0.3, Df=1e-4, DF=1e-4, eps=b["eps"])
        dt = 0.4 * h
    else:
        p = _Params(eps=b["eps"])
        dt = 1e-3 * min(1.0, (256 * h) ** 2) if h < 1 / 256 else 1e-3
    gamma = 0.2 * (1 + 0.5 * _noise(seed + 1, geom, shape, h))
    f = gamma * b["phi"] * (1 - b["phi"]) / b["eps"]
    F = 1 + 0.1 * _noise(seed + 2, geom, shape, h)
    if geom == PLANAR:
        F = F * (1 - b["C"])
    u = [x.to(fl) for x in b["u"]] if b["u"] else []
    return dict(b, p=p, dt=dt, f=f.contiguous(), F=F.contiguous(), u=u, C=b["C"].to(fl), fl=fl,
                geom=geom, shape=shape)


def _batch_sizes(case):
    rng = np.random.default_rng(case["pattern"])
    if case["geom"] == PLANAR:
        return [(case["nr"], case["pattern"])] * case["instances"]
    n = case["nr"]
    return [[(n // 4, n // 2), (n // 2, n), (n, 2 * n)][int(rng.integers(0, 3))]
            for _ in range(case["instances"])]


def _batch_problem(case, seed):
    """Instances grouped by size, each group stacked along the first axis."""
    geom, sizes = case["geom"], _batch_sizes(case)
    n = len(sizes)
    r = 10.0 ** (4 * _rand(seed, 2 * n).view(2, n) - 2)
    groups = []
    for size in sorted(set(sizes)):
        ids = [i for i, s in enumerate(sizes) if s == size]
        nr, nz = size
        Bi, Da = (r[q, ids].cuda().view(-1, 1, 1) for q in (0, 1))
        shape = (1, nz, nr)
        if geom == AXI:
            b = _bubble(AXI, shape, seed, True, 0.2)
            h, phi, eps = b["h"], b["phi"], b["eps"]
            u = [x.float().double() for x in b["u"]]
            dt, D = 0.1 * h, 4e-3
            p = _Params(ka=Da / 0.4, kd=Bi / 0.4, Df=D, DF=D, eps=eps)
            F = 1 + 0.1 * _noise(seed + 2, geom, shape, h)
        else:
            h = 8.0 / nz
            eps = 0.75 * h
            y = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5) * h - 4
            phi = _phi(-y.view(1, -1, 1).expand(shape), h, eps)
            dt, u = 0.256 * h * h, None
            p = _Params(ka=Da, kd=Bi, Df=1.0, DF=1.0, eps=eps)
            F = phi * (1 + 0.1 * _noise(seed + 2, geom, shape, h))
        gamma = 0.1 * (1 + 0.5 * _noise(seed + 1, geom, shape, h))
        f = gamma * phi * (1 - phi) / eps
        groups.append(dict(ids=ids, shape=shape, h=h, dt=dt, p=p, phi=phi, u=u,
                           f=f.expand(len(ids), -1, -1), F=F.expand(len(ids), -1, -1)))
    return groups


def _rollout_problem(case, seed):
    shape = (1, case["ny"], case["nx"])
    b = _bubble(PLANAR, shape, seed, False, 0.25)
    p = _Params(eps=b["eps"])
    gamma = 0.05 * (1 + _noise(seed + 1, PLANAR, shape, b["h"]))
    return dict(b, p=p, dt=1e-3, gamma=gamma, F=(1 - b["C"]), shape=shape)


def _interface_problem(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    fl = torch.float64 if case.get("f64") else torch.float32
    b = _bubble(CART, shape, seed, True, 0.25)
    p = _Params(ka=4.0, kd=4.0, eps=b["eps"])
    gamma = 0.3 * (1 + _noise(seed + 1, CART, shape, b["h"]))
    f = gamma * b["phi"] * (1 - b["phi"]) / b["eps"]
    umax = max(float(x.abs().max()) for x in b["u"])
    return dict(b, p=p, f=f, u=[x.to(fl) for x in b["u"]], Cf=b["C"].to(fl), shape=shape, fl=fl,
                umax=umax, dt=0.2 * b["h"] / umax)


def _moving_problem(case, seed):
    shape = (1, case["ny"], case["nx"])
    h = 1.0 / max(shape)
    j = (_rand(seed, 2) - 0.5).tolist()
    R = 0.15 * min(shape[1:]) * h
    centre = [(0.5 * case["nx"] + j[0]) * h, (0.72 * case["ny"] + j[1]) * h]
    C = _fraction(PLANAR, shape, h, centre, R, 32)
    eps = 0.75 * h
    p = _Params(ka=1 / 0.3, kd=1 / 0.3, Df=1e-4, DF=1e-4, eps=eps)
    phi = 0.5 * (1 - torch.tanh(_redistance(C, h, 2, 24, 0.5 * h) / (2 * eps)))
    f = 0.2 * (1 + 0.5 * _noise(seed + 1, PLANAR, shape, h)) * phi * (1 - phi) / eps
    F = (1 - C) * (1 + 0.1 * _noise(seed + 2, PLANAR, shape, h))
    u = [x.float() for x in _vortex_faces(case["nx"], case["ny"], h)]
    umax = max(float(x.abs().max()) for x in u)
    return dict(C=C, p=p, f=f, F=F, u=u, h=h, eps=eps, dt=0.4 * h / umax, shape=shape)


# --------------------------------------------------------- prepare and run
def _state(ctx, x):
    return sfx.sfx_df_pack(x.contiguous()) if ctx.precision == sfx.SFX_F32 else x.clone()


def _context(geom, shape, h, f64):
    return sfx.Context(geom, shape[2], shape[1], shape[0], h, sfx.SFX_F64 if f64 else sfx.SFX_F32)


def prepare(case, seed):
    kind, T = case["kind"], sfx._lib
    s = dict(kind=kind, n=0)
    if kind == "step":
        q = _step_problem(case, seed)
        ctx = _context(q["geom"], q["shape"], q["h"], case["f64"])
        opts = sfx.default_opts(tol=TOL)
        if case["tuned"]:          # a static interface, and the schedule of the benchmark
            opts.nu1, opts.nu2 = 3, 0
            for key, v in ((T.SFX_TUNE_REUSE_DRIFT, 1), (T.SFX_TUNE_PREDICT, 0),
                           (T.SFX_TUNE_F32_FAST_RESID, 1)):
                ctx.sfx_set_tuning(key, v)
        s.update(ctx=ctx, opts=opts, p=q["p"], dt=q["dt"], phi=q["phi"], C=q["C"], u=q["u"],
                 f=_state(ctx, q["f"]), F=_state(ctx, q["F"]))
        s["sigma"] = torch.empty(q["shape"], dtype=q["fl"], device="cuda")
        s["force"] = torch.empty((len(_centres(q["geom"], q["shape"], 1)),) + q["shape"],
                                 dtype=q["fl"], device="cuda")
    elif kind == "moving":
        q = _moving_problem(case, seed)
        ctx = _context(PLANAR, q["shape"], q["h"], False)
        ctx.sfx_set_tuning(T.SFX_TUNE_F32_REDIST, 1)     # phi is rebuilt every step
        opts = sfx.default_opts(tol=TOL, nu1=4, nu2=0)
        s.update(ctx=ctx, opts=opts, p=q["p"], dt=q["dt"], C=q["C"], u0=q["u"], h=q["h"],
                 u=[torch.empty_like(x) for x in q["u"]], chi=torch.empty_like(q["C"]),
                 phi=torch.empty_like(q["C"]), f=_state(ctx, q["f"]), F=_state(ctx, q["F"]))
        s["sigma"] = torch.empty(q["shape"], device="cuda")
        s["force"] = torch.empty((2,) + q["shape"], device="cuda")
    elif kind == "batch":
        groups = _batch_problem(case, seed)
        inst = [None] * len(_batch_sizes(case))
        for g in groups:
            nz, nr = g["shape"][1:]
            ka, kd = (x.flatten().tolist() for x in (g["p"].ka, g["p"].kd))
            for k, i in enumerate(g["ids"]):
                inst[i] = (nr, nz, g["h"], g["dt"], _Params(**dict(vars(g["p"]), ka=ka[k], kd=kd[k])))
        B = sfx.Batch(inst, geom=case["geom"])
        B.sfx_batch_set_schedule(256, 3, 60)
        B.sfx_batch_reuse_phi(True)
        rows = [None] * len(inst)
        for g in groups:
            for k, i in enumerate(g["ids"]):
                rows[i] = (g["phi"], g["f"][k], g["F"][k], g["u"])
        phi, f, F = (torch.cat([r[q].reshape(-1) for r in rows]) for q in range(3))
        u = [torch.cat([r[3][d].reshape(-1) for r in rows]).float() if rows[0][3] else None
             for d in range(2)]
        s.update(B=B, phi=phi, f=sfx.sfx_df_pack(f), F=sfx.sfx_df_pack(F), u=u)
    elif kind == "rollout":
        q = _rollout_problem(case, seed)
        ctx = _context(PLANAR, q["shape"], q["h"], case["f64"])
        p = q["p"]
        s.update(setup=sfx.RolloutSetup(context=ctx, params=p, phi=q["phi"], C=q["C"], F0=q["F"],
                                        dt=q["dt"], nsteps=case["steps"]),
                 gamma=q["gamma"].requires_grad_(True),
                 theta=torch.tensor([p.ka, p.kd, p.Df, p.DF], dtype=torch.float64,
                                    requires_grad=True))
    else:
        q = _interface_problem(case, seed)
        ctx = _context(CART, q["shape"], q["h"], case.get("f64", False))
        s.update(ctx=ctx, p=q["p"], dt=q["dt"], C=q["C"], Cf=q["Cf"], u=q["u"], umax=q["umax"],
                 h=q["h"], eps=q["eps"])
        if kind == "phase":
            s.update({k: torch.empty_like(q["C"]) for k in ("chi", "phi", "delta")})
        if kind == "interface":
            s.update(phi=q["phi"], f=_state(ctx, q["f"]), sigma=torch.empty_like(q["Cf"]),
                     kappa=torch.empty_like(q["Cf"]))
            s["ma"], s["cap"] = (torch.empty((3,) + q["shape"], dtype=q["fl"], device="cuda")
                                 for _ in range(2))
    return s


def run(s):
    kind, n = s["kind"], s["n"]
    s["n"] += 1
    if kind == "step":
        u = list(s["u"]) + [None] * (3 - len(s["u"]))
        st = s["ctx"].sfx_surfactant_step(s["p"], s["phi"], s["f"], s["F"], s["dt"], *u,
                                          opts=s["opts"])
        s["ctx"].sfx_marangoni_force(s["p"], s["f"], s["phi"], s["C"], s["sigma"], s["force"])
        return dict(f=s["f"], F=s["F"], sigma=s["sigma"], force=s["force"], mass_f=st.mass_f,
                    mass_F=st.mass_F)
    if kind == "moving":             # the vortex reverses: u = u0 cos(pi t / 2)
        ctx, dt = s["ctx"], s["dt"]
        for x, x0 in zip(s["u"], s["u0"]):
            torch.mul(x0, math.cos(math.pi * (n + 0.5) * dt / 2), out=x)
        ctx.sfx_vof_advect(s["u"][0], s["u"][1], None, dt, s["C"], n % 2)
        ctx.sfx_phase_field_build(s["C"], s["chi"], s["phi"], eps=s["p"].eps)
        ctx.sfx_surfactant_step(s["p"], s["phi"], s["f"], s["F"], dt, s["u"][0], s["u"][1],
                                opts=s["opts"])
        ctx.sfx_marangoni_force(s["p"], s["f"], s["phi"], s["C"].float(), s["sigma"], s["force"])
        return {k: s[k] for k in ("C", "phi", "f", "F", "sigma", "force")}
    if kind == "batch":
        s["B"].sfx_batch_step(s["phi"], s["f"], s["F"], TOL, ur=s["u"][0], uz=s["u"][1])
        return dict(f=s["f"], F=s["F"])
    if kind == "rollout":
        loss = sfx.SurfactantRollout.apply(s["gamma"], s["theta"], s["setup"])
        g = torch.autograd.grad(loss, (s["gamma"], s["theta"]))
        return dict(loss=loss.detach(), gamma=g[0], theta=g[1])
    ctx = s["ctx"]
    if kind == "vof":
        ctx.sfx_vof_advect(*s["u"], s["dt"], s["C"], n % 2)
        return s["C"]
    if kind == "phase":
        ctx.sfx_phase_field_build(s["C"], s["chi"], s["phi"], s["delta"], iters=24, dtau=s["h"] / 3,
                                  eps=s["eps"])
        return {k: s[k] for k in ("chi", "phi", "delta")}
    ctx.sfx_acdi_step(s["phi"], s["dt"], 1.1 * s["umax"], s["eps"], *s["u"], clip=True)
    ctx.sfx_marangoni_force(s["p"], s["f"], s["phi"], s["Cf"], s["sigma"], s["ma"])
    ctx.sfx_capillary_force(s["p"], s["phi"], s["Cf"], s["sigma"], s["cap"], s["kappa"])
    return {k: s[k] for k in ("phi", "sigma", "ma", "kappa", "cap")}


def work(case):
    """Unique bytes of a pass (each input read once, each output written
    once) and the operations of one evaluation of each formula."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(a * b for a, b in _batch_sizes(case))
        d = 2 if case["geom"] == AXI else 0
        return dict(bytes=n * (16 + 16 + 8 + 4 * d), flops=n * (300 + 100 * d))
    n = case["nx"] * case["ny"] * case.get("nz", 1)
    w = 8 if case.get("f64") else 4
    if kind == "step":
        d = 2 if case["nz"] == 1 else 3
        du = d if case["flow"] else 0
        # f, F in and out, phi, velocities, C; sigma and force out
        return dict(bytes=n * (32 + 8 + w * (du + 1 + 1 + d)), flops=n * (300 + 100 * du))
    if kind == "moving":
        return dict(bytes=n * (32 + 16 + 8 + 4 * (2 + 1 + 2)), flops=n * 1500)
    if kind == "rollout":
        # per step and direction: the state in and out, phi
        return dict(bytes=n * case["steps"] * 2 * 40, flops=n * case["steps"] * 800)
    if kind == "vof":
        return dict(bytes=n * (16 + 12), flops=n * 60)
    if kind == "phase":
        return dict(bytes=n * 32, flops=n * 24 * 25)
    return dict(bytes=n * (16 + 8 + w * (3 + 1 + 1 + 1 + 3 + 3)), flops=n * 500)


# ------------------------------------------------------- the same in 64 bits
# Fields are (..., ny, nx) in 2D (leading axes hold independent blocks) and
# (nz, ny, nx) in 3D; direction d runs along dimension -1 - d.
def _nb(a, d, s):
    """Neighbour values, the cell's own beyond a wall."""
    x = -1 - d
    n = a.shape[x]
    if s > 0:
        return torch.cat([a.narrow(x, 1, n - 1), a.narrow(x, n - 1, 1)], x)
    return torch.cat([a.narrow(x, 0, 1), a.narrow(x, 0, n - 1)], x)


def _split(a, d):
    """Left and right cells of the interior faces in direction d."""
    n = a.shape[-1 - d]
    return a.narrow(-1 - d, 0, n - 1), a.narrow(-1 - d, 1, n - 1)


def _volume(geom, shape, h):
    i = torch.arange(shape[-1], device="cuda", dtype=torch.float64)
    if geom == AXI:
        return math.pi * (2 * i + 1) * h ** 3
    return torch.full_like(i, h ** (3 if geom == CART else 2))


def _area(geom, shape, h, d):
    """Areas of all faces in direction d (broadcast along x)."""
    i = torch.arange(shape[-1] + (d == 0), device="cuda", dtype=torch.float64)
    if geom != AXI:
        return torch.full_like(i, h ** (2 if geom == CART else 1))
    return 2 * math.pi * i * h * h if d == 0 else math.pi * (2 * i + 1) * h * h


def _grad(a, d, h):
    return (_nb(a, d, 1) - _nb(a, d, -1)) / (2 * h)


def _normals(phi, eps, h, nd):
    g = [_grad(phi, d, h) for d in range(nd)]
    m = torch.sqrt(sum(x * x for x in g))
    w = (m / (1e-3 * (phi * (1 - phi) / eps)) - 1).clamp(max=1)
    w = torch.where((m >= 1e-30) & (w > 0), w, torch.zeros_like(w))
    return [torch.where(w > 0, w * (x / m), torch.zeros_like(w)) for x in g]


class _System:
    """The coupled implicit problem of one step: residuals, diagonal blocks
    and a red-black Newton solve."""

    def __init__(self, geom, h, p, phi, dt):
        self.geom, self.h, self.p, self.phi, self.dt = geom, h, p, phi, dt
        self.nd = 3 if geom == CART else 2
        n = _normals(phi, p.eps, h, self.nd)
        # drift per unit diffusivity on the interior faces
        self.B = []
        for s in (-2 * (0.5 - phi) / p.eps, -(1 - phi) / p.eps):
            self.B.append([0.5 * sum(_split(s * x, d)) for d, x in enumerate(n)])
        self.pe = phi + p.eta
        self.finf = p.gamma_inf * phi * (1 - phi) / p.eps
        self.V = _volume(geom, phi.shape, h)

    def faces(self, which, D):
        for d in range(self.nd):
            B = D * self.B[which][d]
            A = _area(self.geom, self.phi.shape, self.h, d)
            A = A[1:-1] if d == 0 else A
            left = B < 0
            z = torch.zeros_like(B)
            yield d, A * (torch.where(left, B, z) - D / self.h), A * (torch.where(left, z, B) + D / self.h)

    def flux(self, a, which, D):
        """(1/V) sum of the face fluxes of field a."""
        out = torch.zeros_like(a)
        for d, cL, cR in self.faces(which, D):
            L, R = _split(a, d)
            G = cL * L + cR * R
            x = -1 - d
            pad = torch.zeros_like(a.narrow(x, 0, 1))
            out = out + torch.cat([G, pad], x) - torch.cat([pad, G], x)
        return out / self.V

    def diagonal(self, which, D, like):
        out = torch.zeros_like(like)
        for d, cL, cR in self.faces(which, D):
            x = -1 - d
            n = out.shape[x]
            out.narrow(x, 0, n - 1).add_(cL)
            out.narrow(x, 1, n - 1).sub_(cR)
        return out / self.V

    def residual(self, f, F, fs, Fs, th=None):
        ka, kd, Df, DF = th if th is not None else (self.p.ka, self.p.kd, self.p.Df, self.p.DF)
        q = ka * F / self.pe * (self.finf - f) - kd * f
        return ((fs - f) / self.dt + self.flux(f, 0, Df) + q,
                (Fs - F) / self.dt + self.flux(F, 1, DF) - q)

    def block(self, f, F):
        """Diagonal 2x2 blocks of -J, as (a, b, c, d) with det."""
        p = self.p
        u, v = p.ka * F / self.pe, p.ka * (self.finf - f) / self.pe
        a = 1 / self.dt - self.diagonal(0, p.Df, f) + u + p.kd
        d = 1 / self.dt - self.diagonal(1, p.DF, F) + v
        return a, -v, -(u + p.kd), d

    def colours(self, like):
        s = 0
        for d in range(self.nd):
            shape = [1] * like.dim()
            shape[-1 - d] = -1
            s = s + torch.arange(like.shape[-1 - d], device="cuda").view(shape)
        red = (s % 2 == 0).expand(like.shape)
        return red, ~red

    def solve(self, fs, Fs):
        f, F = fs.clone(), Fs.clone()
        best, stall, colours = math.inf, 0, self.colours(fs)
        scale = fs.abs().max() / self.dt, Fs.abs().max() / self.dt
        for _ in range(40):
            rf, rF = self.residual(f, F, fs, Fs)
            now = max(float(rf.abs().max() / scale[0]), float(rF.abs().max() / scale[1]))
            if now < 1e-15 or (now >= 0.5 * best and now < 1e-11):
                stall += 1
                if now < 1e-15 or stall > 2:
                    break
            best = min(best, now)
            a, b, c, d = self.block(f, F)
            det = a * d - b * c
            u, v = self.p.ka * F / self.pe, self.p.ka * (self.finf - f) / self.pe
            ef, eF = torch.zeros_like(f), torch.zeros_like(F)
            for _ in range(8):
                for m in colours:
                    x = (u + self.p.kd) * ef - v * eF
                    sf = rf - ef / self.dt + self.flux(ef, 0, self.p.Df) - x
                    sF = rF - eF / self.dt + self.flux(eF, 1, self.p.DF) + x
                    ef = torch.where(m, ef + (d * sf - b * sF) / det, ef)
                    eF = torch.where(m, eF + (a * sF - c * sf) / det, eF)
            f, F = f + ef, F + eF
        return f, F

    def adjoint(self, f, F, lf, lF):
        """nu of (-J)^T nu = lam, dL/dtheta of the step."""
        p = self.p
        f, F = f.detach().requires_grad_(True), F.detach().requires_grad_(True)
        th = [torch.tensor(float(v), device="cuda", dtype=torch.float64, requires_grad=True)
              for v in (p.ka, p.kd, p.Df, p.DF)]
        zero = torch.zeros_like(f)
        R = self.residual(f, F, zero, zero, th)
        with torch.no_grad():
            a, b, c, d = self.block(f, F)
            det = a * d - b * c
        nf, nF = torch.zeros_like(lf), torch.zeros_like(lF)
        scale = max(float(lf.abs().max()), float(lF.abs().max()))
        for it in range(400):
            for m in self.colours(lf):
                jf, jF = torch.autograd.grad(R, (f, F), (nf, nF), retain_graph=True)
                rf, rF = lf + jf, lF + jF
                nf = torch.where(m, nf + (d * rf - c * rF) / det, nf)
                nF = torch.where(m, nF + (a * rF - b * rf) / det, nF)
            if it % 10 == 9 and max(float(rf.abs().max()), float(rF.abs().max())) < 3e-16 * scale:
                break
        return nf, nF, torch.stack(torch.autograd.grad(R, th, (nf, nF)))


def _advect(geom, h, u, dt, xi, bc):
    """The explicit BCG step."""
    nd = 3 if geom == CART else 2
    slopes, parts = [], []
    for d in range(nd):
        m, q = _nb(xi, d, -1), _nb(xi, d, 1)
        dl, dr, dc = xi - m, q - xi, 0.5 * (q - m)
        lim = torch.minimum(dc.abs(), 2 * torch.minimum(dl.abs(), dr.abs()))
        slopes.append(torch.where(dl * dr <= 0, torch.zeros_like(xi), torch.where(dc > 0, lim, -lim)))
        n = xi.shape[-1 - d]
        vb = 0.5 * (u[d].narrow(-1 - d, 0, n) + u[d].narrow(-1 - d, 1, n))
        parts.append(0.5 * dt * vb * torch.where(vb > 0, dl, dr) / h)
    div = torch.zeros_like(xi)
    for d in range(nd):
        x, n = -1 - d, xi.shape[-1 - d]
        tr = sum(parts[t] for t in range(nd) if t != d)
        c = u[d] * dt / h
        wall = torch.full_like(xi.narrow(x, 0, 1), bc)
        left = torch.cat([wall, xi + 0.5 * (1 - c.narrow(x, 1, n)) * slopes[d] - tr], x)
        right = torch.cat([xi + 0.5 * (-1 - c.narrow(x, 0, n)) * slopes[d] - tr, wall], x)
        G = _area(geom, xi.shape, h, d) * u[d] * torch.where(u[d] > 0, left, right)
        div = div + G.narrow(x, 1, n) - G.narrow(x, 0, n)
    return xi - dt * div / _volume(geom, xi.shape, h)


def _eos(p, f, phi):
    dl = phi * (1 - phi) / p.eps
    G = torch.where(dl >= 1e-3 / p.eps, f / dl.clamp(min=1e-300), torch.zeros_like(f))
    return p.sigma0 * (1 + p.E * torch.log1p(-(G / p.gamma_inf).clamp(max=1 - 1e-12)))


def _volume_below(m, a):
    """Unit-cube volume below m.x = a (rows of m: non-negative, sum 1) and
    its derivative in a."""
    m, _ = torch.sort(m, dim=0)
    t = torch.where(a <= 0.5, a, 1 - a).clamp(min=0)
    if m.shape[0] == 2:
        m1, m2 = m[0].clamp(min=1e-300), m[1]
        corner = t < m[0]
        v = torch.where(corner, t * t / (2 * m1 * m2), (t - 0.5 * m1) / m2)
        dv = torch.where(corner, t / (m1 * m2), 1 / m2)
    else:
        m1, m2, m3 = m
        s1, s2 = m1.clamp(min=1e-300), m2.clamp(min=1e-300)
        k6, k2 = 1 / (6 * s2 * m3), 1 / (2 * s2 * m3)
        u, w = t - m2, t - m3
        base, dbase = (3 * t * t - 3 * t * m1 + m1 * m1) * k6, (2 * t - m1) * k2
        v = torch.where(m3 >= m1 + m2, (t - 0.5 * (m1 + m2)) / m3, base - (u ** 3 + w ** 3) * k6 / s1)
        dv = torch.where(m3 >= m1 + m2, 1 / m3, dbase - (u * u + w * w) * k2 / s1)
        r = (t < m3) & (t < m1 + m2)
        v, dv = torch.where(r, base - u ** 3 * k6 / s1, v), torch.where(r, dbase - u * u * k2 / s1, dv)
        r = t < m2
        v, dv = torch.where(r, (t * t - t * m1 + m1 * m1 / 3) * k2, v), torch.where(r, dbase, dv)
        r = t < m1
        v, dv = torch.where(r, t ** 3 * k6 / s1, v), torch.where(r, t * t * k2 / s1, dv)
    v = torch.where(a <= 0.5, v, 1 - v)
    out = (a <= 0) | (a >= 1)
    v = torch.where(a <= 0, torch.zeros_like(v), torch.where(a >= 1, torch.ones_like(v), v))
    return v, torch.where(out, torch.zeros_like(dv), dv)


def _youngs(C, nd):
    """Youngs normal: minus the 1-2-1 weighted centred difference."""
    out = []
    for d in range(nd):
        g = C
        for t in range(nd):
            m, q = _nb(g, t, -1), _nb(g, t, 1)
            g = m - q if t == d else m + 2 * g + q
        out.append(g)
    return torch.stack(out)


def _plane(m, C):
    """(normalised |m|, |m|_2 / |m|_1, plane offset) of the cells' fractions."""
    s = m.abs().sum(0)
    n = torch.where(s > 0, m.abs() / s.clamp(min=1e-300), torch.zeros_like(m))
    lo, hi = torch.zeros_like(C), torch.ones_like(C)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        less = _volume_below(n, mid)[0] < C
        lo, hi = torch.where(less, mid, lo), torch.where(less, hi, mid)
    return n, torch.sqrt((n * n).sum(0)), 0.5 * (lo + hi)


def _interface_area(C, nd, h):
    """delta_m of the interface cells."""
    out = torch.zeros_like(C)
    cut = (C > 1e-6) & (C < 1 - 1e-6)
    n, l2, a = _plane(_youngs(C, nd)[:, cut], C[cut])
    out[cut] = torch.where(l2 > 0, l2 * _volume_below(n, a)[1], torch.zeros_like(a)) / h
    return out


def _marangoni(p, f, phi, C, h, nd, dm=None):
    s = _eos(p, f, phi)
    g = [_grad(s, d, h) for d in range(nd)]
    n = _normals(phi, p.eps, h, nd)
    dm = _interface_area(C, nd, h) if dm is None else dm
    t = sum(a * b for a, b in zip(n, g))
    return s, torch.stack([dm * (a - b * t) for a, b in zip(g, n)])


def _vof(C, u, dt, h, nd, order):
    H = (C > 0.5).double()
    for d in (reversed(range(nd)) if order else range(nd)):
        x, n = -1 - d, C.shape[-1 - d]
        c = u[d] * dt / h
        cf = c.narrow(x, 1, n - 1)
        L, R = _split(C, d)
        Cu = torch.where(cf > 0, L, R)
        Q = Cu.clamp(0, 1) * cf          # full and empty upwind cells
        cut = (Cu > 0) & (Cu < 1) & (cf != 0)
        m = _youngs(C, nd)
        m = torch.stack([torch.where(cf > 0, *_split(y, d))[cut] for y in m])
        cc, cu = cf[cut], Cu[cut]
        nn, l2, a = _plane(m, cu)
        lo = torch.where(cc > 0, 1 - cc, torch.zeros_like(cc))
        hi = torch.where(cc > 0, torch.ones_like(cc), -cc)
        flip = m[d] < 0
        lo, hi = torch.where(flip, 1 - hi, lo), torch.where(flip, 1 - lo, hi)

        def below(t):
            w = nn.clone()
            w[d] = w[d] * t
            s = w.sum(0).clamp(min=1e-300)
            return torch.where(t > 0, t * _volume_below(w / s, a / s)[0], torch.zeros_like(t))
        q = torch.where(l2 > 0, below(hi) - below(lo), cu * (hi - lo))
        Q[cut] = torch.where(cc > 0, q, -q)
        pad = torch.zeros_like(C.narrow(x, 0, 1))
        C = C - (torch.cat([Q, pad], x) - torch.cat([pad, Q], x)) + H * (c.narrow(x, 1, n) - c.narrow(x, 0, n))
    return C


def _redistance(C, h, nd, iters, dtau):
    c0 = 2 * h * (C - 0.5)
    s = torch.sign(c0)
    near, acc = torch.zeros_like(C, dtype=torch.bool), torch.zeros_like(C)
    for d in range(nd):
        m, q = _nb(c0, d, -1), _nb(c0, d, 1)
        near |= (c0 * m < 0) | (c0 * q < 0)
        w = torch.maximum(0.5 * (q - m).abs(), torch.maximum((q - c0).abs(), (c0 - m).abs()))
        acc += w * w
    dist = h * c0 / torch.sqrt(acc).clamp(min=1e-300)
    chi = c0.clone()
    for _ in range(iters):
        g = torch.zeros_like(C)
        for d in range(nd):
            a, b = s * (chi - _nb(chi, d, -1)) / h, s * (_nb(chi, d, 1) - chi) / h
            g += torch.maximum(a.clamp(min=0) ** 2, b.clamp(max=0) ** 2)
        # a cell with chi0 = 0 stays
        chi = torch.where(near, chi - dtau / h * (s * chi.abs() - dist),
                          chi - dtau * s * (torch.sqrt(g) - 1))
    return chi


def _pair(x):
    hi = x.float().double()
    return torch.stack([hi, x - hi], -1)


def _coupled(geom, h, p, phi, u, dt, f, F):
    if u:
        u = [x.double() for x in u]
        f, F = _advect(geom, h, u, dt, f, p.bc_f), _advect(geom, h, u, dt, F, p.bc_F)
    return _System(geom, h, p, phi, dt).solve(f, F)


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        q = _step_problem(case, seed)
        p, h, geom, nd = q["p"], q["h"], q["geom"], 3 if q["geom"] == CART else 2
        f, F = _coupled(geom, h, p, q["phi"], q["u"], q["dt"], q["f"], q["F"])
        s, force = _marangoni(p, f, q["phi"], q["C"].double(), h, nd)
        V = _volume(geom, f.shape, h)
        st = (lambda x: x) if case["f64"] else _pair
        return dict(f=st(f), F=st(F), sigma=s, force=force, mass_f=float((V * f).sum()),
                    mass_F=float((V * F).sum()))
    if kind == "moving":
        q = _moving_problem(case, seed)
        p, h, dt = q["p"], q["h"], q["dt"]
        a = math.cos(math.pi * 0.5 * dt / 2)
        u = [(x * a).double() for x in q["u"]]
        C = _vof(q["C"], u, dt, h, 2, 0)
        phi = 0.5 * (1 - torch.tanh(_redistance(C, h, 2, 24, 0.5 * h) / (2 * q["eps"])))
        f, F = _coupled(PLANAR, h, p, phi, u, dt, q["f"], q["F"])
        s, force = _marangoni(p, f, phi, C.float().double(), h, 2)
        return dict(C=C, phi=phi, f=_pair(f), F=_pair(F), sigma=s, force=force)
    if kind == "batch":
        rows = [None] * len(_batch_sizes(case))
        for g in _batch_problem(case, seed):
            n = len(g["ids"])
            u = [x.expand(n, -1, -1) for x in g["u"]] if g["u"] else None
            phi = g["phi"].expand(n, -1, -1)
            f, F = _coupled(case["geom"], g["h"], g["p"], phi, u, g["dt"], g["f"], g["F"])
            for k, i in enumerate(g["ids"]):
                rows[i] = (f[k].reshape(-1), F[k].reshape(-1))
        return dict(f=_pair(torch.cat([r[0] for r in rows])), F=_pair(torch.cat([r[1] for r in rows])))
    if kind == "rollout":
        q = _rollout_problem(case, seed)
        p, h, phi = q["p"], q["h"], q["phi"]
        dl = phi * (1 - phi) / p.eps
        S, states = _System(PLANAR, h, p, phi, q["dt"]), [(q["gamma"] * dl, q["F"])]
        for _ in range(case["steps"]):
            states.append(S.solve(*states[-1]))
        f = states[-1][0].detach().requires_grad_(True)
        force = _marangoni(p, f, phi, q["C"], h, 2)[1]
        loss = h * h * (force * force).sum()
        lf, lF = torch.autograd.grad(loss, f)[0], torch.zeros_like(q["F"])
        theta = torch.zeros(4, device="cuda", dtype=torch.float64)
        for f1, F1 in reversed(states[1:]):
            nf, nF, t = S.adjoint(f1, F1, lf, lF)
            lf, lF, theta = nf / q["dt"], nF / q["dt"], theta + t
        return dict(loss=loss.detach().cpu(), gamma=lf * dl, theta=theta.cpu())
    q = _interface_problem(case, seed)
    h, p, u = q["h"], q["p"], [x.double() for x in q["u"]]
    if kind == "vof":
        return _vof(q["C"], u, q["dt"], h, 3, 0)
    if kind == "phase":
        chi = _redistance(q["C"], h, 3, 24, h / 3)
        phi = 0.5 * (1 - torch.tanh(chi / (2 * q["eps"])))
        return dict(chi=chi, phi=phi, delta=phi * (1 - phi) / q["eps"])
    eps, dt, ve = q["eps"], q["dt"], 1e-6
    ps = _advect(CART, h, u, dt, q["phi"], 1.0)
    pc = ps.clamp(0, 1)
    psi = eps * torch.log((pc + ve) / (1 - pc + ve))
    g = [_grad(psi, d, h) for d in range(3)]
    m = torch.sqrt(sum(x * x for x in g))
    out = ps.clone()
    for d in range(3):
        n = torch.where(m < 0.1, torch.zeros_like(m), g[d] / m.clamp(min=1e-300))
        (L, R), (nL, nR), (sL, sR) = _split(ps, d), _split(n, d), _split(psi, d)
        t = torch.tanh(0.5 * (sL + sR) / (2 * eps))
        G = 1.1 * q["umax"] * (eps * (R - L) / h - 0.25 * (1 - t * t) * 0.5 * (nL + nR)) * dt / h
        k = ps.shape[-1 - d]
        out.narrow(-1 - d, 0, k - 1).add_(G)
        out.narrow(-1 - d, 1, k - 1).sub_(G)
    phi = out.clamp(0, 1)
    C = q["Cf"].double()
    s, ma = _marangoni(p, q["f"], phi, C, h, 3)
    n = _normals(phi, eps, h, 3)
    kappa = torch.zeros_like(phi)
    for d in range(3):
        L, R = _split(n[d], d)
        G, k = 0.5 * (L + R) / h, phi.shape[-1 - d]
        kappa.narrow(-1 - d, 0, k - 1).sub_(G)
        kappa.narrow(-1 - d, 1, k - 1).add_(G)
    ds = torch.sqrt(sum(_grad(C, d, h) ** 2 for d in range(3)))
    return dict(phi=phi, sigma=s, ma=ma, kappa=kappa, cap=torch.stack([s * kappa * ds * x for x in n]))
