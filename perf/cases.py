"""The work this library does for its users, as cases that can be timed and checked.

Every case goes through the public Python API (`Simulation`, `Ensemble`,
`run_window`, `kinetic_energy`).  One pass sets the state from a device
array, advances it (or pulls a cotangent back through a step) and reads the
result: the loop body of a DNS between two outputs, of an adjoint gradient,
or of an ensemble.  FP32 runs return their results rounded to FP32, the
precision they are computed in; FP64 runs return FP64.

`exact` evaluates the same scheme (Cao, Pan & Xu, arXiv:2005.08736) in plain
64-bit torch, written from the paper's equations: WENO5 and the tangential
reconstructions (Sec. 2.1, Remark 1), the BGK flux by moments of the
Maxwellian (Eq. (5)), the linear fit (Eq. (7)), S2O4 (Eq. (6)); gradients by
autograd through it.
"""
import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_2005_08736_gb300.solver import (Config, Ensemble, Simulation, channel_config, isotropic_config,
                                           kinetic_energy, run_window)

RECON = {"linear": 0, "weno-js": 1, "weno-z": 2}
FLUX = {"smooth": 0, "full": 1}


def listed():
    return [
        # A small Taylor-Green run (the 32^3 verification set-up, 20 steps): latency and launches.
        _flow("taylor_green_32", "vortex", (32, 32, 32), "fp32", "linear", "smooth", steps=20),
        # The headline: one step of Taylor-Green 256^3, launch shape tuned as a long run does once.
        _flow("taylor_green_256", "vortex", (256, 256, 256), "fp32", "linear", "smooth", tuned=True),
        # The FP64 reference run at 128^3 that FP32 results are held against.
        _flow("taylor_green_128_fp64", "vortex", (128, 128, 128), "fp64", "linear", "smooth"),
        # A ragged box with nonlinear weights and the smooth flux (under-resolved low-Mach flow).
        _flow("vortex_ragged_wenojs", "vortex", (100, 83, 77), "fp32", "weno-js", "smooth", steps=2),
        # Compressible isotropic turbulence at full size: WENO-Z, full flux.
        _flow("isotropic_256", "isotropic", (256, 256, 256), "fp32", "weno-z", "full"),
        # The same physics at the size of the gradient studies, in FP64.
        _flow("isotropic_64_fp64", "isotropic", (64, 64, 64), "fp64", "weno-z", "full"),
        # Strong compressibility: characteristic variables, turbulent Mach 0.9, odd sizes.
        _flow("isotropic_char_ragged", "isotropic", (90, 75, 67), "fp32", "weno-z", "full", char=True,
              mach=0.9),
        # The channel at Re_tau 180: walls, stretched grid, constant body force, noisy start.
        _flow("channel_128x128x96", "channel", (128, 128, 96), "fp32", "linear", "smooth", steps=5),
        # A small channel box held at constant mass flux, resolved fluctuations.
        _flow("channel_small_massflux", "channel", (50, 43, 38), "fp32", "linear", "smooth", steps=5,
              mass_flux=True),
        # One adjoint step of the 64^3 isotropic gradient in FP32, with the differentiable
        # reconstruction that gradients are taken with (WENO-Z's weights have kinks).
        dict(_flow("adjoint_64", "isotropic", (64, 64, 64), "fp32", "weno-js", "full", k0=4.0), do="adjoint"),
        # A differentiable window with a checkpoint, FP64: final state and energy gradient.
        dict(_flow("gradient_window_fp64", "isotropic", (40, 36, 33), "fp64", "weno-js", "smooth", steps=3,
                   k0=4.0), do="window"),
        # A batch of independent boxes of uneven sizes advanced together.
        dict(_flow("ensemble_mixed", "isotropic", (0, 0, 0), "fp32", "weno-z", "full", k0=4.0), do="ensemble",
             sizes="32,48,64,96,32,48,64,96"),
    ]


def _flow(name, kind, n, prec, recon, flux, steps=1, tuned=False, char=False, mach=0.5, mass_flux=False,
          k0=8.0):
    """A case: `steps` steps of CFL size from a seeded field of `kind` on an
    n[0] x n[1] x n[2] grid."""
    return dict(name=name, do="steps", kind=kind, nx=n[0], ny=n[1], nz=n[2], prec=prec, recon=recon,
                flux=flux, steps=steps, tuned=tuned, char=char, mach=mach, mass_flux=mass_flux, k0=k0)


# Cells times steps a drawn case may hold at most, by precision and flux: no
# drawn case costs more than the largest listed one.
_MOST = {("fp32", "smooth"): 1.6e7, ("fp32", "full"): 4e6, ("fp64", "smooth"): 1.6e6, ("fp64", "full"): 2e5}


def draw(rng):
    do = rng.choice(["steps", "steps", "steps", "steps", "adjoint", "window", "ensemble"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    flux = rng.choice(["smooth", "full"])
    recon = rng.choice(["linear", "weno-js", "weno-z"]) if flux == "smooth" else rng.choice(["weno-js", "weno-z"])
    kind = rng.choice(["vortex", "isotropic", "channel"]) if do == "steps" else "isotropic"
    if do in ("adjoint", "window"):
        recon = rng.choice(["linear", "weno-js"]) if flux == "smooth" else "weno-js"
    if kind == "channel":
        recon, flux = "linear", "smooth"
    if do == "ensemble":
        prec = "fp32"
    steps = {"steps": rng.choice([1, 2, 5]), "window": rng.choice([2, 3])}.get(do, 1)
    share = {"steps": steps, "adjoint": 8, "window": 12 * steps, "ensemble": 1}[do]
    most = _MOST[prec, flux] / share
    side = (most ** (1.0 / 3.0)) / 16.0

    def cells():
        return max(12, int(16.0 * math.exp(rng.uniform(0.0, math.log(max(side, 1.01))))))

    c = _flow("", kind, (cells(), cells(), cells()), prec, recon, flux, steps=steps,
              char=recon != "linear" and do == "steps" and rng.random() < 0.25, mach=rng.choice([0.3, 0.4, 0.5]),
              mass_flux=kind == "channel" and rng.random() < 0.5, k0=4.0,
              tuned=do == "steps" and rng.random() < 0.25)
    c["do"] = do
    if do == "ensemble":
        c.update(nx=0, ny=0, nz=0)
        c["sizes"] = ",".join(str(rng.randrange(20, 65)) for _ in range(rng.randrange(3, 9)))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs ---

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _config(case, n):
    """The library configuration of a case on an n[0] x n[1] x n[2] grid."""
    kind = case["kind"]
    if kind == "channel":
        kw = dict(force_mode=1, mass_flux=1.0) if case["mass_flux"] else {}
        c = channel_config(*n, prec=case["prec"], **kw)
    elif kind == "isotropic":
        c = isotropic_config(n[0], prec=case["prec"], mach_t=case["mach"], k0=case["k0"], recon=case["recon"],
                             flux=case["flux"])
    else:
        c = Config(*n, prec={"fp64": 0, "fp32": 1}[case["prec"]], recon=RECON[case["recon"]],
                   flux=FLUX[case["flux"]], tau_num_C=1.0 if case["flux"] == "full" else 0.0)
    c.nx, c.ny, c.nz = n
    if case["do"] in ("adjoint", "window"):
        c.tau_num_C = 0.0  # |p_l - p_r| is not differentiable where the jump vanishes
    c.recon_vars = int(case["char"])
    return c


def _waves(n, gen, kmax, count, device):
    """A seeded smooth periodic field of a few low modes on the unit box, |f| <~ 1; [nz][ny][nx]."""
    ax = [2 * math.pi * (torch.arange(m, device=device, dtype=torch.float64) + 0.5) / m for m in n]
    f = torch.zeros(n[2], n[1], n[0], dtype=torch.float64, device=device)
    for _ in range(count):
        k = torch.randint(-kmax, kmax + 1, (3,), generator=gen).tolist()
        ph, a = (torch.rand(2, generator=gen, dtype=torch.float64) * 2 * math.pi).tolist()
        f += math.sin(a) / math.sqrt(count) * torch.sin(k[0] * ax[0][None, None, :] + k[1] * ax[1][None, :, None] +
                                                        k[2] * ax[2][:, None, None] + ph)
    return f


def _vortex(cfg, seed, device):
    """Taylor-Green vortex (Sec. 3.1, Ma 0.1), translated by a seeded offset,
    with seeded smooth perturbations of 2 % of the velocity."""
    n = (cfg.nx, cfg.ny, cfg.nz)
    gen = torch.Generator().manual_seed(seed)
    off = (torch.rand(3, generator=gen, dtype=torch.float64) * 2 * math.pi).tolist()
    x, y, z = [2 * math.pi * (torch.arange(m, device=device, dtype=torch.float64) + 0.5) / m + o
               for m, o in zip(n, off)]
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    u = torch.sin(x) * torch.cos(y) * torch.cos(z)
    v = -torch.cos(x) * torch.sin(y) * torch.cos(z)
    p = cfg.p_ref + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2) / 16
    w = [_waves(n, gen, 3, 4, device) for _ in range(4)]
    return torch.stack([1 + 0.002 * w[3], u + 0.02 * w[0], v + 0.02 * w[1], 0.02 * w[2], p])


def _isotropic(cfg, seed, k0, mach, device):
    """Random solenoidal velocity with E(k) ~ k^4 exp(-2 k^2/k0^2) (Sec. 3.4)
    at turbulent Mach number `mach`, with isentropic density and pressure
    fluctuations of the same spectrum, of the relative size mach^2/4 that a
    developed field has."""
    n = (cfg.nx, cfg.ny, cfg.nz)
    gen = torch.Generator(device=device).manual_seed(seed)
    k = [torch.fft.fftfreq(m, 1.0 / m, device=device, dtype=torch.float64) for m in n]
    kx, ky, kz = k[0][None, None, :], k[1][None, :, None], k[2][:, None, None]
    k2 = kx * kx + ky * ky + kz * kz
    amp = torch.sqrt(k2) * torch.exp(-k2 / k0 ** 2)
    noise = torch.randn(4, n[2], n[1], n[0], generator=gen, dtype=torch.float64, device=device)
    uh = [torch.fft.fftn(a) * amp for a in noise]
    div = (kx * uh[0] + ky * uh[1] + kz * uh[2]) / k2.clamp(min=1.0)
    u = [torch.fft.ifftn(h - kk * div).real for h, kk in zip(uh, (kx, ky, kz))]
    s = torch.fft.ifftn(uh[3]).real
    c0 = math.sqrt(1.4 * cfg.p_ref)
    rms = torch.sqrt(sum((a * a).mean() for a in u) / 3)
    s = s * (0.25 * mach * mach / torch.sqrt((s * s).mean()))
    u = [a * (mach * c0 / math.sqrt(3) / rms) for a in u]
    s = s.clamp(-0.5, 0.5)
    return torch.stack([1 + s, u[0], u[1], u[2], cfg.p_ref * (1 + s) ** 1.4])


def _channel(cfg, seed, noisy, device):
    """Channel start of Sec. 3.3: the laminar profile with 10 % velocity
    fluctuations, of cell size (the paper's start) or smooth (a developed flow)."""
    n = (cfg.nx, cfg.ny, cfg.nz)
    gen = torch.Generator().manual_seed(seed)
    w = _widths(cfg, 1, device)[3:-3]
    yc = -1 + torch.cumsum(w, 0) - 0.5 * w
    U = (1.5 * (1 - yc ** 2))[None, :, None].expand(n[2], n[1], n[0])
    if noisy:
        g = torch.Generator(device=device).manual_seed(seed)
        r = torch.rand(3, n[2], n[1], n[0], generator=g, dtype=torch.float64, device=device) * 2 - 1
    else:
        r = torch.stack([_waves(n, gen, 4, 8, device) for _ in range(3)])
    f = 0.1 * U * r
    one = torch.ones_like(f[0])
    return torch.stack([one, U + f[0], f[1], f[2], 100 / 1.4 * one])


def _primitive(case, cfg, seed):
    device = _device()
    if case["kind"] == "channel":
        return _channel(cfg, seed, not case["mass_flux"], device)
    if case["kind"] == "isotropic":
        return _isotropic(cfg, seed, case["k0"], case["mach"], device)
    return _vortex(cfg, seed, device)


def _conservative(prim, gamma=1.4):
    rho, u, v, w, p = prim
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (gamma - 1) + 0.5 * rho * (u * u + v * v + w * w)])


def _members(case, seed):
    """(configuration, primitive field) of every simulation of the case."""
    if case["do"] != "ensemble":
        cfg = _config(case, (case["nx"], case["ny"], case["nz"]))
        return [(cfg, _primitive(case, cfg, seed))]
    out = []
    for i, m in enumerate(int(s) for s in case["sizes"].split(",")):
        cfg = _config(case, (m, m, m))
        out.append((cfg, _primitive(case, cfg, 1000 * seed + i)))
    return out


def _fixed_dt(cfg, prim):
    """The fixed step of the adjoint cases: CFL 0.4 on the start's mean sound speed and largest velocity."""
    h = min(cfg.lx / cfg.nx, cfg.ly / cfg.ny, cfg.lz / cfg.nz)
    c0 = math.sqrt(1.4 * cfg.p_ref)
    return round(0.4 * h / (c0 * (1 + _mach_bound(prim, c0))), 6)


def _mach_bound(prim, c0):
    """Largest velocity component over c0, rounded up to a tenth."""
    return math.ceil(10 * float(prim[1:4].abs().max()) / c0) / 10


def _cotangent(shape, seed):
    gen = torch.Generator(device=_device()).manual_seed(seed + 77)
    return torch.randn(shape, generator=gen, dtype=torch.float64, device=_device())


def prepare(case, seed):
    members = _members(case, seed)
    sims = [Simulation(cfg) for cfg, _ in members]
    s = dict(case=case, sims=sims, prims=[p.contiguous() for _, p in members])
    if case["tuned"]:
        sims[0].init_primitive(s["prims"][0])
        sims[0].step(1)
        sims[0].autotune()
    if case["do"] == "ensemble":
        s["ens"] = Ensemble(sims)
    if case["do"] in ("adjoint", "window"):
        s["q"] = _conservative(s["prims"][0])
        s["dt"] = _fixed_dt(*members[0])
    if case["do"] == "adjoint":
        s["lam"] = _cotangent(s["q"].shape, seed)
    return s


# --------------------------------------------------------------------- run ---

def _fields(q, prec):
    """A conservative state as the run's snapshot: density, momentum, energy in the run's precision."""
    t = torch.float32 if prec == "fp32" else torch.float64
    return {"rho": q[0].to(t), "momentum": q[1:4].to(t), "energy": q[4].to(t)}


def run(state):
    case, sims = state["case"], state["sims"]
    prec, do = case["prec"], case["do"]
    if do == "steps":
        sims[0].init_primitive(state["prims"][0])
        sims[0].step(case["steps"], sync=False)
        return _fields(sims[0].state(device=True), prec)
    if do == "ensemble":
        for sim, prim in zip(sims, state["prims"]):
            sim.init_primitive(prim)
        state["ens"].step(case["steps"], sync=False)
        return [_fields(sim.state(device=True), prec) for sim in sims]
    if do == "adjoint":
        sims[0].init_conservative(state["q"])
        out = torch.empty_like(state["lam"])
        sims[0].adjoint_step(state["dt"], state["lam"], out)
        return out.to(torch.float32 if prec == "fp32" else torch.float64)
    q0 = state["q"].detach().clone().requires_grad_(True)
    q1 = run_window(q0, sims[0], case["steps"], state["dt"], every=2)
    ek = kinetic_energy(q1, sims[0])
    (g,) = torch.autograd.grad(ek, q0)
    t = torch.float32 if prec == "fp32" else torch.float64
    return {"state": _fields(q1.detach(), prec), "gradient": g.to(t), "energy": ek.detach().to(t)}


# Floating-point operations of the closed forms per face, both stages of a
# step, halo excluded: reconstruction of the face fields, the two tangential
# passes and the flux at the four Gauss points.
_FLOPS = {("linear", "smooth"): 3600.0, ("weno-js", "smooth"): 10000.0, ("weno-z", "smooth"): 10700.0,
          ("linear", "full"): 20000.0, ("weno-js", "full"): 37500.0, ("weno-z", "full"): 39000.0}


def work(case):
    ns = [(case["nx"], case["ny"], case["nz"])]
    if case["do"] == "ensemble":
        ns = [(int(s),) * 3 for s in case["sizes"].split(",")]
    per_step = _FLOPS[case["recon"], case["flux"]] * (1.25 if case["char"] else 1.0)
    out = 4 if case["prec"] == "fp32" else 8
    flops = nbytes = 0.0
    for x, y, z in ns:
        cells = x * y * z
        faces = 3 * cells + x * y + y * z + z * x
        step = faces * per_step
        if case["do"] == "adjoint":  # a forward stage, and two stages recomputed and reversed at twice their cost
            flops, nbytes = flops + 3.5 * step, nbytes + cells * 5 * (8 + 8 + out)
        elif case["do"] == "window":  # forward, recomputation and the adjoint of every step
            flops, nbytes = flops + case["steps"] * 5.0 * step, nbytes + cells * 5 * (8 + 2 * out)
        else:
            flops, nbytes = flops + case["steps"] * step, nbytes + cells * 5 * (8 + out)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------- the scheme in 64-bit torch ---

def exact(case, seed):
    members = _members(case, seed)
    if case["do"] == "adjoint":
        cfg, prim = members[0]
        q = _conservative(prim).requires_grad_(True)
        q1 = _step(cfg, q, _fixed_dt(cfg, prim))
        return torch.autograd.grad(q1, q, _cotangent(q.shape, seed))[0]
    if case["do"] == "window":
        cfg, prim = members[0]
        dt = _fixed_dt(cfg, prim)
        q = _conservative(prim).requires_grad_(True)
        q1 = q
        for _ in range(case["steps"]):
            q1 = _step(cfg, q1, dt)
        ek = (0.5 * (q1[1] ** 2 + q1[2] ** 2 + q1[3] ** 2) / q1[0]).mean() / cfg.rho_ref
        (g,) = torch.autograd.grad(ek, q)
        return {"state": _fields(q1.detach(), "fp64"), "gradient": g, "energy": ek.detach()}
    outs = []
    for cfg, prim in members:
        q = _conservative(prim)
        with torch.no_grad():
            for _ in range(case["steps"]):
                q = _step(cfg, q, None)
        outs.append(_fields(q, "fp64"))
    return outs if case["do"] == "ensemble" else outs[0]


def _widths(cfg, d, device):
    """Cell widths along axis d with three ghost cells a side; Sec. 3.3's tanh mapping in y, mirrored at the walls."""
    n, L = ((cfg.nx, cfg.lx), (cfg.ny, cfg.ly), (cfg.nz, cfg.lz))[d]
    if d != 1 or not cfg.y_stretch:
        return torch.full((n + 6,), L / n, dtype=torch.float64, device=device)
    eta = torch.arange(n + 1, dtype=torch.float64, device=device) * (3 * math.pi / n)
    y = torch.tanh(cfg.stretch_b * (eta / (1.5 * math.pi) - 1)) / math.tanh(cfg.stretch_b)
    w = y[1:] - y[:-1]
    return torch.cat([w[:3].flip(0), w, w[-3:].flip(0)])


def _prims(q, cfg):
    inv = 1 / q[0]
    u = [q[1] * inv, q[2] * inv, q[3] * inv]
    p = (cfg.gamma - 1) * (q[4] - 0.5 * q[0] * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
    return q[0], u, p


def _ghosts(q, cfg):
    """Three ghost cells on every side: periodic, or isothermal no-slip walls in y."""
    q = torch.cat([q[..., -3:], q, q[..., :3]], -1)
    if cfg.bc_y:
        def wall(m):
            rho, u, p = _prims(m, cfg)
            T = torch.clamp(2 * cfg.T_wall - p / rho, min=0.5 * cfg.T_wall)
            r = p / T
            return torch.stack([r, -r * u[0], -r * u[1], -r * u[2],
                                p / (cfg.gamma - 1) + 0.5 * r * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)])
        q = torch.cat([wall(q[:, :, :3].flip(2)), q, wall(q[:, :, -3:].flip(2))], 2)
    else:
        q = torch.cat([q[:, :, -3:], q, q[:, :, :3]], 2)
    return torch.cat([q[:, -3:], q, q[:, :3]], 1)


def _weno(q, mode):
    """WENO5 values at the left and right end of the centre cell from five averages."""
    def candidates(a, b, c, d, e):
        return ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
    a, b, c, d, e = q
    right, left = candidates(a, b, c, d, e), candidates(e, d, c, b, a)
    lin = (0.1, 0.6, 0.3)
    if mode == 0:
        return sum(w * p for w, p in zip(lin, left)), sum(w * p for w, p in zip(lin, right))
    beta = [13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2,
            13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2,
            13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2]
    if mode == 1:
        f = [1 / (1e-6 + x) ** 2 for x in beta]
    else:
        tau = (beta[0] - beta[2]).abs()
        f = [1 + tau / (x + 1e-20) for x in beta]

    def mix(p, f):
        w = [x * y for x, y in zip(lin, f)]
        return sum(x * y for x, y in zip(w, p)) / (w[0] + w[1] + w[2])
    return mix(left, f[::-1]), mix(right, f)


def _tangent(f, mode):
    """Values and derivatives (per cell) at the two Gauss abscissae -+1/(2 sqrt 3) of the centre face."""
    s3 = math.sqrt(3.0)
    f0, f1, f2, f3, f4 = f
    if mode == 0:  # the quartic through five averages
        even = 719 / 720 * f2 + (f1 + f3) / 1080 - (f0 + f4) / 4320
        odd = s3 * (7 / 432 * (f0 - f4) + 25 / 216 * (f3 - f1))
        slope = (f0 - f4) / 12 + 2 / 3 * (f3 - f1)
        curve = s3 / 54 * (13 * (f1 + f3) - 24 * f2 - f0 - f4)
        return (even - odd, even + odd), (slope - curve, slope + curve)
    left, right = _weno(f, mode)  # the quadratic through the end values and the average
    b, c = right - left, 3 * (left + right) - 6 * f2
    return (f2 - b / (2 * s3), f2 + b / (2 * s3)), (b - c / s3, b + c / s3)


class _Waves:
    """Left and right eigenvectors of the Euler Jacobian along the normal at the state q (Remark 1)."""

    def __init__(self, q, cfg):
        rho, (self.u, self.v, self.w), p = _prims(q, cfg)
        c2 = cfg.gamma * p / rho
        self.c = torch.sqrt(c2)
        self.ke = 0.5 * (self.u ** 2 + self.v ** 2 + self.w ** 2)
        self.H = (q[4] + p) / rho
        self.b1 = (cfg.gamma - 1) / c2

    def to(self, q):
        a = self.b1 * (self.ke * q[0] - self.u * q[1] - self.v * q[2] - self.w * q[3] + q[4])
        s = (self.u * q[0] - q[1]) / self.c
        return torch.stack([0.5 * (a + s), q[0] - a, q[2] - self.v * q[0], q[3] - self.w * q[0], 0.5 * (a - s)])

    def back(self, o):
        m, d = o[0] + o[1] + o[4], (o[4] - o[0]) * self.c
        return torch.stack([m, self.u * m + d, self.v * m + o[2], self.w * m + o[3],
                            self.H * (o[0] + o[4]) + self.ke * o[1] + self.u * d + self.v * o[2] + self.w * o[3]])


def _moments(rho, u, p, half):
    """<u^n>, <v^n>, <w^n> of the Maxwellian (n <= 6), <u^n> over u > 0 (half = 1) or u < 0 (-1)."""
    th = p / rho
    if half == 0:
        mu = [torch.ones_like(th), u[0]]
    else:
        x = u[0] / torch.sqrt(2 * th)
        m0 = 0.5 * torch.special.erfc(-half * x)
        mu = [m0, u[0] * m0 + half * torch.sqrt(th / (2 * math.pi)) * torch.exp(-x * x)]
    ms = [mu, [torch.ones_like(th), u[1]], [torch.ones_like(th), u[2]]]
    for m, c in zip(ms, u):
        for k in range(5):
            m.append(c * m[k + 1] + (k + 1) * th * m[k])
    return ms


def _inner(N, th):
    """<xi^2>, <xi^4> of N internal degrees of freedom."""
    return N * th, N * (N + 2) * th * th


def _psi(m, x, i, j, k):
    """<u^i v^j w^k psi>, psi = (1, u, v, w, (|u|^2 + xi^2)/2)."""
    def M(a, b, c):
        return m[0][a] * m[1][b] * m[2][c]
    base = M(i, j, k)
    return torch.stack([base, M(i + 1, j, k), M(i, j + 1, k), M(i, j, k + 1),
                        0.5 * (M(i + 2, j, k) + M(i, j + 2, k) + M(i, j, k + 2) + base * x[0])])


def _apsi(m, x, a, i, j, k):
    """<(a . psi) u^i v^j w^k psi>."""
    xi = x[0] * _psi(m, x, i, j, k)
    xi = torch.cat([xi[:4], (xi[4] + 0.5 * (x[1] - x[0] ** 2) * m[0][i] * m[1][j] * m[2][k])[None]])
    quad = _psi(m, x, i + 2, j, k) + _psi(m, x, i, j + 2, k) + _psi(m, x, i, j, k + 2) + xi
    return (a[0] * _psi(m, x, i, j, k) + a[1] * _psi(m, x, i + 1, j, k) + a[2] * _psi(m, x, i, j + 1, k) +
            a[3] * _psi(m, x, i, j, k + 1) + 0.5 * a[4] * quad)


def _slope(b, u, th, N):
    """a with <(a . psi) psi> = b for the Maxwellian at (u, theta)."""
    q2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    e = 2 * (b[4] - u[0] * b[1] - u[1] * b[2] - u[2] * b[3]) + (q2 - (N + 3) * th) * b[0]
    a4 = e / ((N + 3) * th * th)
    a1, a2, a3 = ((b[1 + k] - u[k] * b[0]) / th - u[k] * a4 for k in range(3))
    a0 = b[0] - u[0] * a1 - u[1] * a2 - u[2] * a3 - 0.5 * a4 * (q2 + (N + 3) * th)
    return torch.stack([a0, a1, a2, a3, a4])


def _signed(q, cfg, N):
    """int sign(u) psi g of the Maxwellian of q."""
    rho, u, p = _prims(q, cfg)
    x = _inner(N, p / rho)
    plus, minus = _moments(rho, u, p, 1), _moments(rho, u, p, -1)
    return rho * (_psi(plus, x, 0, 0, 0) - _psi(minus, x, 0, 0, 0))


def _time_fit(tau, dt):
    """Coefficients of F and dF (Eq. (7)) of the six time integrals of Eq. (5)."""
    def integrals(t):
        e = -torch.expm1(-t / tau)  # 1 - exp(-t/tau)
        E = torch.exp(-t / tau)
        return [t - tau * e, 2 * tau ** 2 * e - tau * t * E - tau * t, 0.5 * t * t - tau * t + tau ** 2 * e,
                tau * e, tau * t * E - 2 * tau ** 2 * e, -tau ** 2 * e]
    W, Wh = integrals(dt), integrals(0.5 * dt)
    return [(4 * h - w) / dt for w, h in zip(W, Wh)], [4 * (w - 2 * h) / dt ** 2 for w, h in zip(W, Wh)]


def _parts(q, dq, cfg, N, half):
    """rho <u psi>, rho <u (a.u) psi>, rho <u A psi> over the (half) velocity space."""
    rho, u, p = _prims(q, cfg)
    th = p / rho
    x = _inner(N, th)
    a = [_slope(d / rho, u, th, N) for d in dq]
    m = _moments(rho, u, p, 0)
    A = _slope(-(_apsi(m, x, a[0], 1, 0, 0) + _apsi(m, x, a[1], 0, 1, 0) + _apsi(m, x, a[2], 0, 0, 1)), u, th, N)
    if half:
        m = _moments(rho, u, p, half)
    au = _apsi(m, x, a[0], 2, 0, 0) + _apsi(m, x, a[1], 1, 1, 0) + _apsi(m, x, a[2], 1, 0, 1)
    return (rho * _psi(m, x, 1, 0, 0), rho * au, rho * _apsi(m, x, A, 1, 0, 0)), rho, u, p, th


def _flux(states, cfg, N, dt):
    """F and dF at Gauss points: the smooth flux of states[0], or the full flux of (l, r, 0)."""
    q, dq = states[-1]
    V, rho, u, p, th = _parts(q, dq, cfg, N, 0)
    mu = cfg.mu_ref * (th / cfg.T_ref) ** cfg.visc_exp if cfg.visc else torch.full_like(th, cfg.mu_ref)
    tau = mu / p
    if cfg.flux == 0:
        F, dF = V[0] - tau * (V[1] + V[2]), V[2]
    else:
        Vl, _, _, pl, _ = _parts(*states[0], cfg, N, 1)
        Vr, _, _, pr, _ = _parts(*states[1], cfg, N, -1)
        tau = tau + cfg.tau_num_C * ((pl - pr) / (pl + pr)).abs() * dt
        terms = list(V) + [l + r for l, r in zip(Vl, Vr)]
        cf, cd = _time_fit(tau, dt)
        F, dF = sum(c * t for c, t in zip(cf, terms)), sum(c * t for c, t in zip(cd, terms))
    # Prandtl fix: (1/Pr - 1) of the heat flux -tau p c_p dT/dn.
    d = dq[0]
    dp = (cfg.gamma - 1) * (d[4] - u[0] * d[1] - u[1] * d[2] - u[2] * d[3] +
                            0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) * d[0])
    heat = -(1 / cfg.prandtl - 1) * tau * p * 0.5 * (N + 5) * (dp - th * d[0]) / rho
    return torch.cat([F[:4], (F[4] + heat)[None]]), dF


def _face_fluxes(q, wn, w1, w2, cfg, dt):
    """F and dF of every face along the last axis of q [5][t2 + 4][t1 + 4][n + 6] (local frame)."""
    N = (5 - 3 * cfg.gamma) / (cfg.gamma - 1)
    mode = cfg.recon
    nf = q.shape[-1] - 5
    c = [q[..., k:k + nf] for k in range(6)]  # cells f-3 .. f+2
    hl, hr = wn[2:2 + nf], wn[3:3 + nf]
    char = cfg.recon_vars == 1 and mode != 0
    qm = 0.5 * (c[2] + c[3])
    if char:
        basis = _Waves(qm, cfg)
        o = [basis.to(x) for x in c]
        (Ll, Rl), (Lr, Rr) = (map(basis.back, _weno(o[k:k + 5], mode)) for k in (0, 1))
    else:
        (Ll, Rl), (Lr, Rr) = _weno(c[:5], mode), _weno(c[1:], mode)
    q0 = 0.5 * (Rl + Lr) + 0.5 * (_signed(Rl, cfg, N) - _signed(Lr, cfg, N))
    d0 = (c[1] - 15 * c[2] + 15 * c[3] - c[4]) / (6 * (hl + hr))
    fields = [(q0, d0)]
    if cfg.flux:
        dl = (4 * Rl + 2 * Ll - 6 * c[2]) / hl
        dr = -(4 * Lr + 2 * Rr - 6 * c[3]) / hr
        fields = [(Rl, dl), (Lr, dr)] + fields

    def window(f, axis):
        m = f.shape[axis] - 4
        return [f.narrow(axis, k, m) for k in range(5)]

    def tangent(f, axis, basis):
        f = window(f, axis)
        if basis is None:
            return _tangent(f, mode)
        v, d = _tangent([basis.to(x) for x in f], mode)
        return [basis.back(x) for x in v], [basis.back(x) for x in d]

    b1 = _Waves(qm[:, :, 2:-2], cfg) if char else None
    b2 = _Waves(qm[:, 2:-2, 2:-2], cfg) if char else None
    along1 = [(tangent(v, 2, b1), tangent(d, 2, b1)[0]) for v, d in fields]
    F = dF = 0
    for g1 in range(2):
        along2 = []
        for (v, d1), dn in along1:
            v2, d2 = tangent(v[g1], 1, b2)
            along2.append((v2, tangent(dn[g1], 1, b2)[0], tangent(d1[g1], 1, b2)[0], d2))
        for g2 in range(2):
            states = [(v[g2], (dn[g2], d1[g2] / w1[:, None], d2[g2] / w2[:, None, None]))
                      for v, dn, d1, d2 in along2]
            f, df = _flux(states, cfg, N, dt)
            F, dF = F + 0.25 * f, dF + 0.25 * df
    return F, dF


def _rates(q, cfg, dt):
    """L and dL (Eq. (4)) of the interior cells from the state with ghosts."""
    device = q.device
    n = (cfg.nx, cfg.ny, cfg.nz)
    L = dL = 0
    for d, perm in enumerate(((0, 1, 2, 3), (0, 3, 1, 2), (0, 2, 3, 1))):  # to [v][t2][t1][n]
        t1, t2 = (d + 1) % 3, (d + 2) % 3
        comp = [0, 1 + d, 1 + t1, 1 + t2, 4]
        local = q.permute(perm)[comp][:, 1:-1, 1:-1]
        w = [_widths(cfg, a, device) for a in (d, t1, t2)]
        rows = max(1, int(4e6) // ((n[d] + 1) * n[t1]))
        parts = []
        for r0 in range(0, n[t2], rows):
            r1 = min(r0 + rows, n[t2])
            args = (local[:, r0:r1 + 4], w[0], w[1][3:-3], w[2][3 + r0:3 + r1], cfg, dt)
            F, dF = checkpoint(_face_fluxes, *args, use_reentrant=False) if q.requires_grad else _face_fluxes(*args)
            h = w[0][3:-3]
            parts.append(torch.stack([-(x[..., 1:] - x[..., :-1]) / h for x in (F, dF)]))
        both = torch.cat(parts, 2)
        inv = [comp.index(k) for k in range(5)]
        back = [0, 1] + [perm.index(k) + 1 for k in (1, 2, 3)]
        both = both[:, inv].permute(back)
        L, dL = L + both[0], dL + both[1]
    return L, dL


def _step(cfg, q, dt):
    """One S2O4 step (Eq. (6)) of the conservative state; dt None takes the CFL step."""
    w = [_widths(cfg, d, q.device)[3:-3] for d in range(3)]
    if dt is None:
        rho, u, p = _prims(q, cfg)
        c = torch.sqrt(cfg.gamma * p / rho)
        h = (w[0][None, None, :], w[1][None, :, None], w[2][:, None, None])
        dt = cfg.cfl * float(min((hd / (ud.abs() + c)).min() for hd, ud in zip(h, u)))
    L, dL = _rates(_ghosts(q, cfg), cfg, dt)
    _, dLs = _rates(_ghosts(q + dt / 2 * L + dt * dt / 8 * dL, cfg), cfg, dt)
    q1 = q + dt * L + dt * dt / 6 * (dL + 2 * dLs)
    if cfg.force_mode == 0 and cfg.force_x == 0:
        return q1
    fx = cfg.force_x
    if cfg.force_mode:
        vol = w[0][None, None, :] * w[1][None, :, None] * w[2][:, None, None]
        fx = (cfg.mass_flux * vol.sum() - (q1[1] * vol).sum()) / (dt * (0.5 * (q[0] + q1[0]) * vol).sum())
    m = q1[1] + 0.5 * dt * (q1[0] + q[0]) * fx
    E = q1[4] + 0.5 * dt * (m + q[1]) * fx
    return torch.stack([q1[0], m, q1[2], q1[3], E])
