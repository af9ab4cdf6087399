"""The work that users of this framework have it do, as measurable cases.

A case names a call (``kind``), a grid, an initial field and the options of the context.  The
kinds are the public entry points a program calls in its inner loop: one right-hand side, one
Runge-Kutta step with the statistics logged on the device, one step with the time step taken
from the CFL number, one step of a state in host memory, one vector-Jacobian product, the
gradient of a final-time functional through a checkpointed trajectory, and one step of an
ensemble of uneven grids.  ``exact`` evaluates the same operators in plain torch FP64.
"""
from __future__ import annotations

import math

import torch

from paper_2211_16718_gb300 import autograd as A
from paper_2211_16718_gb300 import ns3d

GAMMA, PRANDTL, EPS, HARTEN = 1.4, 0.72, 1e-6, 0.1
MU_HIT = 0.003            # decaying turbulence at Re_lambda 50 (rho = 1, u0 = 0.3, k0 = 4)
L = 2.0 * math.pi
PRECISION = {"fp64": ns3d.NS3D_FP64, "fp32": ns3d.NS3D_FP32_BULK, "strict": ns3d.NS3D_FP64_STRICT}
STORAGE = {"auto": ns3d.NS3D_STORAGE_AUTO, "lean": ns3d.NS3D_STORAGE_LEAN}
ENSEMBLE_SIZES = (32, 48, 64, 96, 128)


def _case(kind, nx, ny, nz, field="hit", mu=MU_HIT, precision="fp64", rk="rk4", **more):
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, field=field, mu=mu, precision=precision, rk=rk, **more)


def listed():
    return [
        # one Euler right-hand side of a small shock tube: a library call inside another code's
        # time loop, where launches and latency count; odd sizes, strong jumps
        dict(_case("rhs", 40, 25, 18, field="sod", mu=0.0), name="sod_rhs_small"),
        # the 32^3 Taylor-Green box, KE and enstrophy logged every step
        dict(_case("step", 32, 32, 32, field="tgv", mu=0.1 / 1600), name="tgv32_rk4_step"),
        # a flat ragged box with lean viscous storage, SSP-RK3, adaptive time step
        dict(_case("cfl_step", 100, 75, 50, rk="ssprk3", storage="lean"), name="ragged_lean_cfl_step"),
        # the all-FP64 form, used to check the other modes
        dict(_case("step", 96, 96, 96, precision="strict", rk="ssprk3"), name="hit96_strict_ssprk3_step"),
        # decaying turbulence at the sizes of everyday runs, statistics every step
        dict(_case("step", 128, 128, 128), name="hit128_rk4_step"),
        dict(_case("step", 256, 256, 256), name="hit256_rk4_step"),
        # the largest plain FP64 grid of the configurations (5.4 GB state)
        dict(_case("step", 512, 512, 512), name="hit512_rk4_step"),
        # the FP32-bulk mode at the size it is compared at
        dict(_case("step", 512, 512, 512, precision="fp32"), name="hit512_fp32bulk_rk4_step"),
        # a host code that keeps the state in pinned memory and calls in once per step
        dict(_case("host_step", 192, 192, 192), name="hit192_host_step"),
        # one linearisation, as an outer optimiser or a Krylov method calls it
        dict(_case("vjp", 128, 128, 128), name="hit128_rhs_vjp"),
        # gradient of the final kinetic energy through a checkpointed trajectory (64^3, Re 400)
        dict(_case("gradient", 64, 64, 64, field="tgv", mu=0.1 / 400, nsteps=4, every=2), name="tgv64_ke_gradient"),
        # 48 independent realisations of uneven sizes, graph schedule
        dict(_case("ensemble", 32, 128, 128, count=48), name="ensemble48_step"),
    ]


def _size(rng, lo, hi):
    """Log-uniform size in [lo, hi], a multiple of 8 in one case out of three."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, n // 8 * 8) if rng.random() < 0.33 else n


def draw(rng):
    kind = rng.choice(["rhs", "rhs", "step", "step", "step", "cfl_step", "strict", "fp32", "host_step", "vjp",
                       "gradient", "ensemble"])
    rk = rng.choice(["rk4", "ssprk3"])
    if kind == "ensemble":
        lo = _size(rng, 12, 48)
        hi = _size(rng, lo, 128)
        return _case("ensemble", lo, hi, hi, rk=rk, count=rng.randint(4, 48))
    if kind == "gradient":
        n = [_size(rng, 20, 64) for _ in range(3)]
        return _case("gradient", *n, field=rng.choice(["tgv", "hit"]), mu=0.1 / 400, rk=rk, nsteps=rng.randint(2, 4),
                     every=rng.randint(1, 3))
    if kind == "host_step":
        return _case("host_step", _size(rng, 24, 256), _size(rng, 24, 256), _size(rng, 24, 256), rk=rk)
    if kind == "strict":
        n = [_size(rng, 16, 128) for _ in range(3)]
        return _case("step", *n, precision="strict", rk=rk)
    if kind == "vjp":
        return _case("vjp", *[_size(rng, 12, 160) for _ in range(3)], mu=rng.choice([0.0, MU_HIT]))
    if kind == "rhs":
        field = rng.choice(["sod", "hit"])
        return _case("rhs", *[_size(rng, 8, 256) for _ in range(3)], field=field,
                     mu=rng.choice([0.0, MU_HIT]) if field == "hit" else 0.0)
    more = {"storage": rng.choice(["auto", "lean"])}
    return _case("step" if kind == "fp32" else kind, *[_size(rng, 16, 384) for _ in range(3)], rk=rk,
                 precision="fp32" if kind == "fp32" else "fp64", **more)


# ---- inputs ---------------------------------------------------------------------------------
def _mesh(nx, ny, nz):
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") * (L / n) for n in (nz, ny, nx)]
    return ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]


def _conserved(rho, vel, p):
    u = torch.empty((5,) + tuple(vel[0].shape), dtype=torch.float64, device="cuda")
    u[0] = rho
    for m in range(3):
        u[1 + m] = rho * vel[m]
    u[4] = p / (GAMMA - 1.0) + 0.5 * rho * (vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2)
    return u


def _hit(nx, ny, nz, gen, u0=0.3, k0=4.0):
    """Solenoidal random-phase velocity with E(k) ~ k^4 exp(-2 (k/k0)^2), RMS u0; rho = 1, p = 1/gamma."""
    kz = torch.fft.fftfreq(nz, 1.0 / nz, dtype=torch.float64, device="cuda")[:, None, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device="cuda")[None, :, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, dtype=torch.float64, device="cuda")[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    amp = torch.sqrt(k2) * torch.exp(-k2 / (k0 * k0))  # sqrt(E(k)) / k, up to a factor
    for k, n in ((kx, nx), (ky, ny), (kz, nz)):  # the Nyquist modes carry no direction
        amp = torch.where((2 * k.abs() >= n).expand(amp.shape), torch.zeros((), dtype=amp.dtype, device="cuda"), amp)
    uh = [torch.fft.rfftn(torch.randn((nz, ny, nx), dtype=torch.float64, device="cuda", generator=gen)) for _ in range(3)]
    div = (kx * uh[0] + ky * uh[1] + kz * uh[2]) / torch.where(k2 > 0, k2, torch.ones((), dtype=k2.dtype, device="cuda"))
    vel = []
    for m, k in enumerate((kx, ky, kz)):
        vel.append(torch.fft.irfftn((uh[m] - k * div) * amp, s=(nz, ny, nx)))
        uh[m] = None
    rms = math.sqrt(sum(float((v * v).mean()) for v in vel) / 3.0)
    for v in vel:
        v.mul_(u0 / max(rms, 1e-30))
    return _conserved(1.0, vel, 1.0 / GAMMA)


def _tgv(nx, ny, nz, gen, v0=0.1):
    """Taylor-Green vortex, isothermal, moved by a random phase (off the grid's symmetry planes)
    with a random smooth perturbation of 1 % that breaks its symmetry."""
    Z, Y, X = _mesh(nx, ny, nz)
    r = torch.rand(64, dtype=torch.float64, device="cuda", generator=gen).cpu().tolist()
    X, Y, Z = X + L * r[0], Y + L * r[1], Z + L * r[2]

    def ripple(at):
        f = 0.0
        for j in range(3):
            k = [1 + int(3 * r[at + 5 * j + d]) for d in range(3)]
            f = f + (r[at + 5 * j + 3] - 0.5) * torch.sin(k[0] * X + k[1] * Y + k[2] * Z + L * r[at + 5 * j + 4])
        return 0.01 * f

    vel = [v0 * (torch.sin(X) * torch.cos(Y) * torch.cos(Z) + ripple(3)),
           v0 * (-torch.cos(X) * torch.sin(Y) * torch.cos(Z) + ripple(18)), v0 * ripple(33)]
    p = 1.0 / GAMMA + (v0 * v0 / 16.0) * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0)
    return _conserved(GAMMA * p, vel, p)


def _sod(nx, ny, nz, gen):
    """Periodic shock tube along a random axis, its two jumps at random places, with a weak smooth
    disturbance so that no flux is constant across it."""
    Z, Y, X = _mesh(nx, ny, nz)
    r = torch.rand(16, dtype=torch.float64, device="cuda", generator=gen).cpu().tolist()
    s = (X, Y, Z)[int(3 * r[0])]
    left = torch.remainder(s + L * r[1], L) < 0.5 * L
    wave = 1.0 + 0.02 * torch.sin(X + L * r[2]) * torch.cos(Y + L * r[3]) * torch.cos(Z + L * r[4])
    one = torch.ones((), dtype=torch.float64, device="cuda")
    rho = torch.where(left, one, 0.125 * one) * wave
    p = torch.where(left, one / GAMMA, 0.1 * one / GAMMA) * wave
    vel = [0.1 * (wave - 1.0) * (m + 1) for m in range(3)]
    return _conserved(rho, vel, p)


def _field(case, seed, n=None):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    nx, ny, nz = n or (case["nx"], case["ny"], case["nz"])
    return {"hit": _hit, "tgv": _tgv, "sod": _sod}[case["field"]](nx, ny, nz, gen)


def _ensemble_grids(case):
    """Sizes of the ensemble's cubes: the five standard ones, or equal ratios between nx and ny."""
    if (case["nx"], case["ny"]) == (ENSEMBLE_SIZES[0], ENSEMBLE_SIZES[-1]):
        return [ENSEMBLE_SIZES[i % 5] for i in range(case["count"])]
    lo, hi = case["nx"], case["ny"]
    return [int(round(lo * (hi / lo) ** ((i % 5) / 4.0))) for i in range(case["count"])]


def _dt(u, cfl=0.4):
    return cfl / float(_wavespeed(u))


def _cotangent(u, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 104729 + 5)
    return torch.randn(u.shape, dtype=torch.float64, device="cuda", generator=gen)


def _options(case):
    return dict(mu_eff=case["mu"], precision=PRECISION[case["precision"]],
                rk=ns3d.NS3D_RK4 if case["rk"] == "rk4" else ns3d.NS3D_SSPRK3,
                storage=STORAGE[case.get("storage", "auto")])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        sizes = _ensemble_grids(case)
        states = [_field(case, 1000 * seed + i, (n, n, n)) for i, n in enumerate(sizes)]
        batch = ns3d.Batch([ns3d.default_params(n, n, n, **_options(case)) for n in sizes])
        batch.set_states(states)
        batch.set_dt([_dt(u) for u in states])
        return dict(kind=kind, batch=batch, states=states)
    u = _field(case, seed)
    s = dict(kind=kind, solver=ns3d.Solver(case["nx"], case["ny"], case["nz"], **_options(case)), u=u)
    if kind in ("step", "gradient", "host_step"):
        s["dt"] = _dt(u)
    if kind == "rhs":
        s["out"] = torch.empty_like(u)
    elif kind == "step":
        s["stats"] = torch.zeros(ns3d.NS3D_STATS_NDOUBLE, dtype=torch.float64, device="cuda")
    elif kind == "host_step":
        host = torch.empty(u.shape, dtype=torch.float64, pin_memory=True)
        host.copy_(u)
        s["u"], s["host"] = host.numpy(), host
    elif kind == "vjp":
        s["lam"], s["out"] = _cotangent(u, seed), torch.empty_like(u)
    elif kind == "gradient":
        s["nsteps"], s["every"] = case["nsteps"], case["every"]
    return s


def run(s):
    kind = s["kind"]
    if kind == "ensemble":
        s["batch"].step(1, "graph")
        return s["states"]
    solver, u = s["solver"], s["u"]
    if kind == "rhs":
        return solver.rhs(u, s["out"])
    if kind == "step":
        solver.rk_step(u, s["dt"], 1)
        return {"u": u, "stats": solver.stats_async(u, s["stats"])}
    if kind == "cfl_step":
        dt = solver.dt_from_cfl(u, 0.4)
        return {"u": solver.rk_step(u, dt, 1), "dt": dt}
    if kind == "host_step":
        stats = solver.step_host(u, s["dt"], 1)
        return {"u": s["host"], "stats": torch.tensor([stats[f] for f in ns3d.STATS_FIELDS], dtype=torch.float64)}
    if kind == "vjp":
        return solver.rhs_vjp(u, s["lam"], s["out"])
    u0 = u.detach().requires_grad_()
    ke = A.functional(A.trajectory(u0, solver, s["dt"], s["nsteps"], s["every"]), solver, "ke")
    (grad,) = torch.autograd.grad(ke, u0)
    return {"grad": grad, "ke": ke.detach()}


# ---- work and tolerances ---------------------------------------------------------------------
def work(case):
    """Bytes: every input read once, every output written once (states of five FP64 fields).
    Flops of the method per point: a right-hand side 3 x 735 (reconstruction and upwinding) + 260
    (primitives, gradients, viscous fluxes, divergence); a vector-Jacobian product about four
    times that; the statistics 60."""
    n = case["nx"] * case["ny"] * case["nz"]
    stages = 4 if case["rk"] == "rk4" else 3
    rhs, vjp, state = 3 * 735 + 260, 4 * (3 * 735 + 260), 5 * 8
    kind = case["kind"]
    if kind == "ensemble":
        n = sum(m ** 3 for m in _ensemble_grids(case))
    if kind == "rhs":
        return {"bytes": 2 * state * n, "flops": rhs * n}
    if kind == "vjp":
        return {"bytes": 3 * state * n, "flops": vjp * n}
    if kind == "gradient":  # forward steps, the recomputed stages of every step, one VJP per stage
        return {"bytes": 2 * state * n, "flops": case["nsteps"] * stages * (2 * rhs + vjp) * n}
    stats = 60 if kind in ("step", "cfl_step", "host_step") else 0
    return {"bytes": 2 * state * n, "flops": (stages * rhs + stats) * n}


def tolerance(case):
    # relative 2-norm and largest difference: four times the largest distance from exact() seen
    # over the listed cases and two dozen drawn ones
    if case["precision"] == "fp32":
        return {"rel": 5e-8, "max": 4e-7}
    if case["kind"] == "rhs":
        return {"rel": 1.3e-13, "max": 3.5e-12}
    if case["kind"] == "vjp":
        return {"rel": 3.3e-13, "max": 2e-11}
    if case["kind"] == "gradient":
        return {"rel": 3.5e-14, "max": 1.1e-12}
    if case["kind"] == "cfl_step":  # the time step comes from a double-float wave speed (48 bits)
        return {"rel": 9e-15, "max": 2.2e-14}
    return {"rel": 5e-15, "max": 2.2e-14}


# ---- the operators in plain torch FP64 ---------------------------------------------------------
def _prim(u):
    rho = u[0]
    vel = [u[1 + m] / rho for m in range(3)]
    p = (GAMMA - 1.0) * (u[4] - 0.5 * rho * (vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2))
    return rho, vel, p


def _wavespeed(u):
    rho, vel, p = _prim(u)
    c = torch.sqrt(GAMMA * p / rho)
    n = (u.shape[3], u.shape[2], u.shape[1])
    return max(float(((vel[d].abs() + c) / (L / n[d])).max()) for d in range(3))


def _weno(a, b, c, d, e):
    """Left-biased WENO5 value of the stencil a..e at the interface right of c."""
    b1 = 13.0 / 12.0 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    b2 = 13.0 / 12.0 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    b3 = 13.0 / 12.0 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    w1, w2, w3 = 0.1 / (EPS + b1) ** 2, 0.6 / (EPS + b2) ** 2, 0.3 / (EPS + b3) ** 2
    del b1, b2, b3
    q1 = (2 * a - 7 * b + 11 * c) / 6
    q2 = (-b + 5 * c + 2 * d) / 6
    q3 = (2 * c + 5 * d - e) / 6
    return (w1 * q1 + w2 * q2 + w3 * q3) / (w1 + w2 + w3)


def _both(q, dim):
    """Left- and right-biased values at the interface i + 1/2 of every point i."""
    s = [torch.roll(q, -j, dim) for j in range(-2, 4)]
    return _weno(*s[:5]), _weno(*s[:0:-1])


def _convective(u, D):
    """-(F_{i+1/2} - F_{i-1/2}) / dx along direction D (0 = x), Roe flux with Harten's fix."""
    dim = 2 - D
    h = L / u.shape[3 - D]
    nxt = lambda q: torch.roll(q, -1, dim)  # noqa: E731
    rho, vel, p = _prim(u)
    un = vel[D]
    f = [u[1 + D], u[1] * un, u[2] * un, u[3] * un, (u[4] + p) * un]
    f[1 + D] = f[1 + D] + p
    fs, du = [], []
    for v in range(5):
        a, b = _both(u[v], dim)
        du.append(b - a)
        if v == 1 + D:
            f0 = a + b
    for v in range(1, 5):
        a, b = _both(f[v], dim)
        fs.append(a + b)
    fs.insert(0, f0)
    sr, H = torch.sqrt(rho), (u[4] + p) / rho
    sb = nxt(sr)
    wa, wb = sr / (sr + sb), sb / (sr + sb)
    V = [wa * q + wb * nxt(q) for q in vel]
    Hr = wa * H + wb * nxt(H)
    q2 = 0.5 * (V[0] ** 2 + V[1] ** 2 + V[2] ** 2)
    c2 = (GAMMA - 1.0) * (Hr - q2)
    c = torch.sqrt(c2)
    t1, t2 = (1 if D == 0 else 0), (1 if D == 2 else 2)
    vn = V[D]
    phi = (GAMMA - 1.0) / c2 * (q2 * du[0] + du[4] - V[0] * du[1] - V[1] * du[2] - V[2] * du[3])
    ac = 0.5 * (vn * du[0] - du[1 + D]) / c
    a1, a5 = 0.5 * phi + ac, 0.5 * phi - ac
    a2, a3, a4 = du[0] - phi, du[1 + t1] - V[t1] * du[0], du[1 + t2] - V[t2] * du[0]
    dl = HARTEN * c

    def fix(lam):
        m = lam.abs()
        return torch.where(m < dl, (lam * lam + dl * dl) / (2 * dl), m)

    l1, l5, l2 = fix(vn - c), fix(vn + c), vn.abs()
    A1, A2, A3, A4, A5 = l1 * a1, l2 * a2, l2 * a3, l2 * a4, l5 * a5
    S, cD = A1 + A5, c * (A5 - A1)
    d0 = S + A2
    dis = [d0, None, None, None, S * Hr + cD * vn + A2 * q2 + A3 * V[t1] + A4 * V[t2]]
    dis[1 + D], dis[1 + t1], dis[1 + t2] = d0 * vn + cD, d0 * V[t1] + A3, d0 * V[t2] + A4
    out = []
    for v in range(5):
        F = 0.5 * (fs[v] - dis[v])
        out.append((torch.roll(F, 1, dim) - F) / h)
    return torch.stack(out)


def _d4(q, D):
    dim = q.dim() - 1 - D
    r = lambda j: torch.roll(q, -j, dim)  # noqa: E731
    return (8 * (r(1) - r(-1)) - (r(2) - r(-2))) / (12.0 * L / q.shape[dim])


def _viscous(u, mu):
    rho, vel, p = _prim(u)
    T = GAMMA * p / rho
    G = [[_d4(q, d) for d in range(3)] for q in vel]
    div = (G[0][0] + G[1][1] + G[2][2]) * (2.0 / 3.0)
    kap = mu / ((GAMMA - 1.0) * PRANDTL)
    out = [torch.zeros_like(rho)] + [0.0] * 4
    for d in range(3):
        tau = [mu * (G[m][d] + G[d][m] - (div if m == d else 0.0)) for m in range(3)]
        en = vel[0] * tau[0] + vel[1] * tau[1] + vel[2] * tau[2] + kap * _d4(T, d)
        for c, q in enumerate(tau + [en]):
            out[1 + c] = out[1 + c] + _d4(q, d)
    return torch.stack(out)


def _rhs(u, mu, part=lambda f, *a: f(*a)):
    """R(u); `part` wraps each direction (checkpointing under autograd)."""
    r = part(_convective, u, 0)
    r = r + part(_convective, u, 1)
    r = r + part(_convective, u, 2)
    return r + part(_viscous, u, mu) if mu > 0 else r


def _step(u, dt, case, part=lambda f, *a: f(*a)):
    R = lambda q: _rhs(q, case["mu"], part)  # noqa: E731
    if case["rk"] == "rk4":
        k = R(u)
        acc = k
        k = R(u + 0.5 * dt * k)
        acc = acc + 2 * k
        k = R(u + 0.5 * dt * k)
        acc = acc + 2 * k
        return u + (dt / 6) * (acc + R(u + dt * k))
    a = u + dt * R(u)
    b = 0.75 * u + 0.25 * (a + dt * R(a))
    return u / 3 + (2.0 / 3.0) * (b + dt * R(b))


def _stats(u):
    """The ten statistics of the library, its status word and the reserved slot."""
    rho, vel, p = _prim(u)
    n = (u.shape[3], u.shape[2], u.shape[1])
    vol = (L / n[0]) * (L / n[1]) * (L / n[2])
    wx = _d4(vel[2], 1) - _d4(vel[1], 2)
    wy = _d4(vel[0], 2) - _d4(vel[2], 0)
    wz = _d4(vel[1], 0) - _d4(vel[0], 1)
    ke = (0.5 * rho * (vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2)).mean()
    ens = (0.5 * rho * (wx ** 2 + wy ** 2 + wz ** 2)).mean()
    return [float(u[v].sum()) * vol for v in range(5)] + [float(ke), float(ens), float(rho.min()), float(p.min()),
                                                           float(_wavespeed(u)), 0.0, 0.0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        out = []
        for i, n in enumerate(_ensemble_grids(case)):
            u = _field(case, 1000 * seed + i, (n, n, n))
            out.append(_step(u, _dt(u), case))
        return out
    u = _field(case, seed)
    if kind == "rhs":
        return _rhs(u, case["mu"])
    if kind == "vjp":
        lam, grad = _cotangent(u, seed), torch.zeros_like(u)
        parts = [lambda q, d=d: _convective(q, d) for d in range(3)]
        if case["mu"] > 0:
            parts.append(lambda q: _viscous(q, case["mu"]))
        for f in parts:
            x = u.clone().requires_grad_()
            grad += torch.autograd.grad((f(x) * lam).sum(), x)[0]
        return grad
    if kind == "gradient":
        from torch.utils.checkpoint import checkpoint
        dt = _dt(u)
        x = u.clone().requires_grad_()
        q = x
        for _ in range(case["nsteps"]):
            q = _step(q, dt, case, lambda f, *a: checkpoint(f, *a, use_reentrant=False))
        ke = (0.5 * (q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / q[0]).mean()
        return {"grad": torch.autograd.grad(ke, x)[0], "ke": ke.detach()}
    dt = _dt(u)
    new = _step(u, dt, case)
    if kind == "cfl_step":
        return {"u": new, "dt": dt}
    st = _stats(new)
    if kind == "host_step":
        st = st[:len(ns3d.STATS_FIELDS)]
    return {"u": new, "stats": torch.tensor(st, dtype=torch.float64)}
