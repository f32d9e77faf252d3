"""The work this framework is measured on: one pass each through its public entry points.

A case is a dict of plain values.  `kind` names the loop it stands for:

  step     one exchange of a coupled flow solver: a new field in, `steps` particle steps, the sources and
           the particles out
  micro    the same with droplet microphysics: the vapour and energy sources too
  couple   a run of asynchronous two-way coupling from a given field: the new field, the sources still
           pending and the particles
  adjoint  the gradients of a loss of the time-summed sources: through autograd on an FP64 handle, through
           the handle's own calls on particles sorted once on an FP32 one

Particles are uniform in the box with lognormal diameters (median 20 um, geometric deviation 1.5), fields are
divergence-free random Fourier fields of rms 1 or a Taylor-Green vortex, as in the package's own workloads.
A handle of a mixed precision holds and computes its sources and gradients in FP32; the program that runs
one works on FP32 fields and takes them as such.
"""
from __future__ import annotations

import math

import torch

RHO_P, MU, GRAVITY = 1000.0, 1.8e-5, (0.0, 0.0, -9.81)
RHO_F = 1.2  # fluid density of the Reynolds number and of the coupled fluid
K = 10       # steps between sorts
# droplet microphysics: vapour diffusivity, conductivity, specific heat, latent heat, Prandtl number, least diameter
D_V, KAPPA, CP, LATENT, PRANDTL, D_MIN, T_INIT = 2.5e-5, 0.025, 4186.0, 2.5e6, 0.71, 1e-7, 285.0
NU, SWEEPS, INTERVAL = 1e-3, 10, 5  # coupled fluid: viscosity, Jacobi sweeps, particle steps per interval


def _case(name, kind, grid, n, steps, dt, precision, **more):
    c = dict(kind=kind, nx=grid[0], ny=grid[1], nz=grid[2], n=n, steps=steps, dt=dt, precision=precision, chunk=8,
             field="fourier", physics="default", vmax=0.0)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a solver that exchanges fields every step on a very small case: latency and launches
        _case("exchange_small", "step", (16, 16, 16), 3001, 1, 1e-3, "mixed_f32", field="taylor_green", vmax=1.0),
        # the FP64 reference run of the method on a small box (the default precision of a handle)
        _case("fp64_tg32", "step", (32, 32, 32), 100_000, 20, 1e-3, "fp64", field="taylor_green"),
        # FP64 at volume
        _case("fp64_128", "step", (128, 128, 128), 30_000_000, 10, 5e-4, "fp64"),
        # production: many particles per GPU in mixed precision, the largest case
        _case("mixed_256", "step", (256, 256, 256), 500_000_000, 10, 5e-4, "mixed_f32"),
        # the smaller storage form: BF16 velocities
        _case("bf16_128", "step", (128, 128, 128), 100_000_000, 10, 5e-4, "mixed_bf16"),
        # a box whose sides are no multiples of a chunk, an odd number of particles, 4 per cell
        _case("mixed_ragged", "step", (100, 84, 60), 2_000_003, 10, 1e-3, "mixed_f32", vmax=0.5),
        # the paper's own choices: nearest grid point, semi-implicit Euler, Schiller-Naumann drag
        _case("paper_128", "step", (128, 128, 128), 60_000_000, 10, 5e-4, "mixed_f32", physics="paper"),
        # sources that are continuous in the positions: cloud-in-cell deposit
        _case("cic_128", "step", (128, 128, 128), 20_000_000, 10, 5e-4, "mixed_f32", physics="cic"),
        # cloud droplets that grow and evaporate
        _case("micro_128", "micro", (128, 128, 128), 40_000_000, 10, 5e-4, "mixed_f32"),
        # two-way coupling on the device: two intervals of five steps
        _case("couple_128", "couple", (128, 128, 128), 60_000_000, 10, 5e-4, "mixed_f32", chunk=32),
        # calibration of diameters, drag and field in FP64 (through torch.autograd)
        _case("adjoint_fp64", "adjoint", (64, 64, 64), 2_000_000, 40, 1e-3, "fp64", field="tg_fourier", every=20),
        # the same in FP32, at volume
        _case("adjoint_fp32", "adjoint", (64, 64, 64), 10_000_000, 40, 1e-3, "mixed_f32", field="tg_fourier",
              every=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: kinds and options in the proportions of the listed ones, sizes over their logarithm."""
    what = rng.choice(["fp64", "fp64", "mixed", "mixed", "mixed", "bf16", "paper", "cic", "micro", "couple", "adjoint64",
                       "adjoint32"])
    if rng.random() < 0.4:
        grid = tuple(_log(rng, 12, 160) for _ in range(3))  # any sides
        chunk = rng.choice([4, 8, 16])
    else:
        chunk = rng.choice([8, 8, 16, 32])
        grid = tuple(max(16, chunk * max(1, round(_log(rng, 16, 192) / chunk))) for _ in range(3))
    dt = rng.choice([5e-4, 1e-3])
    steps = rng.choice([1, 2, 5, 7, 10, 20])
    vmax = rng.choice([0.0, 0.0, 0.5, 1.0])
    more = dict(chunk=chunk, vmax=vmax)
    if what == "fp64":
        n = _log(rng, 1e3, 2e8 / steps / 2)
        return _case(None, "step", grid, n, steps, dt, "fp64", physics=rng.choice(["default", "default", "cic"]), **more)
    if what in ("mixed", "bf16"):
        return _case(None, "step", grid, _log(rng, 2e3, min(2e8, 1e9 / steps)), steps, dt,
                     "mixed_f32" if what == "mixed" else "mixed_bf16", **more)
    if what in ("paper", "cic"):
        return _case(None, "step", grid, _log(rng, 1e4, 3e8 / steps), steps, dt, "mixed_f32", physics=what, **more)
    if what == "micro":
        prec = rng.choice(["mixed_f32", "mixed_f32", "mixed_bf16", "fp64"])
        return _case(None, "micro", grid, _log(rng, 1e4, (5e7 if prec == "fp64" else 4e8) / steps), steps, dt, prec, **more)
    if what == "couple":
        prec = rng.choice(["mixed_f32", "mixed_f32", "fp64"])
        steps = INTERVAL * rng.choice([1, 2, 4])
        return _case(None, "couple", grid, _log(rng, 1e4, (1e8 if prec == "fp64" else 1e9) / steps), steps, dt, prec, **more)
    steps = rng.choice([7, 20, 50])
    every = rng.choice([5, 10, 20])
    if what == "adjoint64":
        return _case(None, "adjoint", grid, _log(rng, 1e3, 5e7 / steps), steps, dt, "fp64", every=every,
                     physics=rng.choice(["default", "default", "cic"]), **more)
    return _case(None, "adjoint", grid, _log(rng, 1e3, 2e8 / steps), steps, dt, "mixed_f32", every=every, **more)


# ---- inputs --------------------------------------------------------------------------------------------

def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _box(case):
    n = _grid(case)
    return tuple(q / max(n) for q in n)  # cubic cells, the longest side 1


def _fourier(n, gen, comps=3, kmax=8):
    """Random Fourier field of rms 1 at the cell centres [nz, ny, nx, comps], divergence-free for three."""
    nx, ny, nz = n
    kx, ky, kz = (torch.arange(-min(kmax, (m - 1) // 2), min(kmax, (m - 1) // 2) + 1, device="cuda") for m in n)
    Kz, Ky, Kx = torch.meshgrid(kz, ky, kx, indexing="ij")
    k = torch.stack([Kx, Ky, Kz]).double()
    kn = k.square().sum(0).sqrt()
    keep = (kn >= 1) & (kn <= kmax)
    kn = torch.where(keep, kn, torch.ones_like(kn))
    amp = torch.where(keep, kn ** (-11.0 / 6.0), torch.zeros_like(kn))
    c = torch.randn((comps, *kn.shape, 2), generator=gen, device="cuda", dtype=torch.float64)
    c = torch.view_as_complex(c) * amp
    if comps == 3:
        c = c - k * ((c * k).sum(0) / kn.square())
    spec = torch.zeros((comps, nz, ny, nx), dtype=torch.complex128, device="cuda")
    spec[:, (kz % nz)[:, None, None], (ky % ny)[None, :, None], (kx % nx)[None, None, :]] = c
    u = torch.fft.ifftn(spec, dim=(1, 2, 3)).real
    u = u / u.square().mean().sqrt()
    return u.permute(1, 2, 3, 0).contiguous()


def _taylor_green(n):
    z, y, x = torch.meshgrid(*((torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * (2 * math.pi / m)
                               for m in (n[2], n[1], n[0])), indexing="ij")
    return torch.stack([x.sin() * y.cos() * z.cos(), -x.cos() * y.sin() * z.cos(), torch.zeros_like(x)], -1)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, N, box = case["n"], _grid(case), _box(case)
    if case["field"] == "taylor_green":
        U = _taylor_green(N) * (0.8 + 0.4 * torch.rand((), generator=gen, device="cuda", dtype=torch.float64))
    elif case["field"] == "tg_fourier":
        U = _taylor_green(N) + (0.1 / math.sqrt(8.0)) * _fourier(N, gen)
    else:
        U = _fourier(N, gen)
    f64 = case["precision"] == "fp64"
    d = dict(U=U if f64 else U.float())
    pos = torch.rand((3, n), generator=gen, device="cuda", dtype=torch.float64)
    for q in range(3):
        pos[q] *= box[q]
    d["pos"] = pos
    # the tails are cut at 4.3 geometric deviations
    g = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64).clamp_(-4.3, 4.3)
    d["d"] = g.mul_(math.log(1.5)).exp_().mul_(20e-6)
    d["vel"] = None
    if case["vmax"]:
        d["vel"] = torch.rand((3, n), generator=gen, device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0).mul_(case["vmax"])
    if case["kind"] == "micro":
        F = _fourier(N, gen, comps=2)
        # chamber air near water saturation
        d["T"] = (285.0 + 3.0 * F[..., 0]).contiguous()
        d["rv"] = (0.0105 * (1.0 + 0.05 * F[..., 1])).contiguous()
    if case["kind"] == "adjoint":
        # dL/dJ of a fit that is off by a trend and by noise
        d["lam"] = 1.0 + 0.5 * torch.randn((3, N[0] * N[1] * N[2]), generator=gen, device="cuda", dtype=torch.float64)
        if not f64:
            d["lam"] = d["lam"].float()
    return d


PHYSICS = {
    "default": dict(),
    "paper": dict(gather="ngp", integrator="semi_implicit", drag="schiller_naumann", rho_f=RHO_F),
    "cic": dict(deposit="cic"),
}


def prepare(case, seed):
    from paper_2603_26691_gb300.sim import Sim

    data = _inputs(case, seed)
    sim = Sim(_grid(case), box=_box(case), chunk_edge=case["chunk"], precision=case["precision"])
    sim.set_params(rho_p=RHO_P, mu=MU, g=GRAVITY, reorder_every=K)
    if case["physics"] != "default":
        sim.set_physics(**PHYSICS[case["physics"]])
    s = dict(case=case, sim=sim, U=data["U"])
    if case["kind"] == "adjoint":
        s.update(pos=data["pos"], vel=data["vel"], lam=data["lam"], d=data["d"])
        if case["precision"] == "fp64":
            s.update(d=data["d"].requires_grad_(), U=data["U"].requires_grad_(),
                     alpha=torch.ones((), dtype=torch.float64, requires_grad=True))
        else:
            sim.set_fluid(data["U"])
        return s
    sim.reserve(case["n"])
    sim.add_particles(data["pos"], data["d"], data["vel"])
    if case["kind"] == "micro":
        sim.set_microphysics(True, D_v=D_V, kappa_f=KAPPA, cp_p=CP, latent_heat=LATENT, prandtl=PRANDTL, d_min=D_MIN,
                             T_init=T_INIT)
        sim.set_thermo(data["T"], data["rv"])
    if case["kind"] == "couple":
        sim.couple_params(rho_f=RHO_F, nu=NU, sweeps=SWEEPS, steps_per_interval=INTERVAL)
    return s


def run(state):
    case, sim = state["case"], state["sim"]
    f64 = case["precision"] == "fp64"
    if case["kind"] == "adjoint":
        if f64:
            from paper_2603_26691_gb300.autograd import lagrangian_sources

            leaves = (state["d"], state["alpha"], state["U"])
            J = lagrangian_sources(*leaves, sim, state["pos"], state["vel"], case["steps"], case["dt"], case["every"])
            gd, ga, gU = torch.autograd.grad(J, leaves, state["lam"])
            return dict(J=J.detach(), gd=gd, ga=ga, gU=gU)
        sim.clear_particles()
        sim.add_particles(state["pos"], state["d"], state["vel"])
        sim.reorder()
        sim.adjoint_forward(case["steps"], case["dt"], case["every"])
        J = sim.sources(reset=True)
        gd, ga, gU = sim.adjoint_backward(state["lam"])
        return dict(J=J.float(), gd=gd.float(), ga=ga, gU=gU.float())
    sim.set_fluid(state["U"])
    out = {}
    if case["kind"] == "couple":
        sim.couple_run(case["steps"] // INTERVAL, case["dt"])
        u, src = sim.fluid(host=False), sim.pending_sources(host=False)
        out["u"] = u if f64 else u.float()
    else:
        sim.step(case["steps"], case["dt"])
        src = sim.sources(reset=True)
    out["src"] = src if f64 else src.float()
    if case["kind"] == "micro":
        ms = sim.micro_sources(reset=True, host=False)
        out["micro"] = ms if f64 else ms.float()
    # (particle temperatures have a host copy only, which a step loop does not take; the energy source holds them)
    out["pos"], out["vel"], out["d"], out["ids"] = sim.particles(host=False)
    return out


# ---- the least bytes and operations of a pass -----------------------------------------------------------

def work(case):
    n, steps = case["n"], case["steps"]
    nc = case["nx"] * case["ny"] * case["nz"]
    f64 = case["precision"] == "fp64"
    state = {"fp64": 56, "mixed_f32": 32, "mixed_bf16": 26}[case["precision"]]
    # gather 63, drag and integrator about 60, relocation and deposit about 20 operations a step
    flops = {"default": 143, "paper": 110, "cic": 143 + 72}[case["physics"]]
    fld = 24 if f64 else 12
    if case["kind"] == "adjoint":
        # particles, field and dL/dJ read once; J, dL/dd and dL/dU written once; a step forward and a step back
        return {"bytes": n * (24 + 8 + (24 if case["vmax"] else 0) + (8 if f64 else 4)) + nc * (2 * fld + 2 * fld),
                "flops": n * steps * (flops + 350.0)}
    # the state read and written once (the field is frozen over a pass), the particles given out, field in, sources out
    by = n * (2 * state + 60) + nc * 2 * fld
    if case["kind"] == "micro":
        by += n * (16 if f64 else 32) + nc * (32 if f64 else 16)
        flops += 120
    if case["kind"] == "couple":
        by += nc * fld
    return {"bytes": float(by), "flops": float(n * steps * flops + (nc * 30 * SWEEPS * steps / INTERVAL if case["kind"] == "couple" else 0))}


# ---- the same in 64 bits, in plain torch ------------------------------------------------------------------

class _Exact:
    """One step of one block of particles in FP64 torch, written from the method's equations."""

    def __init__(self, case, U):
        self.n, self.L = _grid(case), _box(case)
        self.h = [self.L[q] / self.n[q] for q in range(3)]
        self.inv_h = [self.n[q] / self.L[q] for q in range(3)]
        self.U = U.double().reshape(-1, 3)
        self.phys, self.dt = case["physics"], case["dt"]
        self.mixed = case["precision"] != "fp64"
        self.nc = self.n[0] * self.n[1] * self.n[2]

    def cells(self, x):
        i = [torch.floor(x[q].detach() * self.inv_h[q]).clamp(0, self.n[q] - 1).long() for q in range(3)]
        return i, i[0] + self.n[0] * (i[1] + self.n[1] * i[2])

    def stencil(self, x):
        f, lo, hi = [], [], []
        for q in range(3):
            s = x[q] * self.inv_h[q] - 0.5
            fl = torch.floor(s.detach())
            f.append(s - fl)
            a = fl.long() % self.n[q]
            lo.append(a)
            hi.append((a + 1) % self.n[q])
        out = []
        for k in range(8):
            dx, dy, dz = k & 1, (k >> 1) & 1, k >> 2
            w = (f[0] if dx else 1 - f[0]) * (f[1] if dy else 1 - f[1]) * (f[2] if dz else 1 - f[2])
            c = (hi[0] if dx else lo[0]) + self.n[0] * ((hi[1] if dy else lo[1]) + self.n[1] * (hi[2] if dz else lo[2]))
            out.append((w, c))
        return out

    def wrap(self, x):
        return [x[q] - self.L[q] * torch.floor(x[q].detach() / self.L[q]) for q in range(3)]

    def motion(self, x, v, d, up, alpha=1.0):
        """New position and velocity (lists of three) and the impulse given to the fluid, parcel weight 1."""
        dt = self.dt
        a = 18.0 * MU * alpha / (RHO_P * d * d)
        m = RHO_P * math.pi / 6.0 * d ** 3
        if self.phys == "paper":
            re = RHO_F / MU * torch.sqrt(sum((up[q] - v[q]) ** 2 for q in range(3))) * d
            a = a * torch.where(re <= 1000.0, 1.0 + 0.15 * re ** 0.687, 0.44 / 24.0 * re)
            vn = [(v[q] + dt * (a * up[q] + GRAVITY[q])) / (1.0 + a * dt) for q in range(3)]
            xn = [x[q] + dt * vn[q] for q in range(3)]
        else:
            E1 = -torch.expm1(-a * dt)
            w = [up[q] + GRAVITY[q] / a for q in range(3)]
            vn = [w[q] * E1 + v[q] * (1.0 - E1) for q in range(3)]
            xn = [x[q] + w[q] * dt + (v[q] - w[q]) * (E1 / a) for q in range(3)]
        J = [-m * (vn[q] - v[q] - GRAVITY[q] * dt) for q in range(3)]
        return self.wrap(xn), vn, J, m

    def gather(self, st, F):
        # in a field of m columns, at the cells of a stencil
        return [sum(w * F[c, q] for w, c in st) for q in range(F.shape[1])]

    def key(self, x, B):
        i, _ = self.cells(x)
        if self.mixed:  # an offset that FP32 rounds up to a whole cell is offset 0 of the next one
            i = [torch.where((x[q] * self.inv_h[q] - i[q]).float() >= 1.0, (i[q] + 1) % self.n[q], i[q]) for q in range(3)]
        nc = [(self.n[q] + B - 1) // B for q in range(3)]
        chunk = i[0] // B + nc[0] * (i[1] // B + nc[1] * (i[2] // B))
        mort, b = torch.zeros_like(chunk), 0
        while (1 << b) < B:
            for q in range(3):
                mort |= ((i[q] >> b) & 1) << (3 * b + q)
            b += 1
        return chunk * B ** 3 + mort


def _rho_sat(T):
    t = T - 273.15
    a = t + 243.04
    rs = 610.94 / 461.5 * torch.exp(17.625 * t / a) / T
    return rs, rs * (17.625 * 243.04 / (a * a) - 1.0 / T)


def _transfer(d, T, tf, rv, re, dt):
    """Diameter and temperature after a step of vapour and heat transfer (coefficients held, exact in time)."""
    A = math.pi * (2.0 + 0.6 * PRANDTL ** (1.0 / 3.0) * torch.sqrt(re)) * KAPPA * d
    B = 2.0 * math.pi * D_V * d
    rs, s = _rho_sat(T)
    den = A + LATENT * B * s
    k = den / (RHO_P * math.pi / 6.0 * d ** 3 * CP)
    delta = (A * (tf - T) + LATENT * B * (rv - rs)) / den
    x = k * dt
    p1 = -torch.expm1(-x) / x
    p2 = torch.where(x < 1e-3, 0.5 - x / 6 + x * x / 24, (1.0 - p1) / x)
    dq = 8.0 * D_V / RHO_P * dt * ((rv - rs) - s * delta * x * p2)
    return torch.sqrt(torch.clamp(d * d + dq, min=D_MIN ** 2)), T + delta * x * p1


def exact(case, seed):
    kind, n, steps = case["kind"], case["n"], case["steps"]
    if n * steps > (4.5e8 if kind == "adjoint" else 7e8):
        return None  # would take too long
    data = _inputs(case, seed)
    return _exact_adjoint(case, data) if kind == "adjoint" else _exact_steps(case, data)


def _deposit(S, J, cells, nc):
    for q in range(3):
        S[q].index_add_(0, cells, J[q])


def _exact_steps(case, data):
    n, dt, block = case["n"], case["dt"], 8_000_000
    e = _Exact(case, data["U"])
    x, d = data["pos"], data["d"].clone()
    v = torch.zeros_like(x) if data["vel"] is None else data["vel"]
    T = torch.full_like(d, T_INIT) if case["kind"] == "micro" else None
    TH = torch.stack([data["T"].reshape(-1), data["rv"].reshape(-1)], 1) if T is not None else None
    S = torch.zeros((3, e.nc), dtype=torch.float64, device="cuda")
    MS = torch.zeros((2, e.nc), dtype=torch.float64, device="cuda")
    last, since = None, K
    for step in range(case["steps"]):
        if since >= K:
            # the storage order: particles sorted by cell, equal cells in the order they had
            p = torch.argsort(e.key(x, case["chunk"]), stable=True)
            x, v, d = x[:, p], v[:, p], d[p]
            T = T[p] if T is not None else None
            since = 0
        since += 1
        if case["kind"] == "couple" and step % INTERVAL == 0:
            last, S = (S if step else None), torch.zeros_like(S)
            nxt = _fluid(e, last, dt)
        for a in range(0, n, block):
            b = slice(a, min(n, a + block))
            xb, vb, db = [x[q, b] for q in range(3)], [v[q, b] for q in range(3)], d[b]
            _, c0 = e.cells(xb)
            st = e.stencil(xb)
            up = [e.U[c0, q] for q in range(3)] if case["physics"] == "paper" else e.gather(st, e.U)
            xn, vn, J, m = e.motion(xb, vb, db, up)
            if T is not None:
                tf, rv = e.gather(st, TH)
                re = RHO_F / MU * torch.sqrt(sum((up[q] - vb[q]) ** 2 for q in range(3))) * db
                d1, T1 = _transfer(db, T[b], tf, rv, re, dt)
                dm = RHO_P * math.pi / 6.0 * (d1 - db) * (d1 * d1 + d1 * db + db * db)
                J = [J[q] - dm * vn[q] for q in range(3)]
                MS[0].index_add_(0, c0, -dm)
                MS[1].index_add_(0, c0, -CP * (m * (T1 - T[b]) + dm * T1))
                d[b], T[b] = d1, T1
            if case["physics"] == "cic":
                for w, c in st:
                    _deposit(S, [w * J[q] for q in range(3)], c, e.nc)
            else:
                _deposit(S, J, c0, e.nc)
            for q in range(3):
                x[q, b], v[q, b] = xn[q], vn[q]
        if case["kind"] == "couple" and step % INTERVAL == INTERVAL - 1:
            e.U = nxt
    out = {}
    if case["kind"] == "couple":
        out["u"] = e.U.reshape(case["nz"], case["ny"], case["nx"], 3)
    out["src"] = S  # coupled: the last interval's sources, which the fluid has not received
    if T is not None:
        out["micro"] = MS
    if case["precision"] != "fp64" and case["steps"] > K:
        # a second sort: FP32 positions decide some cells differently, which moves every particle behind them
        return dict(out, pos=None, vel=None, d=None, ids=None)
    return dict(out, pos=x, vel=v, d=d, ids=None)


def _fluid(e, S, dt):
    """The next coupled field: the previous interval's sources, then Jacobi sweeps of an implicit diffusion step."""
    nx, ny, nz = e.n
    us = e.U.reshape(nz, ny, nx, 3)
    if S is not None:
        us = us + (S / (RHO_F * e.h[0] * e.h[1] * e.h[2])).reshape(3, nz, ny, nx).permute(1, 2, 3, 0)
    lam = [NU * INTERVAL * dt / (e.h[q] ** 2) for q in range(3)]
    u = us
    for _ in range(SWEEPS):
        u = (us + sum(lam[q] * (torch.roll(u, 1, 2 - q) + torch.roll(u, -1, 2 - q)) for q in range(3))) / (1.0 + 2.0 * sum(lam))
    return u.reshape(-1, 3)


def _exact_adjoint(case, data):
    n, block = case["n"], 400_000
    e = _Exact(case, data["U"])
    lam = data["lam"].double()
    d0, U0 = data["d"], e.U.clone()
    order = None
    if case["precision"] != "fp64":  # sorted once before the run; its gradients in that order
        order = torch.argsort(e.key(data["pos"], case["chunk"]), stable=True)
    J = torch.zeros((3, e.nc), dtype=torch.float64, device="cuda")
    gd, ga, gU = torch.zeros_like(d0), 0.0, torch.zeros_like(U0)
    for a in range(0, n, block):
        b = slice(a, min(n, a + block))
        d = d0[b].clone().requires_grad_()
        e.U = U0.clone().requires_grad_()
        alpha = torch.ones((), dtype=torch.float64, device="cuda", requires_grad=True)
        x = [data["pos"][q, b] for q in range(3)]
        v = [torch.zeros_like(d0[b]) if data["vel"] is None else data["vel"][q, b] for q in range(3)]
        loss = 0.0
        for _ in range(case["steps"]):
            _, c0 = e.cells(x)
            st = e.stencil(x)
            Uc = [(w, e.U[c]) for w, c in st]
            up = [sum(w * u[:, q] for w, u in Uc) for q in range(3)]
            xn, vn, Jp, _ = e.motion(x, v, d, up, alpha)
            for w, c in (st if case["physics"] == "cic" else [(1.0, c0)]):
                for q in range(3):
                    loss = loss + (lam[q][c] * (w * Jp[q])).sum()
                    J[q].index_add_(0, c, (w * Jp[q]).detach())
            x, v = xn, vn
        g = torch.autograd.grad(loss, (d, alpha, e.U))
        gd[b] = g[0]
        ga += float(g[1])
        gU += g[2]
    shape = (case["nz"], case["ny"], case["nx"], 3) if case["precision"] == "fp64" else (e.nc, 3)
    return dict(J=J, gd=gd if order is None else gd[order], ga=torch.tensor(ga, dtype=torch.float64), gU=gU.reshape(shape))
