"""The work a user has this library do, as cases that can be timed and whose results can be compared.

Each case goes through the public entry points of ``paper_2605_27004_gb300``: a context is made once
(``prepare``), and a pass gives it new initial fields, advances it and reads the observables (or the
gradients) back as device tensors. Sizes are those of the repository's own workloads, cut to runs
that a program repeats, plus odd ones; ``draw`` gives more cases of the same ranges.

Kinds:
  flow     init, step(n), moments (and the conserved totals where ``totals`` is set)
  sampled  init, then ``samples`` times step(n) and the velocity: a decay measurement
  train    one optimisation step: simulate() with recorded checkpoints, a loss, its gradients
  scalar   a scalar carried by a frozen velocity field (advection-diffusion), step(n), phi
  coupled  a flow and a scalar advanced together, the flow's velocity handed over every step
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_27004_gb300 import inputs, lbm
from paper_2605_27004_gb300.autograd import simulate, theta_matrix, theta_vector

ELEM = {"fp64": 8, "fp32": 4, "fp32s": 4, "fp16s": 2}
TRAIN_TAU = 0.6


def _case(name, kind, lattice, dims, steps, storage="fp32s", scheme="pull", tau=0.6, walls="none", **more):
    c = {"kind": kind, "lattice": lattice, "nx": dims[0], "ny": dims[1], "nz": dims[2], "steps": steps,
         "storage": storage, "scheme": scheme, "tau": tau, "walls": walls}
    if name:
        c["name"] = name
    return c | more


def listed():
    return [
        # A 2D shear wave in FP64 on a small box: verification runs against linear theory.
        _case("shear_2d_fp64", "flow", 9, (64, 64, 1), 1000, storage="fp64", tau=0.8, totals=True),
        # The 2D Taylor-Green decay measurement: short runs with the velocity read in between.
        _case("decay_2d_sampled", "sampled", 9, (96, 80, 1), 16, tau=1.0, samples=25),
        # FP64 in 3D: the mode that parity and finite-difference checks run in.
        _case("tg_64_fp64", "flow", 19, (64, 64, 64), 50, storage="fp64"),
        # A small 3D box in the default storage: parameter studies, where launches count.
        _case("tg_64_fp32", "flow", 19, (64, 64, 64), 200),
        # The Taylor-Green vortex at 256^3 in the default storage: the ordinary forward run.
        _case("tg_256_fp32", "flow", 19, (256, 256, 256), 50),
        # A large box in place with FP16 storage: the biggest forward runs.
        _case("tg_512_fp16_aa", "flow", 19, (512, 512, 512), 16, storage="fp16s", scheme="aa"),
        # Odd sizes on the 27-velocity lattice, FP16 storage.
        _case("ragged_d3q27_fp16", "flow", 27, (149, 131, 113), 40, storage="fp16s", tau=0.7),
        # Flow through a porous medium of overlapping spheres, default storage, totals monitored.
        _case("porous_256_fp32", "flow", 27, (256, 256, 256), 30, tau=0.7, walls="porous", totals=True),
        # The same medium with FP16 storage in place.
        _case("porous_256_fp16_aa", "flow", 27, (256, 256, 256), 30, storage="fp16s", scheme="aa", tau=0.7,
              walls="porous"),
        # One step of the recovery of Theta from a velocity field: forward, loss, backward.
        _case("train_128_fp32", "train", 19, (128, 128, 128), 100, K=20),
        # The gradient at FP16 storage, in place: the large differentiable runs.
        _case("train_192_fp16_aa", "train", 19, (192, 192, 192), 40, storage="fp16s", scheme="aa", K=20),
        # A scalar carried by a flow that evolves with it.
        _case("coupled_scalar", "coupled", 19, (96, 88, 80), 30),
    ]


def _span(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, cells, d):
    """A box of about `cells` cells: rows of any length, odd ones and multiples of 32 among them."""
    side = cells ** (1.0 / d)
    n = [max(12, int(round(side * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(d)]
    if rng.random() < 0.5:
        n[0] = max(32, 32 * round(n[0] / 32))
    n[d - 1] = max(8, int(round(cells / math.prod(n[:d - 1]))))
    return tuple(n) + (1,) * (3 - d)


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "flow2d", "sampled", "train", "scalar", "coupled", "fp64"])
    tau = round(rng.uniform(0.55, 1.0), 3)
    scheme = rng.choice(["pull", "aa"])
    if kind in ("flow2d", "sampled"):
        cells = _span(rng, 2000, 200000 if kind == "sampled" else 4000000)
        storage = rng.choice(["fp32s", "fp64"] if cells < 70000 else ["fp32s", "fp16s"])
        dims = _dims(rng, cells, 2)
        if kind == "sampled":
            return _case(None, "sampled", 9, dims, rng.randint(4, 24), storage, scheme, tau, samples=rng.randint(5, 25))
        return _case(None, "flow", 9, dims, rng.randint(40, 400), storage, scheme, tau,
                     totals=storage != "fp16s" and rng.random() < 0.5)
    lattice = rng.choice([19, 19, 27])
    if kind == "fp64":
        return _case(None, "flow", lattice, _dims(rng, _span(rng, 8000, 400000), 3), rng.randint(10, 60), "fp64",
                     scheme, tau)
    storage = rng.choice(["fp32s", "fp16s"])
    if kind == "train":
        cells = _span(rng, 40000, 6000000)
        K = rng.choice([5, 10, 20])
        steps = min(100, max(K, K * int(1.5e8 / cells / K)))
        return _case(None, "train", 19, _dims(rng, cells, 3), steps, storage, scheme, TRAIN_TAU, K=K)
    if kind in ("scalar", "coupled"):
        cells = _span(rng, 40000, 16000000 if kind == "scalar" else 4000000)
        steps = max(4, min(60, int(3e8 / cells)))
        walls = rng.choice(["none", "porous"]) if kind == "scalar" else "none"
        return _case(None, kind, lattice, _dims(rng, cells, 3), steps, storage, scheme, tau, walls)
    cells = _span(rng, 40000, 60000000)
    walls = rng.choice(["none", "none", "porous"])
    if walls == "porous":
        cells = min(cells, 17000000)
    steps = max(4, min(200, int(7e8 / cells)))
    return _case(None, "flow", lattice, _dims(rng, cells, 3), steps, storage, scheme, tau, walls)


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _dim(case):
    return 2 if case["lattice"] == 9 else 3


def _mesh(case, device):
    """(x, y, z) angles 2 pi x / nx ... of every cell, shaped to broadcast over [nz, ny, nx]."""
    out = []
    for a, n in enumerate((case["nx"], case["ny"], case["nz"])):
        shape = [1, 1, 1]
        shape[2 - a] = n
        out.append((torch.arange(n, dtype=torch.float64, device=device) * (2 * math.pi / n)).reshape(shape))
    return out


def _velocity(case, seed, amp, mean=0.0):
    """A Taylor-Green vortex of seeded phase and six seeded shear modes, [d, N], max about `amp`."""
    r = np.random.default_rng(seed)
    x, y, z = _mesh(case, "cuda")
    d, dims = _dim(case), (case["nz"], case["ny"], case["nx"])
    px, py, pz = r.uniform(0, 2 * math.pi, 3)
    cz = torch.cos(z + pz) if d == 3 else torch.ones_like(z)
    u = torch.zeros((d,) + dims, dtype=torch.float64, device="cuda")
    u[0] += 0.5 * torch.sin(x + px) * torch.cos(y + py) * cz
    u[1] -= 0.5 * torch.cos(x + px) * torch.sin(y + py) * cz
    for _ in range(6):
        k = r.integers(1, 4, 3) * r.choice([-1, 1], 3)
        a, b = r.choice(d, 2, replace=False)  # u_a varies along the other axes only: divergence-free
        phase = r.uniform(0, 2 * math.pi)
        arg = sum((int(k[c]) * (x, y, z)[c] for c in range(d) if c != a), torch.zeros_like(x)) + phase
        u[a] += r.uniform(0.05, 0.12) * torch.sin(arg)
    u *= amp
    u[0] += mean
    return u.reshape(d, -1)


def _theta(case, seed):
    if _dim(case) == 2:
        a = np.random.default_rng(seed + 17).uniform(0.0, 0.4)
        return inputs.theta_from_atilde([[1.0, a], [a, 1.0]])
    return inputs.theta_spd(seed + 17)


def _solid(case, seed):
    if case["walls"] == "none":
        return None
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    small = min(nx, ny, nz)
    r = min(8.0, small / 10.0)
    return inputs.porous_spheres(nx, ny, nz, r, 2 * r, 0.30, seed=seed + 5)


def _fields(case, seed):
    """Everything a pass starts from, on the device in the context's field type."""
    dt = torch.float64 if case["storage"] == "fp64" else torch.float32
    kind, N = case["kind"], case["nx"] * case["ny"] * case["nz"]
    f = {"Theta": _theta(case, seed), "solid": _solid(case, seed)}
    f["u"] = _velocity(case, seed, 0.02, 0.03 if f["solid"] is not None else 0.01).to(dt)
    if kind in ("flow", "sampled"):
        x, y, _ = _mesh(case, "cuda")
        rho = 1.0 - 3e-4 * (torch.cos(2 * x) + torch.cos(2 * y))
        f["rho"] = rho.expand(case["nz"], case["ny"], case["nx"]).reshape(N).to(dt).contiguous()
    if kind == "train":
        f["target"] = _velocity(case, seed + 1000, 0.02, 0.01).to(dt)
        f["theta"] = torch.tensor(theta_vector(f["Theta"]), dtype=torch.float32)
        f["Theta"] = theta_matrix(f["theta"].numpy(), _dim(case))
    if kind in ("scalar", "coupled"):
        x, y, z = _mesh(case, "cuda")
        c = np.random.default_rng(seed + 29).uniform(0, 2 * math.pi, 3)
        blob = torch.exp(2.0 * (torch.cos(x - c[0]) + torch.cos(y - c[1]) + torch.cos(z - c[2]) - 3.0))
        f["phi"] = (1.0 + 0.5 * blob).expand(case["nz"], case["ny"], case["nx"]).reshape(N).to(dt).contiguous()
        f["ThetaS"] = _theta(case, seed + 41)
    return f


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case = case
    f = _fields(case, seed)
    dims = (case["nx"], case["ny"], case["nz"])
    opt = {"solid": f["solid"], "storage": case["storage"], "scheme": case["scheme"]}
    s.u = f["u"]
    if case["kind"] in ("flow", "sampled", "train", "coupled"):
        s.flow = lbm.LBM(case["lattice"], *dims, case["tau"], f["Theta"], **opt)
    if case["kind"] in ("flow", "sampled"):
        s.rho = f["rho"]
    if case["kind"] == "train":
        s.u.requires_grad_(True)
        s.theta = f["theta"].requires_grad_(True)
        s.target = f["target"]
    if case["kind"] in ("scalar", "coupled"):
        s.phi = f["phi"]
        s.scalar = lbm.ADE(case["lattice"], *dims, case["tau"], f["ThetaS"],
                           u=s.u if case["kind"] == "scalar" else None, **opt)
    if case["kind"] == "coupled":
        s.view = s.scalar.velocity_view()
    return s


def run(s):
    case, n = s.case, s.case["steps"]
    if case["kind"] == "flow":
        s.flow.init(s.rho, s.u)
        s.flow.step(n)
        out = dict(zip(("rho", "u", "Pi"), s.flow.moments(Pi=True)))
        if case.get("totals"):
            out["mass"], out["momentum"] = s.flow.totals()
        return out
    if case["kind"] == "sampled":
        s.flow.init(s.rho, s.u)
        out = []
        for _ in range(case["samples"]):
            s.flow.step(n)
            out.append(s.flow.moments(rho=False, u=True)[1])
        return out
    if case["kind"] == "train":
        u = simulate(s.u, s.theta, case["tau"], s.flow, n, case["K"])
        loss = ((u - s.target) ** 2).sum(dim=0).mean()
        du0, dtheta = torch.autograd.grad(loss, (s.u, s.theta))
        return {"u": u.detach(), "loss": loss.detach(), "du0": du0, "dtheta": dtheta}
    if case["kind"] == "scalar":
        s.scalar.init(s.phi)
        s.scalar.step(n)
        return s.scalar.scalar()
    s.flow.init(None, s.u)
    s.flow.moments_into(u=s.view)
    s.scalar.init(s.phi)
    for _ in range(n):
        s.flow.step(1)
        s.flow.moments_into(u=s.view)
        s.scalar.step(1)
    return {"u": s.flow.moments(rho=False)[1], "phi": s.scalar.scalar()}


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------
def work(case):
    """Bytes: the initial fields read once, the results written once, and for every time step the
    populations read once and written once (a scalar also reads its velocity); the adjoint step
    reads lambda and the state and writes lambda. Flops: about 14 per population and collision."""
    q, d, e = case["lattice"], _dim(case), ELEM[case["storage"]]
    N, n = case["nx"] * case["ny"] * case["nz"], case["steps"]
    fe = 8 if case["storage"] == "fp64" else 4
    fluid = N * (0.70 if case["walls"] == "porous" else 1.0)
    step = 2 * q * e * fluid
    flop = 14 * q * fluid
    if case["kind"] == "flow":
        fields = (1 + d) * N * fe + (1 + d + d * (d + 1) // 2) * N * fe
        return {"bytes": fields + n * step, "flops": n * flop}
    if case["kind"] == "sampled":
        k = case["samples"]
        return {"bytes": (1 + d) * N * fe + k * (d * N * fe + n * step), "flops": k * n * flop}
    if case["kind"] == "train":
        adj = (2 * q * fe + q * e) * N
        return {"bytes": 4 * d * N * fe + n * (step + adj), "flops": n * 4 * flop}
    if case["kind"] == "scalar":
        return {"bytes": 2 * N * fe + n * (step + d * fe * fluid), "flops": n * flop}
    return {"bytes": (2 * d + 2) * N * fe + n * (2 * step + 2 * d * N * fe), "flops": n * 2 * flop}


# ---------------------------------------------------------------------------------------------
# The method in plain 64-bit torch
# ---------------------------------------------------------------------------------------------
def _lattice(q):
    """Velocities and weights of the set, in any order (only moments leave this file)."""
    d = 2 if q == 9 else 3
    w1 = {0: 2.0 / 3.0, 1: 1.0 / 6.0, -1: 1.0 / 6.0}
    c, w = [], []
    for z in ((0,) if d == 2 else (0, 1, -1)):
        for y in (0, 1, -1):
            for x in (0, 1, -1):
                if q == 19:
                    m = abs(x) + abs(y) + abs(z)
                    if m == 3:
                        continue
                    w.append((1 / 3, 1 / 18, 1 / 36)[m])
                else:
                    w.append(w1[x] * w1[y] * (w1[z] if d == 3 else 1.0))
                c.append((x, y, z))
    return c, w


class _Plain:
    """BGK with the third-order anisotropic equilibrium on [nz, ny, nx] tensors, pre-collision state."""

    def __init__(self, case, Theta, solid=None):
        self.c, self.w = _lattice(case["lattice"])
        self.d, self.tau = _dim(case), case["tau"]
        self.dims = (case["nz"], case["ny"], case["nx"])
        self.opp = [self.c.index((-x, -y, -z)) for x, y, z in self.c]
        self.K = [[Theta[a][b] - (1 / 3 if a == b else 0.0) for b in range(self.d)] for a in range(self.d)]
        self.wall, self.solid = None, None
        if solid is not None:
            self.solid = torch.as_tensor(np.asarray(solid), device="cuda").reshape(self.dims) != 0
            self.wall = [self.stream(self.solid, i) for i in range(len(self.c))]

    def stream(self, f, i):
        x, y, z = self.c[i]
        return torch.roll(f, (z, y, x), (0, 1, 2)) if (x or y or z) else f

    def shared(self, u):
        """|u|^2 and K~ u of the equilibrium."""
        usq = sum(v * v for v in u)
        Ku = [sum(self.K[a][b] * u[b] for b in range(self.d)) for a in range(self.d)]
        return usq, Ku

    def feq(self, i, rho, u, usq, Ku):
        c = self.c[i][:self.d]
        on = [a for a in range(self.d) if c[a]]
        h = sum(c[a] * self.K[a][b] * c[b] for a in on for b in on) - sum(self.K[a][a] for a in range(self.d)) / 3
        if not on:
            return self.w[i] * rho * (1 + 4.5 * h - 1.5 * usq)
        uc = sum(c[a] * u[a] for a in on)
        cK = sum(c[a] * Ku[a] for a in on)
        return self.w[i] * rho * (1 + 4.5 * h - 1.5 * usq + uc * (3 + 13.5 * h - 4.5 * usq + uc * (4.5 + 4.5 * uc)) - 9 * cK)

    def start(self, rho, u):
        s = self.shared(u)
        return [self.feq(i, rho, u, *s) for i in range(len(self.c))]

    def moments(self, f, Pi=False):
        rho = sum(f[1:], f[0].clone())
        j = []
        for a in range(self.d):
            m = torch.zeros_like(rho)
            for i, c in enumerate(self.c):
                if c[a]:
                    m = m + f[i] if c[a] > 0 else m - f[i]
            j.append(m)
        u = [m / rho for m in j]
        if not Pi:
            return rho, u
        P = []
        pairs = [(0, 0), (1, 1), (0, 1)] if self.d == 2 else [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
        for a, b in pairs:
            P.append(sum(f[i] * (c[a] * c[b]) for i, c in enumerate(self.c) if c[a] * c[b]))
        return rho, u, P

    def step(self, f, u=None, rebuild=False):
        """One collide-and-stream; `u` given: that of a scalar. `rebuild` leaves the given list alone."""
        rho, v = self.moments(f) if u is None else (sum(f[1:], f[0].clone()), u)
        s = self.shared(v)
        post = f if not rebuild else [None] * len(f)
        for i in range(len(f)):
            post[i] = f[i] + (self.feq(i, rho, v, *s) - f[i]) / self.tau
        del rho, s
        if self.wall is None:
            for i in range(len(f)):
                post[i] = self.stream(post[i], i)
            return post
        out = [torch.where(self.wall[i], post[self.opp[i]], self.stream(post[i], i)) for i in range(len(f))]
        return out

    def fluid(self, t):
        return t if self.solid is None else torch.where(self.solid, torch.zeros_like(t), t)

    def flat(self, ts):
        return torch.stack([self.fluid(t).reshape(-1) for t in ts])


def exact(case, seed):
    f0 = _fields(case, seed)
    dims, d, n = (case["nz"], case["ny"], case["nx"]), _dim(case), case["steps"]
    u0 = f0["u"].double().reshape((d,) + dims)
    if case["kind"] == "train":
        return _exact_train(case, f0, u0)
    if case["kind"] in ("flow", "sampled"):
        m = _Plain(case, f0["Theta"], f0["solid"])
        f = m.start(f0["rho"].double().reshape(dims), list(u0))
        del f0, u0
        if case["kind"] == "sampled":
            out = []
            for _ in range(case["samples"]):
                for _ in range(n):
                    f = m.step(f)
                out.append(m.flat(m.moments(f)[1]))
            return out
        for _ in range(n):
            f = m.step(f)
        rho, u, P = m.moments(f, Pi=True)
        out = {"rho": m.fluid(rho).reshape(-1), "u": m.flat(u), "Pi": m.flat(P)}
        if case.get("totals"):
            out["mass"] = float(out["rho"].sum())
            out["momentum"] = (out["rho"] * out["u"]).sum(dim=1).cpu().numpy()
        return out
    s = _Plain(case, f0["ThetaS"], f0["solid"])
    phi = f0["phi"].double().reshape(dims)
    if case["kind"] == "scalar":
        v = list(u0)
        g = s.start(phi, v)
        for _ in range(n):
            g = s.step(g, v)
        return s.fluid(sum(g[1:], g[0])).reshape(-1)
    m = _Plain(case, f0["Theta"])
    f = m.start(torch.ones(dims, dtype=torch.float64, device="cuda"), list(u0))
    g = s.start(phi, m.moments(f)[1])
    for _ in range(n):
        f = m.step(f)
        g = s.step(g, m.moments(f)[1])
    return {"u": m.flat(m.moments(f)[1]), "phi": sum(g[1:], g[0]).reshape(-1)}


def _exact_train(case, f0, u0):
    from torch.utils.checkpoint import checkpoint
    d, n = _dim(case), case["steps"]
    u0 = u0.clone().requires_grad_(True)
    theta = f0["theta"].double().cuda().requires_grad_(True)
    m = _Plain(case, f0["Theta"])
    at = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}

    def with_theta(th):
        m.K = [[th[at[min(a, b), max(a, b)]] - (1 / 3 if a == b else 0.0) for b in range(d)] for a in range(d)]

    def first(u, th):
        with_theta(th)
        return torch.stack(m.start(torch.ones(u.shape[1:], dtype=u.dtype, device=u.device), list(u)))

    def one(f, th):
        with_theta(th)
        return torch.stack(m.step(list(f), rebuild=True))

    f = checkpoint(first, u0, theta, use_reentrant=False)
    for _ in range(n):
        f = checkpoint(one, f, theta, use_reentrant=False)
    u = torch.stack(m.moments(list(f))[1]).reshape(d, -1)
    loss = ((u - f0["target"].double()) ** 2).sum(dim=0).mean()
    du0, dtheta = torch.autograd.grad(loss, (u0, theta))
    return {"u": u.detach(), "loss": loss.detach(), "du0": du0.reshape(d, -1), "dtheta": dtheta}
