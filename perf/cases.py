"""Timed cases of the framework's public entry points, with 64-bit references.

Every case is one pass of a program that keeps its lattice contexts: it sets a
state, advances it and reads what it wants to know, all through
``paper_1905_04597_gb300.glbm``. Fields are FP64 tensors on the GPU. The
kinds, and what each stands for:

  shock     a 1D shock tube (Sec. 5.1 of the paper): the smallest lattices, many
            steps per call.
  channel   a batch of 2D channels of one geometry at several Knudsen numbers
            (Secs. 5.3, 5.4): equilibrium start, steps, all moment fields of
            every instance. Lattices: "iso" level k+1 on both axes, "d1q3" D1Q3
            along x, "zv" D1Q3 along x times the 2N+2 hierarchy along y.
  box       the same for a 3D product lattice.
  mixed     a batch of channels of different levels, sizes and forces.
  gradient  the differentiable flow rate, forward and backward, as one step of
            an optimiser of tau, g and the wall speeds calls it.
  fields    import of populations, the analysis of one state (moment fields,
            channel diagnostics, conservation sums) and their export: a restart
            or a post-processing pass, without steps.
"""
import math

import numpy as np
import torch

from paper_1905_04597_gb300 import glbm

# ---- cases ----------------------------------------------------------------


def listed():
    return [
        # the shock tube as the benchmark runs it, and with a higher level on
        # the paper's 800 nodes in FP64
        dict(name="shock_fp32", kind="shock", k=1, nx=1000, n=1, prec=32, steps=500),
        dict(name="shock_fp64", kind="shock", k=2, nx=800, n=1, prec=64, steps=500),
        # the smoke check's lattice: one call of a few steps, all launch latency
        dict(name="channel_tiny_fp64", kind="channel", lattice="iso", k=3, nx=40, ny=24, n=1,
             prec=64, steps=5, wall=0.05, g=1e-5),
        # the headline Couette workload, end to end
        dict(name="couette_fp32", kind="channel", lattice="iso", k=3, nx=512, ny=256, n=3,
             prec=32, steps=100, wall=0.05, g=0.0),
        # the same channel in FP64, one instance
        dict(name="couette_fp64", kind="channel", lattice="iso", k=3, nx=512, ny=256, n=1,
             prec=64, steps=20, wall=0.05, g=0.0),
        # the largest 2D workload: force-driven flow on D2Q289
        dict(name="poiseuille_fp32", kind="channel", lattice="iso", k=7, nx=1024, ny=128, n=8,
             prec=32, steps=20, wall=0.0, g=1e-6),
        # the paper's channel model G-D1Q8 x D1Q3 on its 200 rows, a width that
        # is no multiple of a tile
        dict(name="channel_zv_fp32", kind="channel", lattice="zv", k=2, nx=1000, ny=200, n=3,
             prec=32, steps=50, wall=0.05, g=0.0),
        # a Knudsen-minimum sweep with G-D1Q28 x D1Q3 in FP64 on x-uniform
        # channels: many steps on very small lattices
        dict(name="knudsen_fp64", kind="channel", lattice="zv", k=12, nx=1, ny=200, n=5,
             prec=64, steps=500, wall=0.0, g=1e-7),
        # a 3D channel on D3Q125 with ragged sizes
        dict(name="box_fp32", kind="box", k=1, nx=250, ny=61, nz=45, n=1, prec=32, steps=20,
             wall=0.05, g=0.0),
        # 64 channels of mixed level, height and drive
        dict(name="mixed_fp32", kind="mixed", n=64, nx=64, kmax=7, hmin=32, hmax=512, steps=20),
        # one optimiser step through the differentiable flow rate
        dict(name="gradient_fp32", kind="gradient", k=4, nx=256, ny=128, prec=32, steps=200,
             every=100, kn=0.1, g=1e-6),
        # restart and post-processing of a large lattice
        dict(name="fields_fp32", kind="fields", k=3, nx=2048, ny=256, prec=32, wall=0.05, g=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shock", "channel", "channel", "channel", "box", "mixed", "gradient",
                       "fields"])
    prec = rng.choice([32, 32, 64])
    if kind == "shock":
        return dict(kind=kind, k=rng.randint(0, 7 if prec == 32 else 2),
                    nx=_log_int(rng, 60, 4000), n=rng.randint(1, 3), prec=prec,
                    steps=_log_int(rng, 50, 1000))
    if kind == "channel":
        lattice = rng.choice(["iso", "iso", "d1q3", "zv"])
        k = rng.randint(0, 12 if lattice == "zv" else 7)
        n = rng.randint(1, 4)
        nx, ny = _log_int(rng, 1, 1500), _log_int(rng, 2 * k + 3, 400)
        q = (2 * k + 3) ** 2 if lattice == "iso" else 3 * (2 * k + 4)
        # at most the population updates of the largest listed case
        steps = min(_log_int(rng, 2, 200), max(1, int(4e9 / (q * nx * ny * n * (prec / 32) ** 3))))
        wall, g = rng.choice([(round(rng.uniform(0.01, 0.08), 3), 0.0), (0.0, 1e-6),
                              (round(rng.uniform(0.01, 0.05), 3), 1e-6)])
        return dict(kind=kind, lattice=lattice, k=k, nx=nx, ny=ny, n=n, prec=prec, steps=steps,
                    wall=wall, g=g)
    if kind == "box":
        k = rng.randint(0, 2)
        nx, ny, nz = _log_int(rng, 8, 256), _log_int(rng, 5, 64), _log_int(rng, 3, 48)
        steps = min(_log_int(rng, 2, 60),
                    max(1, int(2e9 / ((2 * k + 3) ** 3 * nx * ny * nz * (prec / 32) ** 3))))
        return dict(kind=kind, k=k, nx=nx, ny=ny, nz=nz, n=1, prec=prec, steps=steps,
                    wall=0.03, g=rng.choice([0.0, 1e-6]))
    if kind == "mixed":
        hmin = rng.randint(10, 40)
        return dict(kind=kind, n=rng.randint(3, 64), nx=rng.randint(20, 96), kmax=rng.randint(2, 7),
                    hmin=hmin, hmax=hmin + _log_int(rng, 20, 300), steps=_log_int(rng, 2, 20))
    if kind == "gradient":
        k = rng.randint(0, 5)
        return dict(kind=kind, k=k, nx=_log_int(rng, 8, 256), ny=_log_int(rng, 16, 128),
                    prec=prec, steps=_log_int(rng, 10, 150), every=rng.choice([10, 32, 100]),
                    kn=round(rng.uniform(0.05, 1.0), 3), g=1e-6)
    return dict(kind=kind, k=rng.randint(0, 5), nx=_log_int(rng, 16, 1500),
                ny=_log_int(rng, 16, 256), prec=prec, wall=0.05, g=rng.choice([0.0, 1e-6]))


# ---- inputs ---------------------------------------------------------------

KN = (0.01, 10.0)  # Knudsen numbers of a batch, spread over the paper's range


def _knudsen(i, n):
    return KN[0] * (KN[1] / KN[0]) ** (i / (n - 1)) if n > 1 else 0.1


def _rng(seed, salt=0):
    return np.random.default_rng([int(seed), salt])


def _smooth(rng, shape, amp):
    """A sum of three random modes over the lattice (periodic in x and z), at most `amp`."""
    dev = torch.device("cuda")
    ax = [torch.arange(s, dtype=torch.float64, device=dev) / s for s in shape]
    out = torch.zeros(shape, dtype=torch.float64, device=dev)
    for _ in range(3):
        a = amp / 3 * float(rng.uniform(0.3, 1.0)) * (1 if rng.integers(0, 2) else -1)
        term = torch.full((), a, dtype=torch.float64, device=dev)
        for d, s in enumerate(ax):
            ph = 2 * math.pi * float(rng.uniform())
            if d == len(shape) - 2:  # the wall-normal axis is not periodic
                f = torch.cos(math.pi * float(rng.uniform(0.5, 3.0)) * s + ph)
            else:
                f = torch.sin(2 * math.pi * int(rng.integers(0, 4)) * s + ph)
            term = term * f.reshape([-1 if e == d else 1 for e in range(len(shape))])
        out += term
    return out


def _macro(rng, shape):
    """Density and velocity fields around a gas at rest."""
    rho = 1.0 + _smooth(rng, shape, 0.02)
    return [rho] + [_smooth(rng, shape, 0.03) for _ in shape]


def _prec(case):
    return glbm.FP64 if case["prec"] == 64 else glbm.FP32_DEV


def _configs(case, seed):
    """The instances of a case as configurations."""
    kind = case["kind"]
    if kind == "shock":
        return [dict(dims=1, k=case["k"], nx=case["nx"], kn=0.01 * (i + 1), prec=_prec(case))
                for i in range(case["n"])]
    if kind in ("channel", "box", "fields"):
        base = dict(dims=2, k=case["k"], nx=case["nx"], ny=case["ny"], prec=_prec(case),
                    u_wall_lo=-case["wall"], u_wall_hi=case["wall"], g=case["g"])
        if kind == "box":
            base.update(dims=3, nz=case["nz"])
        if case.get("lattice") in ("d1q3", "zv"):
            base.update(x_level=1, zv_axes=glbm.ZV_Y if case["lattice"] == "zv" else 0)
        return [dict(base, kn=_knudsen(i, case.get("n", 1))) for i in range(case.get("n", 1))]
    # mixed: levels, heights, Knudsen numbers and drives of the batched workload
    rng = np.random.default_rng(17)
    out = []
    for _ in range(case["n"]):
        c = dict(dims=2, k=int(rng.integers(1, case["kmax"] + 1)), nx=case["nx"],
                 ny=int(rng.integers(case["hmin"], case["hmax"] + 1)),
                 kn=float(10.0 ** rng.uniform(-2.0, 1.0)), prec=glbm.FP32_DEV)
        if rng.integers(0, 2):
            uw = float(rng.uniform(0.0, 0.1))
            c.update(u_wall_lo=-uw, u_wall_hi=uw, g=0.0)
        else:
            c.update(u_wall_lo=0.0, u_wall_hi=0.0, g=float(rng.uniform(1e-7, 1e-5)))
        out.append(c)
    return out


def _shape(c):
    return (c["nx"],) if c["dims"] == 1 else \
        (c["ny"], c["nx"]) if c["dims"] == 2 else (c["nz"], c["ny"], c["nx"])


def _start(case, cfgs, seed):
    """Start fields of every instance, [rho, u_x, ...] each."""
    rng = _rng(seed)
    out = []
    for c in cfgs:
        if case["kind"] == "shock":
            x = torch.arange(c["nx"], device="cuda")
            left, right = float(rng.uniform(0.9, 1.0)), float(rng.uniform(0.125, 0.25))
            rho = torch.where(x < c["nx"] // 2, left, right).to(torch.float64)
            out.append([rho, torch.zeros_like(rho)])
        else:
            out.append(_macro(rng, _shape(c)))
    return out


def _gradient_inputs(case, seed):
    """tau, g and the wall speeds of one optimiser step."""
    rng = _rng(seed)
    tau = case["kn"] * case["ny"] / math.sqrt(2.0 * (case["k"] + 1) / 3.0)
    return [tau * float(rng.uniform(0.8, 1.2)), case["g"] * float(rng.uniform(0.8, 1.2)),
            float(rng.uniform(0.0, 0.02)), float(rng.uniform(0.0, 0.02))]


def _populations(cfg, seed):
    """Populations of a flow away from equilibrium: rest weights times smooth factors."""
    rng = _rng(seed)
    w = _axis_weights(cfg["k"] + 1, 0).to("cuda")
    base = _smooth(rng, _shape(cfg), 0.03)
    q = w.numel()
    f = torch.empty((q, q) + _shape(cfg), dtype=torch.float64, device="cuda")
    tilt = rng.uniform(-0.3, 0.3, size=(q, q))
    for iy in range(q):
        for ix in range(q):
            f[iy, ix] = float(w[iy] * w[ix]) * (1.0 + float(0.05 * tilt[iy, ix]) +
                                                (1.0 + float(tilt[iy, ix])) * base)
    return f.reshape((q * q,) + _shape(cfg))


# ---- one pass -------------------------------------------------------------


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case = case
    if case["kind"] == "gradient":
        s.params = [torch.tensor(v, dtype=torch.float64, requires_grad=True)
                    for v in _gradient_inputs(case, seed)]
        s.config = dict(dims=2, k=case["k"], nx=case["nx"], ny=case["ny"], prec=_prec(case))
        return s
    cfgs = _configs(case, seed)
    s.lat = glbm.Lattice(cfgs, hetero=case["kind"] == "mixed")
    fields = {1: 4, 2: 7, 3: 9}[cfgs[0]["dims"]]
    dev = dict(dtype=torch.float64, device="cuda")
    if case["kind"] == "fields":
        s.f = _populations(cfgs[0], seed)
        s.back = torch.empty_like(s.f)
        s.profile, s.stats = torch.empty(case["ny"], **dev), torch.empty(6, **dev)
    else:
        s.start = _start(case, cfgs, seed)
    nodes = [fields * int(np.prod(_shape(c))) for c in cfgs]
    s.moments = torch.empty(sum(nodes), **dev)  # every instance's fields, one after another
    s.parts = torch.split(s.moments, nodes)
    return s


def run(s):
    case = s.case
    if case["kind"] == "gradient":
        tau, g, lo, hi = s.params
        J = glbm.flow_rate(tau, g, s.config, case["steps"], case["every"], u_wall_lo=lo,
                           u_wall_hi=hi)
        d = torch.autograd.grad(J, s.params)
        return {"J": J.detach(), "dtau": d[0], "dg": d[1], "dwalls": torch.stack(d[2:])}
    lat = s.lat
    if case["kind"] == "fields":
        lat.set_populations(0, s.f)
        lat.moments(0, out=s.parts[0])
        lat.channel_diagnostics(0, s.profile, s.stats)
        sums = np.array(lat.conservation(0))
        lat.get_populations(0, out=s.back)
        return {"moments": s.moments, "profile": s.profile, "stats": s.stats, "sums": sums,
                "populations": s.back}
    for i, start in enumerate(s.start):
        lat.set_equilibrium(i, *start)
    lat.step(case["steps"])
    for i, out in enumerate(s.parts):
        lat.moments(i, out=out)
    return s.moments


def work(case):
    """Bytes and operations no program can do without: each step reads and
    writes every population once (1D lattices stay on the chip), the analysis
    reads them once; about ten operations per population update."""
    if case["kind"] == "gradient":
        q, nodes, e = (2 * case["k"] + 3) ** 2, case["nx"] * case["ny"], case["prec"] // 8
        # forward step and recompute; the adjoint step reads a state and moves
        # the FP64 adjoint populations
        return {"bytes": float(q * nodes * case["steps"] * (5 * e + 16)),
                "flops": 40.0 * q * nodes * case["steps"]}
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _configs(case, 0):
        nodes, e = int(np.prod(_shape(c))), 8 if c["prec"] == glbm.FP64 else 4
        k = c["k"]
        q = (2 * k + 3) ** c["dims"]
        if c.get("x_level") == 1:
            q = 3 * (2 * k + 3 + (1 if c.get("zv_axes") else 0))
        fields = {1: 4, 2: 7, 3: 9}[c["dims"]]
        if case["kind"] == "fields":
            total["bytes"] += nodes * (q * (16 + 3 * e) + 8 * fields)
            total["flops"] += 10.0 * q * nodes
            continue
        io = 8 * nodes * (c["dims"] + 1 + fields)  # start fields read, moments written
        per_step = 0 if c["dims"] == 1 else 2 * q * nodes * e
        total["bytes"] += io + per_step * case["steps"] + (0 if c["dims"] == 1 else 2 * q * nodes * e)
        total["flops"] += 10.0 * q * nodes * (case["steps"] + 2)
    return total


# ---- 64-bit references ----------------------------------------------------
# The method in plain torch: the equilibrium by N-fold convolution of the
# three-outcome distribution (Sec. 2), streaming by rolls, diffuse walls,
# BGK relaxation with the linearised force, raw sums for the moments.


def _equilibrium(N, zv, u):
    """E_i(u) of one axis, stacked along a new first dimension."""
    if zv:
        e = _equilibrium(N, 0, 0.5 * u)
        z = torch.zeros_like(e[:1])
        return 0.5 * (torch.cat([z, e]) + torch.cat([e, z]))
    a = u * u / (2.0 * N * N)
    pm, p0, pp = 1 / 6 - u / (2.0 * N) + a, 2 / 3 - 2 * a, 1 / 6 + u / (2.0 * N) + a
    e = torch.ones_like(u)[None]
    for _ in range(N):
        z = torch.zeros_like(e[:1])
        e = torch.cat([e, z, z]) * pm + torch.cat([z, e, z]) * p0 + torch.cat([z, z, e]) * pp
    return e


def _axis_weights(N, zv):
    return _equilibrium(N, zv, torch.zeros((), dtype=torch.float64))


def _velocities(N, zv):
    return [2 * i - (2 * N + 1) for i in range(2 * N + 2)] if zv else list(range(-N, N + 1))


class _Reference:
    """One instance in FP64; populations f[(iz,) iy, ix, (z,) y, x] (1D: f[ix, x])."""

    def __init__(self, c, tau=None, walls=None, g=None, device="cuda"):
        self.d = c["dims"]
        N = c["k"] + 1
        zy = 1 if c.get("zv_axes", 0) else 0
        self.levels = [(c.get("x_level") or N, 0)] + [(N, zy)] * (self.d - 1)  # x, y, z
        if self.d == 1:
            self.levels = [(N, 0)]
        self.v = [_velocities(*lv) for lv in self.levels]
        self.W = [_axis_weights(*lv).to(device) for lv in self.levels]
        theta = [(4 * n + 3) / 3 if z else n / 3 for n, z in self.levels]
        if tau is None:
            height = c["ny"] if self.d >= 2 else c["nx"]
            tau = c["kn"] * height / math.sqrt(2 * theta[min(1, self.d - 1)])
        self.omega = 1.0 / (tau + 0.5)
        self.theta_x = theta[0]
        self.g = c.get("g", 0.0) if g is None else g
        u = walls if walls is not None else [c.get("u_wall_lo", 0.0), c.get("u_wall_hi", 0.0)]
        u = [torch.as_tensor(w, dtype=torch.float64, device=device) for w in u]
        self.wall = [_equilibrium(*self.levels[0], w) for w in u]
        self.device = device

    def axis(self, a, t):
        """A per-velocity vector of axis a, shaped to broadcast against f."""
        shape = [1] * (2 * self.d)
        shape[self.d - 1 - a] = -1
        return t.reshape(shape)

    def vel(self, a):
        return self.axis(a, torch.tensor(self.v[a], dtype=torch.float64, device=self.device))

    def equilibrium(self, rho, us):
        f = rho
        for a, u in enumerate(us):
            e = _equilibrium(*self.levels[a], u)
            f = f * e.reshape([e.shape[0] if i == self.d - 1 - a else 1 for i in range(self.d)] +
                              list(u.shape))
        return f

    def stream(self, f):
        d = self.d
        if d == 1:  # halfway bounce-back at both ends
            N, L = self.levels[0][0], f.shape[-1]
            out = torch.empty_like(f)
            for n in range(-N, N + 1):
                m = abs(n)
                src, back = f[N + n], f[N - n]
                if n > 0:
                    out[N + n] = torch.cat([back[:m].flip(0), src[:L - m]])
                elif n < 0:
                    out[N + n] = torch.cat([src[m:], back[L - m:].flip(0)])
                else:
                    out[N] = src
            return out
        for a in ([0, 2] if d == 3 else [0]):  # the periodic axes
            dim = d - 1 - a
            f = torch.stack([torch.roll(f.select(dim, i), v, dims=2 * d - 2 - a)
                             for i, v in enumerate(self.v[a])], dim=dim)
        # f now stands at the column it reaches; move it along y between the walls
        yd, qd = 2 * d - 2, d - 2  # the y rows, the y velocities
        vy, ny = self.v[1], f.shape[yd]
        den = sum(v * float(self.W[1][i]) for i, v in enumerate(vy) if v > 0)
        sums = [i for i in range(d) if i != qd]
        absorbed = [0.0, 0.0]
        for i, v in enumerate(vy):
            if v == 0:
                continue
            part = f.select(qd, i).narrow(yd - 1, 0 if v < 0 else ny - v, abs(v))
            part = part.sum(dim=yd - 1)  # the rows that leave
            absorbed[0 if v < 0 else 1] = absorbed[0 if v < 0 else 1] + \
                part.sum(dim=tuple(range(d - 1)))
        rows = []
        for i, v in enumerate(vy):
            p = f.select(qd, i)
            if v != 0:
                h = 0 if v > 0 else 1
                ghost = absorbed[h] / den * float(self.W[1][i])
                e = self.wall[h].reshape([1] * (d - 2) + [-1] + [1] * (d - 1))
                ghost = ghost * e
                if d == 3:
                    ghost = ghost * self.W[2].reshape(-1, 1, 1, 1)
                ghost = ghost.unsqueeze(yd - 1).expand(p.shape[:yd - 1] + (abs(v),) +
                                                       p.shape[yd:])
                keep = p.narrow(yd - 1, max(0, -v), ny - abs(v))
                p = torch.cat([ghost, keep] if v > 0 else [keep, ghost], dim=yd - 1)
            rows.append(p)
        return torch.stack(rows, dim=qd)

    def mean(self, f):
        q = tuple(range(self.d))
        rho = f.sum(dim=q)
        return rho, [(f * self.vel(a)).sum(dim=q) / rho for a in range(self.d)]

    def step(self, X):
        f = self.stream(X)
        rho, us = self.mean(f)
        X = f + self.omega * (self.equilibrium(rho, us) - f)
        if self.d >= 2:
            w = self.vel(0) * self.g / self.theta_x
            for a in range(self.d):
                w = w * self.axis(a, self.W[a])
            X = X + w
        return X

    def moments(self, X):
        f = self.stream(X)
        q = tuple(range(self.d))
        rho, us = self.mean(f)
        c = [self.vel(a) - us[a] for a in range(self.d)]
        c2 = sum(x * x for x in c)
        heat = [0.5 * (f * x * c2).sum(dim=q) for x in c]
        T = (f * c2).sum(dim=q) / (self.d * rho)
        if self.d == 1:
            return torch.stack([rho, us[0], T, heat[0]])
        sxy = (f * c[0] * c[1]).sum(dim=q)
        out = [rho, us[0], us[1], T, heat[0], heat[1], sxy]
        return torch.stack(out + ([us[2], heat[2]] if self.d == 3 else []))


def exact(case, seed):
    if case["kind"] == "gradient":
        # from rest between uniform walls the flow does not depend on x, so one
        # column gives the whole flow rate
        p = [torch.tensor(v, dtype=torch.float64, requires_grad=True)
             for v in _gradient_inputs(case, seed)]
        c = dict(dims=2, k=case["k"], nx=1, ny=case["ny"])
        r = _Reference(c, tau=p[0], g=p[1], walls=p[2:], device="cpu")
        shape = (case["ny"], 1)
        zero = torch.zeros(shape, dtype=torch.float64)
        X = r.equilibrium(torch.ones(shape, dtype=torch.float64), [zero, zero])
        for _ in range(case["steps"]):
            X = r.step(X)
        f = r.stream(X)
        J = (f * r.vel(0)).sum()
        d = torch.autograd.grad(J, p)
        return {"J": J.detach(), "dtau": d[0], "dg": d[1], "dwalls": torch.stack(d[2:])}
    cfgs = _configs(case, seed)
    with torch.no_grad():
        if case["kind"] == "fields":
            c = cfgs[0]
            f = _populations(c, seed)
            q = 2 * c["k"] + 3
            r = _Reference(c)
            m = r.moments(f.reshape((q, q) + _shape(c)))
            mean_u, mean_j = m[1].mean(dim=1), (m[0] * m[1]).mean(dim=1)
            H, theta = c["ny"], (c["k"] + 1) / 3
            tau = 1.0 / r.omega - 0.5
            u0 = c["g"] * H * H / (8 * theta * tau)
            nan = float("nan")
            flow = float(mean_u.sum()) / (c["kn"] * 4 * u0 * H) if c["g"] else nan
            lo, hi = c["u_wall_lo"], c["u_wall_hi"]
            ulo = float(1.5 * mean_u[0] - 0.5 * mean_u[1])
            uhi = float(1.5 * mean_u[-1] - 0.5 * mean_u[-2])
            stats = [float(mean_j.sum()), flow, ulo, uhi, (ulo - lo) / (hi - lo),
                     (hi - uhi) / (hi - lo)]
            sums = [float(m[0].sum()), float((m[0] * m[1]).sum()), float((m[0] * m[2]).sum())]
            return {"moments": m.reshape(-1), "profile": mean_u,
                    "stats": torch.tensor(stats, dtype=torch.float64), "sums": np.array(sums),
                    "populations": f}
        out = []
        for c, start in zip(cfgs, _start(case, cfgs, seed)):
            r = _Reference(c)
            X = r.equilibrium(start[0], start[1:])
            for _ in range(case["steps"]):
                X = r.step(X)
            out.append(r.moments(X).reshape(-1))
        return torch.cat(out)
