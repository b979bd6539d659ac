"""The work that programs built on this solver have it do, as cases that can be timed.

A case is one simulation (or a batch of them) taken through the public calls of
`paper_1507_07294_gb300.lbm`: fields in page-locked host memory go in (`lbm_init_phi`),
the run advances by a number of time steps, and its fields come back (`lbm_read_fields`).
Sizes, parameters and options are those of `inputs.py`, the serving mix and the tests.

`exact` restates the method in float64 torch from the paper's formulas (arXiv:1507.07294,
equation numbers in order of appearance); it uses none of this repository's code.
"""
import math
from dataclasses import replace

import numpy as np
import torch

from paper_1507_07294_gb300 import inputs as I
from paper_1507_07294_gb300 import lbm as L


def _case(name, kind, problem, nx, ny, nz, steps, storage="fp32", pattern="ab", walls=None,
          srt=False, stencil="d3q15", fields="all"):
    return {"name": name, "kind": kind, "problem": problem, "nx": nx, "ny": ny, "nz": nz,
            "steps": steps, "storage": storage, "pattern": pattern,
            "walls": (problem == "rt") if walls is None else walls, "srt": srt,
            "stencil": stencil, "fields": fields}


def listed():
    return [
        # the smallest box of the serving mix, watched step by step: ten calls that each
        # advance one step and wait for its mass and momentum
        _case("watch_32", "watch", "droplet", 32, 32, 32, 10, fields="phi"),
        # the static droplet on 32^3, a stretch of its 500 steps
        _case("droplet_32", "run", "droplet", 32, 32, 32, 100),
        # one small request as a server takes it: create, initialise, step, read, close
        _case("request_64", "request", "rt", 64, 64, 64, 128, walls=True, fields="phi"),
        # Rayleigh-Taylor at Re = 256, the paper's setup on 64 x 64 x 256
        _case("rt_64", "run", "rt", 64, 64, 256, 64),
        # the largest box of the serving mix
        _case("rt_128", "run", "rt", 128, 128, 512, 32),
        # the benchmark workload: 67M cells, FP32
        _case("rt_256", "run", "rt", 256, 256, 1024, 40, fields="phi"),
        # the same grid with populations stored in 16 bits
        _case("rt_256_fp16", "run", "rt", 256, 256, 1024, 40, storage="fp16", fields="phi"),
        # the in-place pattern with 16-bit populations, chosen where memory is short
        _case("inplace_128_bf16", "run", "rt", 128, 128, 512, 32, storage="bf16", pattern="aa"),
        # a box whose sides are no multiples of anything
        _case("ragged_150", "run", "rt", 150, 141, 601, 24),
        # Zalesak's sphere in the paper's 100^3 box (interface tracking, rows of 100)
        _case("zalesak_100", "run", "zalesak", 100, 100, 100, 64, fields="phi"),
        # the deformation flow (interface tracking) on 256^3
        _case("deform_256", "run", "deformation", 256, 256, 256, 32, fields="phi"),
        # sixteen requests of the serving mix advanced together by two quanta of 64 steps
        _case("batch_mix", "batch", "rt", 64, 64, 256, 129, fields="phi"),
    ]


def draw(rng):
    """A case of the same ranges: boxes from 16^3 to 67M cells, rows of every kind."""
    problem = rng.choice(["droplet", "droplet", "rt", "rt", "rt", "deformation", "zalesak"])
    tracking = problem in ("deformation", "zalesak")
    cells = math.exp(rng.uniform(math.log(16 ** 3), math.log(2 ** 24 if tracking else 2 ** 26)))
    side = cells ** (1 / 3)
    if tracking:
        nx = ny = nz = max(8, round(side))
        if rng.random() < 0.4 and nx >= 32:
            nx = ny = nz = nx // 32 * 32
    else:
        nx = side * math.exp(rng.uniform(-0.6, 0.3))
        kind = rng.random()
        if kind < 0.35 and nx >= 24:    # rows that are whole pairs of 32 cells
            nx = max(64, round(nx / 64) * 64)
        elif kind < 0.6 and nx >= 24:   # whole groups of 32 cells
            nx = max(32, round(nx / 32) * 32)
        else:                           # any length
            nx = max(5, round(nx))
        rest = cells / nx
        ny = max(3, round(math.sqrt(rest) * math.exp(rng.uniform(-0.5, 0.2))))
        if rng.random() < 0.5 and ny >= 12:
            ny = round(ny / 8) * 8
        nz = max(3, int(rest / ny))
    n = nx * ny * nz
    # at most about a tenth of the largest listed case's cell updates
    steps = int(min(100, max(2, rng.uniform(0.3, 1.0) * 1.5e8 / n)))
    storage = "fp32" if tracking else rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16"])
    pattern = "aa" if rng.random() < 0.25 else "ab"
    c = _case("", "run", problem, nx, ny, nz, steps, storage, pattern,
              walls=not tracking and (problem == "rt" or rng.random() < 0.3),
              srt=not tracking and rng.random() < 0.1,
              stencil="d3q7" if not tracking and rng.random() < 0.1 else "d3q15",
              fields="phi" if n > 2 ** 24 or tracking else "all")
    if not tracking and n <= 2 ** 18 and rng.random() < 0.3:
        c["kind"] = rng.choice(["watch", "request"])
        if c["kind"] == "watch":
            c["steps"] = 10
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs ------------

# the runs of the batch case: (W, nz, count)
MIX = ((32, 32, 6), (64, 64, 6), (64, 256, 3), (128, 512, 1))


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _coords(nx, ny, nz, walls):
    kw = dict(dtype=torch.float64, device=_device())
    x, y, z = (torch.arange(n, **kw) for n in (nx, ny, nz))
    return x[None, None, :], y[None, :, None], (z + 0.5 if walls else z)[:, None, None]


def _fields(c, seed):
    """(parameters without fields, phi0, u0) of a case: the workload's initial condition
    with its phases, radius, centre and amplitudes drawn from the seed; u0 may be None."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    x, y, z = _coords(nx, ny, nz, c["walls"])
    u0 = None
    if c["problem"] == "rt":
        W = nx
        w = I.rayleigh_taylor(W=W, Re=c.get("re", 256.0 if nx <= 64 else 4000.0),
                              atwood=c.get("at", 0.5), sigma=c.get("sigma", 1e-4), nz=nz,
                              with_fields=False)
        a, b = 2 * math.pi * rng.random(2)
        amp = 0.05 * min(nx, nz / 4) * (0.8 + 0.4 * rng.random())
        h = amp * (torch.cos(2 * math.pi * x / nx + a) + torch.cos(2 * math.pi * y / ny + b))
        phi = torch.tanh(2.0 * (z - h - nz / 2.0) / w.D)
        # settled noise of the start of a run: keeps no two rows alike
        phi = phi * (1.0 - 1e-3 * torch.sin(0.37 * x + 0.71 * y + 0.53 * z + a) ** 2)
    elif c["problem"] == "droplet":
        w = I.droplet(n=8, R=2.0)
        R = min(nx, ny, nz) * (0.22 + 0.06 * rng.random())
        cx, cy, cz = (n * (0.45 + 0.1 * rng.random()) for n in (nx, ny, nz))
        r = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2)
        phi = torch.tanh(2.0 * (R - r) / w.D)
        # a weak Taylor-Green stirring, at rest where walls stand
        U, a, b = 0.004 + 0.004 * rng.random(), *(2 * math.pi * rng.random(2))
        kx, ky = 2 * math.pi / nx, 2 * math.pi / ny
        s = torch.sin(math.pi * z / nz) ** 2 if c["walls"] else 1.0 + 0.0 * z
        ux = U * torch.sin(kx * x + a) * torch.cos(ky * y + b) * s
        uy = -U * torch.cos(kx * x + a) * torch.sin(ky * y + b) * s
        u0 = torch.stack([v.expand(nz, ny, nx) for v in (ux, uy, 0.0 * ux)])
    else:
        w = (I.deformation if c["problem"] == "deformation" else I.zalesak)(n=8)
        n = nx
        R = (0.15 if c["problem"] == "deformation" else 0.4) * n * (0.9 + 0.1 * rng.random())
        c0 = (0.35 if c["problem"] == "deformation" else 0.5) * n * (0.97 + 0.06 * rng.random())
        r = torch.sqrt((x - c0) ** 2 + (y - c0) ** 2 + (z - c0) ** 2)
        d = R - r
        if c["problem"] == "zalesak":  # the slot from the bottom of the sphere to its centre
            qy, qz = torch.abs(y - c0) - 0.08 * n, z - c0
            out = torch.sqrt(qy.clamp(min=0) ** 2 + qz.clamp(min=0) ** 2)
            d = torch.minimum(d, out + torch.maximum(qy, qz).clamp(max=0))
        phi = torch.tanh(2.0 * d / w.D)
        U = w.velocity[1]
        w = replace(w, mobility=U * R / (400.0 if c["problem"] == "deformation" else 200.0),
                    velocity=(w.velocity[0], U, 3000.0))
    phi = phi.expand(nz, ny, nx).contiguous()
    w = replace(w, nx=nx, ny=ny, nz=nz, walls_z=c["walls"], srt_flow=c["srt"],
                stencil=c["stencil"], phi0=None, u0=None, p0=None)
    return w, phi, u0


def _batch_runs(c, seed):
    """The cases of the batch's runs: Rayleigh-Taylor requests of the serving mix."""
    rng = np.random.default_rng(seed + 7919)
    runs = []
    for W, nz, count in MIX:
        for _ in range(count):
            r = dict(c, nx=W, ny=W, nz=nz, re=float(rng.uniform(100, 4000)),
                     at=float(rng.uniform(0.1, 0.9)), sigma=float(rng.uniform(1e-3, 1e-2)))
            runs.append((r, seed * 64 + len(runs)))
    return runs


def _pinned(t):
    """A page-locked host copy (numpy) of a tensor."""
    h = torch.empty(t.shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    h.copy_(t)
    return h.numpy()


def _out_buffers(c):
    n = (c["nz"], c["ny"], c["nx"])
    names = ("phi",) if c["fields"] == "phi" else ("phi", "rho", "p", "u", "mu")
    return {k: torch.empty((3,) + n if k == "u" else n, dtype=torch.float64,
                           pin_memory=torch.cuda.is_available()).numpy() for k in names}


def _mask(c):
    return L.LBM_FIELD_PHI if c["fields"] == "phi" else L.LBM_FIELD_ALL


class _Run:
    """A run's solver and its page-locked buffers."""

    def __init__(self, c, seed, stream=None):
        w, phi, u0 = _fields(c, seed)
        self.case, self.phi, self.u = c, _pinned(phi), None if u0 is None else _pinned(u0)
        self.out = _out_buffers(c)
        self.stream = stream
        self.solver = L.Solver(w, stream=None if stream is None else stream.cuda_stream,
                               init=False, pattern=c["pattern"], storage=c["storage"])
        self.ctx = self.solver.ctx

    def init(self):
        L.lbm_init_phi(self.ctx, self.phi, self.u)

    def read(self):
        return L.lbm_read_fields(self.ctx, _mask(self.case), out=self.out)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        runs = [_Run(r, s, torch.cuda.Stream()) for r, s in _batch_runs(c, seed)]
        stream = torch.cuda.Stream()
        batch = L.Batch(stream=stream.cuda_stream)
        batch.set_split(1 << 20)  # the largest boxes fill the GPU by themselves
        return {"case": c, "runs": runs, "batch": batch, "stream": stream}
    if c["kind"] == "request":
        w, phi, u0 = _fields(c, seed)
        w = replace(w, phi0=phi.cpu().numpy(), u0=None if u0 is None else u0.cpu().numpy())
        return {"case": c, "workload": w}
    r = _Run(c, seed)
    if c["kind"] == "watch":
        r.init()
    return {"case": c, "run": r}


def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        runs = state["runs"]
        for r in runs:
            r.init()
            L.lbm_step(r.ctx, 1)
        left = c["steps"] - 1
        while left > 0:  # a server's quanta
            q = min(64, left)
            state["batch"].step([r.ctx for r in runs], q)
            left -= q
        return {"run%02d" % k: r.read() for k, r in enumerate(runs)}
    if c["kind"] == "request":
        with L.Solver(state["workload"], pattern=c["pattern"], storage=c["storage"]) as s:
            s.step(c["steps"])
            return s.fields(_mask(c))
    r = state["run"]
    if c["kind"] == "watch":
        mass, momentum = [], []
        for _ in range(c["steps"]):
            total, j = L.lbm_step_reduce(r.ctx, 1)
            mass.append(total)
            momentum.append(j)
        return {"mass": np.array(mass), "momentum": np.array(momentum), **r.read()}
    r.init()
    L.lbm_step(r.ctx, c["steps"])
    return r.read()


# --------------------------------------------------------------- what a pass needs ----

def _work_one(c):
    n, tracking = c["nx"] * c["ny"] * c["nz"], c["problem"] in ("deformation", "zalesak")
    pop = 4 if c["storage"] == "fp32" else 2
    # a time step reads and writes every cell's populations (7 + 15, tracking: 7) and its
    # phi u once
    state = (7 if tracking else 22) * pop + 3 * 4
    planes = 1 if c["fields"] == "phi" else 7
    inputs = 0 if c["kind"] == "watch" else 8 * (4 if c["problem"] == "droplet" else 1)
    return {"bytes": n * (2 * state * c["steps"] + inputs + 8 * planes),
            "flops": n * c["steps"] * (110 if tracking else 560)}


def work(case):
    if case["kind"] != "batch":
        return _work_one(case)
    parts = [_work_one(r) for r, _ in _batch_runs(case, 0)]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# -------------------------------------------------------- the method in 64 bits -------

C7 = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1))
C15 = C7 + ((1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1),
            (1, -1, -1), (-1, 1, 1))
W15 = (2 / 9,) + (1 / 9,) * 6 + (1 / 72,) * 8


def _matrix(velocities, rows):
    return torch.tensor([[float(r(*c)) for c in velocities] for r in rows], dtype=torch.float64)


_c2 = lambda x, y, z: x * x + y * y + z * z  # noqa: E731
_q = lambda x, y, z: (5 * _c2(x, y, z) - 13) / 2  # noqa: E731
M7 = _matrix(C7, (lambda x, y, z: 1, lambda x, y, z: x, lambda x, y, z: y, lambda x, y, z: z,
                  lambda x, y, z: 6 - 7 * _c2(x, y, z), lambda x, y, z: 3 * x * x - _c2(x, y, z),
                  lambda x, y, z: y * y - z * z))
M15 = _matrix(C15, (lambda x, y, z: 1, lambda x, y, z: _c2(x, y, z) - 2,
                    lambda x, y, z: (15 * _c2(x, y, z) ** 2 - 55 * _c2(x, y, z) + 32) / 2,
                    lambda x, y, z: x, lambda x, y, z: _q(x, y, z) * x,
                    lambda x, y, z: y, lambda x, y, z: _q(x, y, z) * y,
                    lambda x, y, z: z, lambda x, y, z: _q(x, y, z) * z,
                    lambda x, y, z: 3 * x * x - _c2(x, y, z), lambda x, y, z: y * y - z * z,
                    lambda x, y, z: x * y, lambda x, y, z: y * z, lambda x, y, z: x * z,
                    lambda x, y, z: x * y * z))


class _Exact:
    """One run in float64: the scheme of Sec. II of the paper, collisions in moment space."""

    def __init__(self, c, seed):
        w, phi, u0 = _fields(c, seed)
        self.w, self.walls, self.track, self.t = w, c["walls"], w.velocity, 0
        self.kappa, self.beta = 3 * w.D * w.sigma / 8, 3 * w.sigma / (4 * w.D)
        self.eta = w.mobility / (w.A * (1 / w.sf[1] - 0.5))
        self.shape, dev = (w.nz, w.ny, w.nx), phi.device
        self.M7, self.M15 = M7.to(dev), M15.to(dev)
        self.M7i, self.M15i = (torch.linalg.inv(m).contiguous().to(dev) for m in (M7, M15))
        u = torch.zeros((3,) + self.shape, dtype=torch.float64, device=dev)
        if self.track:
            u = self.velocity(0)
        elif u0 is not None:
            u = u0
        mu, phiu = self.mu(phi), phi * u
        wf = (1 - 3 * w.A,) + (w.A / 2,) * 6
        self.f = torch.stack([wf[i] * self.eta * mu + wf[i] * self.dot(C7[i], phiu) / w.A
                              for i in range(7)])
        self.f[0] = phi + (wf[0] - 1) * self.eta * mu
        self.g, self.old = None, None
        if not self.track:
            rho, uu = self.rho(phi), (u * u).sum(0)
            self.g = torch.stack([rho * W15[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu)
                                  for i in range(15) for cu in (self.dot(C15[i], u),)])

    def dot(self, c, v):
        return sum((s * a for s, a in zip(c, v) if s), torch.zeros_like(v[0]))

    def near(self, a, c):
        """a(x + c): periodic, in z between walls the wall's own neighbour."""
        a = torch.roll(a, (-c[1], -c[0]), (-2, -1))
        if c[2] and self.walls:
            k = (torch.arange(a.shape[0], device=a.device) + c[2]).clamp(0, a.shape[0] - 1)
            return a[k]
        return torch.roll(a, -c[2], 0) if c[2] else a

    def lap(self, a):
        if self.w.stencil == "d3q7":
            return sum(self.near(a, c) for c in C7[1:]) - 6 * a
        return sum(6 * W15[i] * (self.near(a, C15[i]) - a) for i in range(1, 15))

    def grad(self, a):
        out = torch.zeros((3,) + self.shape, dtype=a.dtype, device=a.device)
        d3q7 = self.w.stencil == "d3q7"
        for i, c in enumerate(C7 if d3q7 else C15):
            if i:
                v = (0.5 if d3q7 else 3 * W15[i]) * self.near(a, c)
                for k in range(3):
                    if c[k]:
                        out[k] += c[k] * v
        return out

    def mu(self, phi):
        return 4 * self.beta * phi * (phi * phi - 1) - self.kappa * self.lap(phi)

    def rho(self, phi):
        return 0.5 * (1 + phi) * self.w.rho_l + 0.5 * (1 - phi) * self.w.rho_g

    def velocity(self, t):
        """Eqs. 37 and 41 at the integer nodes."""
        kind, U = self.track[0], self.track[1]
        nz, ny, nx = self.shape
        x, y, z = _coords(nx, ny, nz, False)
        one = torch.ones(self.shape, dtype=torch.float64, device=x.device)
        if kind == "rotation":
            om = U * math.pi / ny
            return torch.stack([0 * one, -om * (z - ny / 2) * one, om * (y - ny / 2) * one])
        a, p = U * math.cos(math.pi * t / self.track[2]), math.pi / nx
        s1, s2 = (lambda v: torch.sin(p * v)), (lambda v: torch.sin(2 * p * v))
        return torch.stack([2 * a * s1(x) ** 2 * s2(y) * s2(z), -a * s2(x) * s1(y) ** 2 * s2(z),
                            -a * s2(x) * s2(y) * s1(z) ** 2])

    def macro(self):
        """phi, mu and (coupled) rho, u, p, grad rho, F of the current populations."""
        w, phi = self.w, self.f.sum(0)
        mu = self.mu(phi)
        if self.track:
            return phi, mu, self.rho(phi), self.velocity(self.t), None, None, None
        rho, gp, lm = self.rho(phi), self.grad(phi), self.lap(mu)
        gr, drho = 0.5 * (w.rho_l - w.rho_g) * gp, w.rho_l - w.rho_g
        fsg = mu * gp
        for k in range(3):
            if w.g[k]:
                fsg[k] += rho * w.g[k]
        den = rho - 0.25 * drho * w.mobility * lm
        u = torch.stack([(sum(C15[i][k] * self.g[i] for i in range(15) if C15[i][k])
                          + 0.5 * fsg[k]) / den for k in range(3)])
        p = 3 / 7 * (self.g[1:].sum(0) + 0.5 * (u * gr).sum(0) - rho * (u * u).sum(0) / 3)
        return phi, mu, rho, u, p, gr, fsg + 0.5 * drho * w.mobility * lm * u

    def stream(self, a, velocities):
        for i, c in enumerate(velocities):
            if any(c):
                a.append(torch.roll(a[0][i], (c[2], c[1], c[0]), (0, 1, 2)))
            else:
                a.append(a[0][i])
        if self.walls:
            for i, c in enumerate(velocities):
                if c[2]:  # halfway bounce-back at both walls
                    k = 0 if c[2] > 0 else -1
                    a[1 + i][k] = a[0][velocities.index(tuple(-v for v in c))][k]
        return torch.stack(a[1:])

    def relax(self, m, eq, rates, src):
        return m - rates * (m - eq) + (1 - 0.5 * rates) * src

    def step(self):
        w = self.w
        phi, mu, rho, u, p, gr, F = self.macro()
        now = phi * u
        dt = torch.zeros_like(now) if self.old is None else now - self.old
        self.old = now
        m = torch.tensordot(self.M7, self.f, 1)
        eq = (phi, now[0], now[1], now[2], 6 * phi - 21 * w.A * self.eta * mu, 0.0, 0.0)
        src = (0.0, dt[0], dt[1], dt[2], 0.0, 0.0, 0.0)
        for k in range(7):
            m[k] = self.relax(m[k], eq[k], w.sf[k], src[k])
        self.f = self.stream([torch.tensordot(self.M7i, m, 1)], C7)
        self.t += 1
        if self.track:
            return
        m = torch.tensordot(self.M15, self.g, 1)
        (ux, uy, uz), (Fx, Fy, Fz), uu = u, F, (u * u).sum(0)
        Y, s = gr / 3 + F, -7 / 3
        udr, udF = (u * gr).sum(0), (u * F).sum(0)
        eq = (0.0, 3 * p + rho * uu, -45 * p - 5 * rho * uu, rho * ux, s * rho * ux, rho * uy,
              s * rho * uy, rho * uz, s * rho * uz, rho * (2 * ux * ux - uy * uy - uz * uz),
              rho * (uy * uy - uz * uz), rho * ux * uy, rho * uy * uz, rho * ux * uz, 0.0)
        src = (udr, -udr / 3 + 2 * udF, -7 / 3 * udr - 10 * udF, Fx, s * Fx, Fy, s * Fy, Fz,
               s * Fz, 4 * ux * Y[0] - 2 * uy * Y[1] - 2 * uz * Y[2],
               2 * uy * Y[1] - 2 * uz * Y[2], ux * Y[1] + uy * Y[0], uy * Y[2] + uz * Y[1],
               ux * Y[2] + uz * Y[0], 0.0)
        nu = 0.5 * (1 + phi) * w.nu_l + 0.5 * (1 - phi) * w.nu_g
        visc = 1 / (3 * nu + 0.5)
        for k in range(15):
            m[k] = self.relax(m[k], eq[k], visc if w.srt_flow or 9 <= k <= 13 else w.sg[k], src[k])
        self.g = self.stream([torch.tensordot(self.M15i, m, 1)], C15)

    def fields(self, which):
        phi, mu, rho, u, p = self.macro()[:5]
        out = {"phi": phi}
        if which == "all":
            out.update(rho=rho, p=p, u=u, mu=mu)
        return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        out = {}
        for k, (r, s) in enumerate(_batch_runs(c, seed)):
            e = _Exact(r, s)
            for _ in range(c["steps"]):
                e.step()
            out["run%02d" % k] = e.fields(c["fields"])
        return out
    e, mass = _Exact(c, seed), []
    for _ in range(c["steps"]):
        e.step()
        mass.append(float(e.f.sum()))
    out = e.fields(c["fields"])
    if c["storage"] != "fp32" and "mu" in out:
        out["mu"] = None  # a second difference of phi: with 16 bits mostly their rounding
    if c["kind"] == "watch":
        # the momenta of all cells cancel but for rounding, and so do the two halves of a
        # Rayleigh-Taylor box: no value of these sums stands in 64 bits
        out = {"mass": np.array(mass) if c["problem"] == "droplet" else None,
               "momentum": None, **out}
    return out
