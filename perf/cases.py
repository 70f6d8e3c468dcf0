"""The work this library is run for, as cases that can be timed and checked.

A case is one job through the public Python entry points: initialise a lattice
(or a batch) from fields on the GPU or in pinned host memory, advance it, and
read density and velocity (and what else that job's user reads) back. The
listed cases follow the repository's own workloads (paper_1801_04586_gb300/
workloads, the benchmark's lines and the tests' shapes); draw() spreads the
same kinds of job over their ranges of size, storage, pattern and boundary.

    kind "flow"     one lattice: init, nsteps steps, Eq. 9 read-out
    kind "host"     the same job through pinned host buffers with the sums of
                    every step (Lattice.run_host)
    kind "adjoint"  gradient of a final-velocity loss by the force field
    kind "batch"    many independent channels and ducts stepped together
"""
import math
import random

import numpy as np
import torch

from paper_1801_04586_gb300 import Batch, Lattice
from paper_1801_04586_gb300.autograd import final_velocity

U0_TG, RE_TG = 0.005, 50.0  # the Taylor-Green vortex of Sec. III.D


def _flow(name, nx, ny, nz, steps, nu, walls=0, storage="f32", pattern="ab", lattice=19, force="uniform", f0=1e-5,
          umax=0.02, pops=False):
    return dict(name=name, kind="flow", nx=nx, ny=ny, nz=nz, steps=steps, nu=nu, walls=walls, storage=storage,
                pattern=pattern, lattice=lattice, force=force, f0=f0, umax=umax, pops=pops)


def listed():
    return [
        # The force-driven Poiseuille channel the method is validated on (Sec. III.B): a lattice so small that a
        # step is a launch's latency; users run thousands of steps and read the profile, or the populations.
        _flow("poiseuille_channel", 16, 32, 32, 200, 0.1, walls=4, f0=1e-6, umax=1e-3, pops=True),
        # The decaying Taylor-Green vortex of the convergence study (Sec. III.D) at its finest grid: thin, with a
        # force field whose strength changes every step.
        dict(name="taylor_green_128", kind="flow", nx=128, ny=128, nz=5, steps=100, nu=U0_TG * 128 / RE_TG, walls=0,
             storage="f32", pattern="ab", lattice=19, force="taylor_green", f0=0.0, umax=U0_TG, pops=False),
        # A channel of sides no tile divides, with a body-force field: what a user's own geometry looks like.
        _flow("channel_ragged_field", 150, 91, 61, 40, 0.03, walls=2, force="field"),
        # The throughput workload (the benchmark's line): periodic Kolmogorov box.
        _flow("kolmogorov_256", 256, 256, 256, 25, 0.01, force="profile"),
        # The same box as a job through host memory, the way a service runs it: upload, steps with the sums of mass
        # and momentum after each, download.
        dict(name="kolmogorov_256_host", kind="host", nx=256, ny=256, nz=256, steps=20, nu=0.01, walls=0,
             storage="f32", pattern="ab", lattice=19, force="profile", f0=1e-5, umax=0.02, pops=False),
        # The mixed-precision square duct (Sec. III.C): 16-bit storage with stochastic rounding, four walls.
        _flow("duct_f16sr", 512, 128, 128, 24, 0.05, walls=6, storage="f16sr", f0=2e-6, umax=1e-2),
        # A memory-bound user's box: 16-bit storage in place, an eighth of the FP32 two-buffer footprint per node.
        _flow("box_inplace_f16", 256, 256, 192, 24, 0.02, storage="f16", pattern="aa", force="profile"),
        # FP32 in place: half the memory at full precision, walls on z, sides that are no powers of two.
        _flow("channel_inplace_f32", 200, 180, 160, 21, 0.02, walls=4, pattern="aa"),
        # The full lattice of Sec. II, FP32.
        _flow("d3q27_f32", 192, 176, 160, 12, 0.02, lattice=27, force="profile"),
        # ... and with 16-bit storage.
        _flow("d3q27_f16", 224, 192, 160, 12, 0.02, storage="f16", lattice=27),
        # The differentiable forced flow: 200 steps forward, checkpoints every 20, gradient by the force.
        dict(name="adjoint_force_64", kind="adjoint", nx=64, ny=64, nz=64, steps=200, every=20, nu=0.02, f0=1e-5),
        # The sweep of 64 uneven channels and ducts, one launch per step.
        dict(name="batch_64_domains", kind="batch", count=64, lo=32, hi=128, steps=40, storage="f32", shapes=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow"] * 7 + ["host", "adjoint", "batch"])
    if kind == "batch":
        return dict(kind="batch", count=_log(rng, 3, 40), lo=rng.choice([24, 32, 48]), hi=rng.choice([96, 113, 128]),
                    steps=rng.randint(8, 48), storage=rng.choice(["f32", "f32", "f16", "bf16"]),
                    shapes=rng.randint(1, 10 ** 6))
    if kind == "adjoint":
        side = _log(rng, 20, 96)
        every = rng.choice([8, 10, 20])
        return dict(kind="adjoint", nx=side, ny=_log(rng, 20, 96), nz=_log(rng, 20, 96),
                    steps=every * rng.randint(2, 6) + rng.choice([0, 0, 3]), every=every, nu=rng.uniform(0.01, 0.05),
                    f0=1e-5)
    while True:
        nx, ny, nz = (_log(rng, 12, 320) for _ in range(3))
        if rng.random() < 0.5:
            nx = max(8, nx // 8 * 8)
        if nx * ny * nz <= 256 ** 3 and min(nx, ny, nz) * 32 >= max(nx, ny, nz):
            break
    n = nx * ny * nz
    lattice = rng.choice([19, 19, 19, 27])
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, nu=rng.uniform(0.01, 0.1), walls=rng.choice([0, 0, 0, 2, 4, 6]),
             storage=rng.choice(["f32", "f32", "f32", "f16", "f16sr", "bf16sr"]), pattern=rng.choice(["ab", "ab", "aa"]),
             lattice=lattice, force=rng.choice(["uniform", "profile", "field"]), f0=rng.choice([1e-6, 1e-5]),
             umax=rng.choice([1e-3, 1e-2, 0.02]), pops=n < 200000 and rng.random() < 0.5)
    c["steps"] = rng.randint(6, 24) if n > 2 ** 20 else rng.randint(16, 90)
    if kind == "host":
        c.update(lattice=19, pattern="ab", storage="f32", pops=False, steps=rng.randint(5, 24))
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _smooth_velocity(c, seed):
    """A few random solenoidal Fourier modes (wavenumbers 1-4 per axis) of root mean square near umax: the initial
    flow of a box, or the disturbance of a channel. (3, nz, ny, nx) float32, on the GPU."""
    rng = random.Random(int(seed) * 31 + 5)
    ax = [torch.arange(m, device="cuda", dtype=torch.float32) * (2.0 * math.pi / m) for m in (c["nx"], c["ny"], c["nz"])]
    u = torch.zeros(3, c["nz"], c["ny"], c["nx"], device="cuda")
    modes = 6
    for _ in range(modes):
        k = [rng.randint(1, 4) * rng.choice([-1, 1]) for _ in range(3)]
        a = [rng.gauss(0, 1) for _ in range(3)]
        kk = sum(v * v for v in k)
        d = sum(p * q for p, q in zip(a, k)) / kk
        a = [p - d * q for p, q in zip(a, k)]
        norm = math.sqrt(sum(p * p for p in a))
        ph = rng.uniform(0, 2 * math.pi)
        # sin(x + y + z + ph) from the phases of the three axes: one (nz, ny, nx) temporary
        arg = (k[2] * ax[2] + ph)[:, None, None] + (k[1] * ax[1])[None, :, None] + (k[0] * ax[0])[None, None, :]
        arg.sin_()
        for m in range(3):
            u[m].add_(arg, alpha=c["umax"] * a[m] / norm / math.sqrt(modes))
    return u


def _phase(seed):
    """Where along x the Taylor-Green vortex sits."""
    return random.Random(int(seed)).uniform(0, 2 * math.pi)


def _force(c, seed):
    """(mode, tensor or None, decay): the force a job sets."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["force"] == "profile":
        F = torch.zeros(3, nz, device="cuda")
        F[0] = c["f0"] * torch.sin(torch.arange(nz, device="cuda", dtype=torch.float64) * (2 * math.pi / nz)).float()
        return F, 0.0
    if c["force"] == "field":
        return torch.randn(3, nz, ny, nx, device="cuda", generator=_gen(seed + 1)) * c["f0"], 0.0
    if c["force"] == "taylor_green":
        # the body force of Sec. III.D, which decays with the vortex it balances, at 2 nu (k1^2 + k2^2)
        k = 2 * math.pi / nx
        x = torch.arange(nx, device="cuda", dtype=torch.float64) * k + _phase(seed)
        y = torch.arange(ny, device="cuda", dtype=torch.float64) * k
        F = torch.zeros(3, nz, ny, nx, device="cuda")
        F[0] = (-0.5 * k * U0_TG ** 2 * torch.sin(2 * x)).float()[None, None, :]
        F[1] = (-0.5 * k * U0_TG ** 2 * torch.sin(2 * y)).float()[None, :, None]
        return F, 2 * c["nu"] * 2 * k * k
    return None, 0.0


def _initial(c, seed):
    """(rho or None, u): the density deviates from 1 by some percent of the flow's size."""
    shape = (c["nz"], c["ny"], c["nx"])
    if c["force"] == "taylor_green":
        k = 2 * math.pi / c["nx"]
        x = torch.arange(c["nx"], device="cuda", dtype=torch.float64) * k + _phase(seed)
        y = torch.arange(c["ny"], device="cuda", dtype=torch.float64) * k
        u = torch.zeros((3,) + shape, device="cuda")
        u[0] = (-U0_TG * torch.cos(x)[None, :] * torch.sin(y)[:, None]).float()[None]
        u[1] = (U0_TG * torch.sin(x)[None, :] * torch.cos(y)[:, None]).float()[None]
        return None, u
    u = _smooth_velocity(c, seed)
    rho = 1.0 + (torch.rand(shape, device="cuda", generator=_gen(seed)) - 0.5) * (0.1 * c["umax"])
    return rho, u


def _uniform(c, seed):
    """Components of a uniform force: mainly along x, a little across."""
    r = random.Random(int(seed) + 99)
    return [float(np.float32(v)) for v in (c["f0"] * r.uniform(0.5, 1.0), 0.1 * c["f0"] * r.uniform(-1, 1), 0.0)]


def _domains(c, seed):
    """Channels and ducts: the sides belong to the case, viscosity and force to the seed."""
    g, r = random.Random(int(c["shapes"])), random.Random(int(seed) + 7)
    out = []
    for _ in range(c["count"]):
        nx, ny, nz = (g.randint(c["lo"], c["hi"]) for _ in range(3))
        out.append(dict(nx=nx, ny=ny, nz=nz, walls=g.choice([4, 6]), nu=r.uniform(0.005, 0.1),
                        fx=float(np.float32(r.uniform(1e-7, 1e-5)))))
    return out


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return dict(c=c, batch=Batch(_domains(c, seed), storage=c["storage"]))
    if c["kind"] == "adjoint":
        lat = Lattice(c["nx"], c["ny"], c["nz"], c["nu"])
        lat.init_equilibrium()
        shape = (3,) + lat.shape
        F = torch.randn(shape, device="cuda", generator=_gen(seed)) * c["f0"]
        target = _smooth_velocity(dict(c, umax=1e-3), seed + 3)
        return dict(c=c, lat=lat, init=lat.export_state(), F=F.requires_grad_(True), target=target)
    lat = Lattice(c["nx"], c["ny"], c["nz"], c["nu"], walls=c["walls"], storage=c["storage"], pattern=c["pattern"],
                  lattice=c["lattice"])
    F, decay = _force(c, seed)
    if F is None:
        lat.set_force_uniform(*_uniform(c, seed))
    elif F.dim() == 2:
        lat.set_force_profile_z(F)
    else:
        lat.set_force_field(F)
    if decay:
        lat.set_force_decay(decay)
    rho, u = _initial(c, seed)
    s = dict(c=c, lat=lat, rho=rho, u=u)
    if c["kind"] == "host":
        for k in ("rho", "u"):
            if s[k] is not None:
                h = torch.empty(s[k].shape, dtype=torch.float32, pin_memory=True)
                h.copy_(s[k])
                s[k] = h
        s["rho_out"] = torch.empty(lat.shape, dtype=torch.float32, pin_memory=True)
        s["u_out"] = torch.empty((3,) + lat.shape, dtype=torch.float32, pin_memory=True)
        s["moments"] = torch.empty(c["steps"] + 1, 4, dtype=torch.float64, pin_memory=True)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c = s["c"]
    if c["kind"] == "batch":
        b = s["batch"]
        b.init_equilibrium()
        b.step(c["steps"])
        fields = [b.macros(d) for d in range(c["count"])]
        return {"rho": torch.cat([f[0].reshape(-1) for f in fields]),
                "u": torch.cat([f[1].reshape(-1) for f in fields])}
    lat = s["lat"]
    if c["kind"] == "adjoint":
        F = s["F"]
        F.grad = None
        u = final_velocity(F, lat, s["init"], c["steps"], c["every"])
        loss = 0.5 * (u - s["target"]).square().sum()
        loss.backward()
        return {"u": u.detach(), "grad": F.grad}
    if c["kind"] == "host":
        lat.run_host(s["rho"], s["u"], c["steps"], s["rho_out"], s["u_out"], s["moments"])
        return {"rho": s["rho_out"], "u": s["u_out"], "moments": s["moments"]}
    lat.init_equilibrium(s["rho"], s["u"])
    lat.step(c["steps"])
    rho, u = lat.macros()
    out = {"rho": rho, "u": u}
    if c["pops"]:
        out["h"] = lat.populations(deviation=True)
    return out


def _nodes(c):
    if c["kind"] == "batch":
        return sum(d["nx"] * d["ny"] * d["nz"] for d in _domains(c, 0))
    return c["nx"] * c["ny"] * c["nz"]


def work(case):
    """The fields a job reads and writes once, its state written once, and the arithmetic of its node updates (about
    300 operations a D3Q19 node, 520 a D3Q27 node, 900 an adjoint node; the adjoint also recomputes its states)."""
    c = dict(case)
    n = _nodes(c)
    if c["kind"] == "adjoint":
        return {"bytes": float(n * 4 * (3 * 4 + 19 * 2)), "flops": float(n * c["steps"] * (300 + 300 + 900))}
    q = c.get("lattice", 19)
    per = 300 if q == 19 else 520
    state = q * (4 if c["storage"] == "f32" else 2)
    read = 0 if c["kind"] == "batch" else 4 * 4
    if c.get("force") in ("field", "taylor_green"):
        read += 12
    write = 16 + (q * 4 if c.get("pops") else 0)
    return {"bytes": float(n * (read + write + state)), "flops": float(n * c["steps"] * per)}


# ---------------------------------------------------------------- the same in 64 bits
class _Exact:
    """The method in 64 bits, as the paper prints it: raw moments by M (Eq. 4), central moments by the binomial
    shift, relaxation with S and the Maxwellian's central moments and the force's (Eqs. 5, A3, A5, A6 / 13, 15, 16),
    back through the inverse, then streaming with halfway bounce-back (Eq. 8). All rates but s2 are 1."""

    def __init__(self, nx, ny, nz, nu, walls, q, device):
        e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        for a, b in ((0, 1), (0, 2), (1, 2)):
            for sb in (1, -1):
                for sa in (1, -1):
                    v = [0, 0, 0]
                    v[a], v[b] = sa, sb
                    e.append(tuple(v))
        if q == 27:
            e += [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]
        self.e, self.q, self.walls, self.shape = e, q, walls, (nz, ny, nx)
        self.exps = [(a, b, d) for a in range(3) for b in range(3) for d in range(3) if q == 27 or 0 in (a, b, d)]
        M = np.array([[float(v[0]) ** m[0] * float(v[1]) ** m[1] * float(v[2]) ** m[2] for v in e] for m in self.exps])
        self.M = torch.from_numpy(M).to(device)
        self.Mi = torch.from_numpy(np.linalg.inv(M)).to(device)
        self.opp = [e.index((-v[0], -v[1], -v[2])) for v in e]
        self.s2 = 1.0 / (3.0 * nu + 0.5)

    def _shift(self, k, axis, v, sign):
        """Central moments from raw ones (sign -1), or back (+1), along one axis."""
        out = dict(k)
        for m in self.exps:
            if m[axis] != 0:
                continue
            at = [tuple(j if a == axis else m[a] for a in range(3)) for j in range(3)]
            if at[1] in k:
                out[at[1]] = k[at[1]] + sign * v * k[m]
            if at[2] in k:
                out[at[2]] = k[at[2]] + 2 * sign * v * k[at[1]] + v * v * k[m]
        return out

    def _eq(self, m):
        return 0.0 if 1 in m else (1.0 / 3.0) ** m.count(2)

    def moments(self, f, F):
        T = self.M @ f
        k = {m: T[i] for i, m in enumerate(self.exps)}
        rho = k[(0, 0, 0)]
        j = [k[m] + 0.5 * F[a] for a, m in enumerate(((1, 0, 0), (0, 1, 0), (0, 0, 1)))]
        return k, rho, j

    def equilibrium(self, rho, u):
        k = {m: rho * self._eq(m) for m in self.exps}
        for a in (2, 1, 0):
            k = self._shift(k, a, u[a], +1)
        return self.Mi @ torch.stack([k[m] for m in self.exps])

    def collide(self, f, F):
        k, rho, j = self.moments(f, F)
        u = [v / rho for v in j]
        for a in range(3):
            k = self._shift(k, a, u[a], -1)
        d = {m: k[m] - rho * self._eq(m) for m in self.exps}
        trace = (1.0 - self.s2) / 3.0 * (d[(2, 0, 0)] + d[(0, 2, 0)] + d[(0, 0, 2)])
        out = {}
        for m in self.exps:
            order, odd = sum(m), [a for a in range(3) if m[a] == 1]
            s = 0.0 if order == 0 else self.s2 if order == 2 else 1.0
            v = (1.0 - s) * d[m] + rho * self._eq(m)
            if m in ((2, 0, 0), (0, 2, 0), (0, 0, 2)):
                v = v - trace
            if len(odd) == 1:  # the force's central moments
                v = v + (1.0 - 0.5 * s) * (1.0 / 3.0) ** m.count(2) * F[odd[0]]
            out[m] = v
        for a in (2, 1, 0):
            out = self._shift(out, a, u[a], +1)
        return self.Mi @ torch.stack([out[m] for m in self.exps])

    def stream(self, f):
        f = f.reshape((self.q,) + self.shape)
        out = []
        for i, v in enumerate(self.e):
            g = torch.roll(f[i], (v[2], v[1], v[0]), (0, 1, 2)) if any(v) else f[i]
            for a in range(3):
                if v[a] and self.walls & (1 << a):
                    at = [slice(None)] * 3
                    at[2 - a] = slice(0, 1) if v[a] > 0 else slice(self.shape[2 - a] - 1, self.shape[2 - a])
                    g = g.clone()
                    g[tuple(at)] = f[self.opp[i]][tuple(at)]
            out.append(g.reshape(-1))
        return torch.stack(out)

    def step(self, f, F):
        return self.stream(self.collide(f, F))

    def start(self, rho, u, F):
        return self.equilibrium(rho, [u[a] - F[a] / (2.0 * rho) for a in range(3)])

    def macros(self, f, F):
        _, rho, j = self.moments(f, F)
        return rho, torch.stack([v / rho for v in j])


EXACT_UPDATES = 2.2e9  # node updates in 64 bits that stay well under 20 seconds on the GPU


def _wide(t, shape):
    return None if t is None else t.double().reshape(shape)


def _exact_flow(c, seed):
    n = _nodes(c)
    if n * c["steps"] > EXACT_UPDATES:
        return None
    x = _Exact(c["nx"], c["ny"], c["nz"], c["nu"], c["walls"], c["lattice"], "cuda")
    F, decay = _force(c, seed)
    if F is None:
        F = _uniform(c, seed)
    elif F.dim() == 2:
        F = F.double()[:, :, None, None].expand(3, c["nz"], c["ny"], c["nx"]).reshape(3, n)
    else:
        F = _wide(F, (3, n))
    at = (lambda t: [v * math.exp(-decay * t) for v in F]) if decay else (lambda t: F)
    rho, u = _initial(c, seed)
    rho = torch.ones(n, dtype=torch.float64, device="cuda") if rho is None else _wide(rho, (n,))
    f = x.start(rho, _wide(u, (3, n)), F)
    sums = []
    for t in range(c["steps"]):
        if c["kind"] == "host":
            _, r, j = x.moments(f, F)
            sums.append(torch.stack([v.sum() for v in [r] + j]))
        f = x.step(f, at(t))
    rho, u = x.macros(f, at(c["steps"]))
    shape = x.shape
    out = {"rho": rho.reshape(shape), "u": u.reshape((3,) + shape)}
    if c["kind"] == "host":
        _, r, j = x.moments(f, F)
        out["moments"] = torch.stack(sums + [torch.stack([v.sum() for v in [r] + j])])
    if c["pops"]:
        w = x.equilibrium(torch.ones(1, dtype=torch.float64, device="cuda"),
                          torch.zeros(3, 1, dtype=torch.float64, device="cuda"))
        out["h"] = (f - w).reshape((x.q,) + shape)
    return out


def _exact_adjoint(c, seed):
    from torch.utils.checkpoint import checkpoint
    n = _nodes(c)
    if n * c["steps"] > 1.5e8:
        return None
    x = _Exact(c["nx"], c["ny"], c["nz"], c["nu"], 0, 19, "cuda")
    F = (torch.randn((3,) + x.shape, device="cuda", generator=_gen(seed)) * c["f0"]).double().reshape(3, n)
    F.requires_grad_(True)
    target = _smooth_velocity(dict(c, umax=1e-3), seed + 3).double().reshape(3, n)
    f = x.equilibrium(torch.ones(n, dtype=torch.float64, device="cuda"),
                      torch.zeros(3, n, dtype=torch.float64, device="cuda"))
    for _ in range(c["steps"]):
        f = checkpoint(x.step, f, F, use_reentrant=False)
    _, u = x.macros(f, F)
    (0.5 * (u - target).square().sum()).backward()
    shape = (3,) + x.shape
    return {"u": u.detach().reshape(shape), "grad": F.grad.reshape(shape)}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "adjoint":
        return _exact_adjoint(c, seed)
    if c["kind"] != "batch":
        return _exact_flow(c, seed)
    if _nodes(c) * c["steps"] > EXACT_UPDATES:
        return None
    rhos, us = [], []
    for d in _domains(c, seed):
        n = d["nx"] * d["ny"] * d["nz"]
        x = _Exact(d["nx"], d["ny"], d["nz"], d["nu"], d["walls"], 19, "cuda")
        F = [d["fx"], 0.0, 0.0]
        f = x.start(torch.ones(n, dtype=torch.float64, device="cuda"),
                    torch.zeros(3, n, dtype=torch.float64, device="cuda"), F)
        for _ in range(c["steps"]):
            f = x.step(f, F)
        rho, u = x.macros(f, F)
        rhos.append(rho)
        us.append(u.reshape(-1))
    return {"rho": torch.cat(rhos), "u": torch.cat(us)}
