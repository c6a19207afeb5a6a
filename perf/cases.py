"""Performance cases: what programs built on this framework ask of it, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed cases, ``draw(rng)`` one more of the
same ranges, ``prepare(case, seed)`` the objects a program holds before the call, ``run(state)`` one
pass, ``work(case)`` the bytes and operations that pass cannot do without, and ``exact(case, seed)``
the same results in 64 bits from plain torch.

All particle sets are square or cubic lattices in the periodic unit box, jittered where "jitter" is
not 0, translated as a whole by a seeded fraction of the spacing, in lattice order or (order =
"shuffled") in a random caller order; the concentration is a Gaussian plume at a seeded place over a
uniform background.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_09488_gb300 import ade, autograd, inputs

C2, C4 = inputs.WENDLAND_C2, inputs.WENDLAND_C4
BACKGROUND = 0.05


# ---- the cases ----------------------------------------------------------------------------------
def _single(name, dim, side, h_dx, steps, **kw):
    c = dict(family="single", dim=dim, side=side, h_dx=h_dx, kernel="c2", ratio=10.0, jitter=0.0, order="lattice",
             steps=steps, call="run", stats=False, tune=False, tau_dt=0.0)
    c.update(kw)
    return {"name": name, **c} if name else c


def _field(name, dim, side, h_dx, steps, **kw):
    c = dict(family="field", dim=dim, side=side, h_dx=h_dx, kernel="c2", ratio=10.0, jitter=0.0, order="lattice",
             steps=steps, call="run", tune=False)
    c.update(kw)
    return {"name": name, **c} if name else c


def _sweep(name, side, h_dx, sets, steps):
    c = dict(family="sweep", dim=2, side=side, h_dx=h_dx, kernel="c2", sets=sets, steps=steps, jitter=0.0,
             order="lattice")
    return {"name": name, **c} if name else c


def _batch(name, plumes, side_lo, side_hi, steps, tune):
    c = dict(family="batch", plumes=plumes, side_lo=side_lo, side_hi=side_hi, steps=steps, tune=tune)
    return {"name": name, **c} if name else c


def _adjoint(name, side, h_dx, steps, every):
    c = dict(family="adjoint", dim=2, side=side, h_dx=h_dx, kernel="c2", ratio=10.0, jitter=0.0, order="lattice",
             steps=steps, every=every)
    return {"name": name, **c} if name else c


def _paper(name, side, ratio, steps):
    c = dict(family="paper", dim=2, side=side, ratio=ratio, jitter=0.45, order="lattice", steps=steps)
    return {"name": name, **c} if name else c


def listed():
    return [
        # the 64 x 64 plume, one step at a time with its mass and extrema read back: the smallest
        # call, as made by a program that watches every step
        _single("plume-64-step-stats", 2, 64, 1.3, 1, stats=True),
        # the convergence ladder's 256^2 rung (28 neighbours) advanced by 50 steps in one call, in
        # the configuration the library chooses by itself
        _single("ladder-256-run50", 2, 256, 1.5025, 50, ratio=100.0),
        # the ladder's top rung (1024^2, 120 neighbours), tuned once, ten steps between two outputs
        _single("ladder-1024-run10", 2, 1024, 3.0425, 10, tune=True),
        # the benchmark's default: the 128^3 cube (250 neighbours), tuned, one step per call
        _single("cube-128-step", 3, 128, 2.0, 1, tune=True),
        # dC/dt of an irregular 3D set of odd size in arbitrary caller order, Wendland C4: a
        # one-off evaluation by a program with its own integrator, nothing tuned
        _single("irregular-57-rate", 3, 57, 3.1, 0, kernel="c4", jitter=0.4, order="shuffled", call="rate"),
        # Cattaneo's form on an irregular 2D set of odd size, eight launched (not replayed) steps
        _single("cattaneo-301-step8", 2, 301, 1.9, 8, jitter=0.35, order="shuffled", call="step", tau_dt=2.0),
        # the paper's own test model at 10^6 irregular particles and about 31,300 neighbours, one
        # step: the largest
        _paper("paper-1m-step", 1000, 0.1, 1),
        # heterogeneous flow (a velocity per particle) on the 1024^2 rung, tuned
        _field("field-1024-run2", 2, 1024, 3.0425, 2, tune=True),
        # heterogeneous flow in 3D on an irregular set, untuned
        _field("field-45-cube-step", 3, 45, 1.8, 1, jitter=0.3, call="step"),
        # eight dispersivity sets on one 512^2 plume (60 neighbours), as in the ratio study
        _sweep("sweep-512x8-run4", 512, 2.1225, 8, 4),
        # the 64 uneven plumes of the batched workload, tuned once
        _batch("batched-64-run4", 64, 32, 512, 4, True),
        # one gradient of a dispersivity inversion: forward 40 steps and backward, through autograd
        _adjoint("adjoint-512-grad", 512, 1.3, 40, 20),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    ratio = round(math.exp(rng.uniform(0.0, math.log(100.0))), 3)
    kind = rng.choice(["single2", "single2", "single3", "rate", "cattaneo", "paper", "field2", "field3", "sweep",
                       "batch", "adjoint"])
    jitter = rng.choice([0.0, 0.2, 0.45])
    order = rng.choice(["lattice", "shuffled"])
    kernel = rng.choice(["c2", "c2", "c4"])
    wide = 2.0 if kernel == "c4" else 1.0          # C4's support is h, C2's 2h
    h2 = round(rng.uniform(1.3, 3.1) * wide, 3)
    h3 = round(rng.uniform(1.2, 2.1) * wide, 3)
    tune = rng.random() < 0.5
    if kind == "single2":
        side = _logint(rng, 64, 1100)
        steps = _logint(rng, 1, 60)
        return _single(None, 2, side, h2, steps, kernel=kernel, ratio=ratio, jitter=jitter, order=order, tune=tune,
                       call=rng.choice(["run", "run", "step"]), stats=jitter == 0.0 and rng.random() < 0.3)
    if kind == "single3":
        return _single(None, 3, _logint(rng, 20, 128), h3, _logint(rng, 1, 8), kernel=kernel, ratio=ratio,
                       jitter=jitter, order=order, tune=tune)
    if kind == "rate":
        dim = rng.choice([2, 3])
        side = _logint(rng, 64, 1100) if dim == 2 else _logint(rng, 20, 110)
        return _single(None, dim, side, h2 if dim == 2 else h3, 0, kernel=kernel, ratio=ratio, jitter=jitter,
                       order=order, call="rate")
    if kind == "cattaneo":
        return _single(None, 2, _logint(rng, 64, 700), h2, _logint(rng, 1, 16), kernel=kernel, ratio=ratio,
                       jitter=jitter, order=order, call=rng.choice(["run", "step"]),
                       tau_dt=round(rng.uniform(1.0, 5.0), 2))
    if kind == "paper":
        return _paper(None, _logint(rng, 100, 700), rng.choice([0.1, 0.01, 0.001]), rng.choice([1, 2]))
    if kind == "field2":
        return _field(None, 2, _logint(rng, 64, 1024), h2, rng.choice([1, 2, 4]), kernel=kernel, ratio=ratio,
                      jitter=jitter, order=order, tune=tune)
    if kind == "field3":
        return _field(None, 3, _logint(rng, 20, 64), h3, rng.choice([1, 2]), kernel=kernel, ratio=ratio,
                      jitter=jitter, order=order, call=rng.choice(["run", "step"]))
    if kind == "sweep":
        return _sweep(None, _logint(rng, 64, 700), round(rng.uniform(1.3, 3.0), 3), rng.randint(1, 20),
                      rng.choice([1, 2, 5, 10]))
    if kind == "batch":
        lo = _logint(rng, 20, 64)
        return _batch(None, rng.randint(2, 64), lo, _logint(rng, 100, 400), rng.choice([1, 3, 8]), tune)
    steps = rng.randint(8, 60)
    return _adjoint(None, _logint(rng, 64, 512), round(rng.uniform(1.3, 2.2), 3), steps, rng.randint(4, steps))


# ---- inputs -------------------------------------------------------------------------------------
def _rng(seed, k=0):
    return np.random.Generator(np.random.PCG64([int(seed) & 0x7FFFFFFF, k]))


def _kernel(case):
    return C4 if case.get("kernel") == "c4" else C2


def _plume(case):
    return inputs.Plume(dim=case["dim"], side=case["side"], h_over_dx=case["h_dx"], kernel=_kernel(case),
                        alpha_T=1e-3, alpha_L=1e-3 * case.get("ratio", 10.0), jitter=case["jitter"])


def _paper_plume(case, seed):
    return inputs.paper_plume(case["side"], case["ratio"], jitter=case["jitter"], seed=int(seed) & 0x7FFFFFFF)


def _particles(plume, case, seed):
    """(xq uint32 [dim][n], C float32 [n], order): order[a] = lattice site of caller particle a."""
    rng = _rng(seed)
    n, dim = plume.n, plume.dim
    x = inputs.lattice_positions(dim, plume.side)
    x += rng.uniform(0.0, 1.0, size=dim) * plume.dx
    if case["jitter"] > 0.0:
        x += rng.uniform(-case["jitter"], case["jitter"], size=x.shape) * plume.dx
    xq = inputs.to_fixed(x, plume.boxv)
    x0 = rng.uniform(0.2, 0.8, size=dim)
    C = BACKGROUND + inputs.gaussian_plume(inputs.from_fixed(xq, plume.boxv), plume.boxv, x0, plume.w, plume.C0)
    order = rng.permutation(n) if case["order"] == "shuffled" else None
    if order is not None:
        xq, C = np.ascontiguousarray(xq[:, order]), C[order]
    return xq, C.astype(np.float32), order


def _lambda(plume, speed):
    return max(plume.alpha_L, plume.alpha_T) * speed + plume.D_m


def _dt(plume, speed):
    return plume.dt if plume.dt > 0.0 else 0.1 * plume.h * plume.h / _lambda(plume, speed)


def _tau(case, plume):
    return case.get("tau_dt", 0.0) * _dt(plume, plume.speed)


VMAX = 0.2


def _velocities(plume, xq, seed):
    """A smooth periodic field, |v| <= VMAX."""
    x = inputs.from_fixed(xq, plume.boxv)
    v = inputs.velocity_field(x, plume.boxv, seed=int(seed) & 0x7FFFFFFF).astype(np.float64)
    top = float(np.sqrt((v * v).sum(axis=0)).max())
    return np.ascontiguousarray((v * min(1.0, 0.99 * VMAX / top)).astype(np.float32))


def _thetas(sets):
    """sets x (alpha_L, alpha_T, D_m), alpha_L / alpha_T from 1 to 100."""
    r = np.geomspace(1.0, 100.0, sets) if sets > 1 else np.array([10.0])
    return np.stack([1e-3 * r, np.full(sets, 1e-3), np.full(sets, 1e-6)], axis=1)


def _batch_plumes(case, seed):
    return inputs.batched_2d(case["plumes"], seed=20210821 + case["plumes"], side_lo=case["side_lo"],
                             side_hi=case["side_hi"])


_BATCH_CASE = dict(jitter=0.0, order="lattice")


def prepare(case, seed):
    f = case["family"]
    if f == "batch":
        plumes = _batch_plumes(case, seed)
        parts = [_particles(p, _BATCH_CASE, seed + 1000 * i)[:2] for i, p in enumerate(plumes)]
        b = ade.Batch([ade.params_for(p) for p in plumes], [x for x, _ in parts], [c for _, c in parts])
        if case["tune"]:
            b.autotune()
        return {"family": f, "obj": b, "steps": case["steps"]}
    plume = _paper_plume(case, seed) if f == "paper" else _plume(case)
    xq, C, _ = _particles(plume, case, seed)
    if f == "sweep":
        rng = _rng(seed, 1)
        sets = case["sets"]
        Cs = C[None, :] * (1.0 + 0.2 * rng.uniform(size=(sets, 1))).astype(np.float32)
        return {"family": f, "obj": ade.Sweep(ade.params_for(plume), xq, Cs, _thetas(sets)), "steps": case["steps"]}
    if f == "adjoint":
        sim = ade.Simulation(ade.params_for(plume), xq, C)
        return {"family": f, "obj": sim, "steps": case["steps"], "every": case["every"],
                "C0": torch.from_numpy(C).cuda(), "target": torch.from_numpy(_target(plume, xq, seed)).cuda(),
                "theta": torch.tensor([plume.alpha_L, plume.alpha_T, plume.D_m], dtype=torch.float64)}
    if f == "field":
        sim = ade.Simulation(ade.params_for(plume, vmax=VMAX), xq, C)
        sim.set_velocity_field(_velocities(plume, xq, seed))
    else:
        tau = _tau(case, plume) if f == "single" else 0.0
        sim = ade.Simulation(ade.params_for(plume, tau=tau), xq, C)
        if tau > 0.0:
            sim.set_flux()
    if case.get("tune"):
        sim.autotune()
    return {"family": f, "obj": sim, "steps": case["steps"], "call": case.get("call", "run"),
            "stats": case.get("stats", False), "flux": f == "single" and case["tau_dt"] > 0.0}


def _target(plume, xq, seed):
    """The observed field of the inversion: a wider plume somewhere else."""
    x0 = _rng(seed, 2).uniform(0.3, 0.7, size=plume.dim)
    C = inputs.gaussian_plume(inputs.from_fixed(xq, plume.boxv), plume.boxv, x0, 2.0 * plume.w, 0.8)
    return (BACKGROUND + C).astype(np.float32)


# ---- one pass -----------------------------------------------------------------------------------
def run(state):
    f, obj, steps = state["family"], state["obj"], state["steps"]
    if f in ("batch", "sweep"):
        obj.run(steps)
        return {"C": obj.C, "xq": obj.xq}
    if f == "adjoint":
        C0 = state["C0"].clone().requires_grad_()
        theta = state["theta"].clone().requires_grad_()
        J = autograd.misfit(obj, C0, theta, state["target"], steps, state["every"])
        J.backward()
        return {"J": J.item(), "dC0": C0.grad, "dtheta": theta.grad.tolist()}
    if state["call"] == "rate":
        return {"rate": obj.rate()}
    out = {}
    if state["call"] == "step":
        obj.step(steps)
    else:
        st = obj.run(steps, stats=state["stats"])
        if state["stats"]:
            out["stats"] = [st.mass, st.c_min, st.c_max]
    out["C"], out["xq"] = obj.C, obj.xq
    if state["flux"]:
        out["flux"] = obj.flux()
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------
def _neighbours(plume, jitter):
    r = plume.support / plume.dx
    if jitter > 0.0 or r > 12.0:
        return math.pi * r * r if plume.dim == 2 else 4.0 / 3.0 * math.pi * r ** 3
    m = int(math.ceil(r))
    g = np.arange(-m, m + 1, dtype=np.float64) ** 2
    r2 = g[:, None] + g[None, :] if plume.dim == 2 else g[:, None, None] + g[None, :, None] + g[None, None, :]
    return float(np.count_nonzero(r2 < r * r) - 1)


def _pair_flops(dim, kernel, field=False):
    # separation, r^2, 1/r, 1 - q, the kernel shape, Eq. 5's factor, the weighted difference
    base = 21 if dim == 2 else 26
    if field:       # harmonic means of the tensor's components, both terms of Eq. 4
        base = 50 if dim == 2 else 85
    return base + (4 if kernel == C4 else 0)


def work(case):
    f = case["family"]
    if f == "batch":
        by = fl = 0.0
        for p in _batch_plumes(case, 0):
            by += p.n * (8.0 * p.dim + 8.0)
            fl += 2.0 * case["steps"] * p.n * _neighbours(p, 0.0) * _pair_flops(p.dim, p.kernel)
        return {"bytes": by, "flops": fl}
    plume = _paper_plume(case, 0) if f == "paper" else _plume(case)
    n, dim = plume.n, plume.dim
    pairs = n * _neighbours(plume, case["jitter"])
    if f == "sweep":
        return {"bytes": n * (8.0 * dim + 8.0 * case["sets"]),
                "flops": 2.0 * case["steps"] * pairs * (16.0 + 6.0 * case["sets"])}
    if f == "adjoint":
        # per step: two applications forward, two for the adjoint, and three directional ones of
        # the state and of its rate
        return {"bytes": n * (4.0 * dim + 12.0), "flops": case["steps"] * pairs * (4.0 * 3.0 + 2.0 * 9.0)}
    per = _pair_flops(dim, plume.kernel, f == "field")
    if case.get("call") == "rate":
        return {"bytes": n * (4.0 * dim + 8.0), "flops": pairs * per}
    extra = 8.0 if f == "single" and case["tau_dt"] > 0.0 else (4.0 * dim if f == "field" else 0.0)
    return {"bytes": n * (8.0 * dim + 8.0 + extra), "flops": 2.0 * case["steps"] * pairs * per}


# ---- the same in 64 bits --------------------------------------------------------------------------
# Neighbours on a (jittered) lattice are found by lattice offsets: every particle within the support
# is at most support / dx + 2 jitter sites away along each axis.
TWO32 = 2.0 ** 32


class _Grid:
    """Fixed-point words on the lattice, x fastest: tensors of shape [side] * dim."""

    def __init__(self, plume, xq, order, slack=0.0):
        self.plume, self.dim = plume, plume.dim
        self.shape = [plume.side] * plume.dim
        self.order = None if order is None else torch.from_numpy(order).cuda()
        self.x = [self.site(torch.from_numpy(a.astype(np.int64)).cuda()) for a in xq]
        reach = plume.support / plume.dx + slack
        m = int(math.ceil(reach))
        if 2 * m + 1 > plume.side:
            raise ValueError("the box is too small for the offsets")
        self.offsets = []
        for flat in np.ndindex(*([2 * m + 1] * plume.dim)):
            o = [k - m for k in flat]
            if any(o) and sum(max(abs(k) - slack, 0.0) ** 2 for k in o) < (plume.support / plume.dx) ** 2 * (1 + 1e-9):
                self.offsets.append(o)

    def site(self, a):
        """Caller order -> lattice."""
        if self.order is not None:
            b = torch.empty_like(a)
            b[self.order] = a
            a = b
        return a.reshape(self.shape)

    def caller(self, a):
        a = a.reshape(-1)
        return a if self.order is None else a[self.order]

    def at(self, a, o):
        """a at the neighbour `o` sites away (o along x first)."""
        return torch.roll(a, [-k for k in o], [self.dim - 1 - i for i in range(self.dim)])

    def separation(self, x, o):
        out = []
        for a in x:
            d = a - self.at(a, o)
            d = torch.remainder(d + (1 << 31), 1 << 32) - (1 << 31)
            out.append(d.to(torch.float64) * (self.plume.box / TWO32))
        return out

    def radial(self, d):
        """(f, r2): f = W'(r) / r, zero outside the support and at r = 0."""
        p = self.plume
        H, dim = p.support, p.dim
        r2 = sum(c * c for c in d)
        q = torch.sqrt(r2) / H
        om = torch.clamp(1.0 - q, min=0.0)
        if p.kernel == C2:
            B = 7.0 / (math.pi * H * H) if dim == 2 else 21.0 / (2.0 * math.pi * H ** 3)
            f = -20.0 * B / (H * H) * om ** 3
        else:
            B = 9.0 / (math.pi * H * H) if dim == 2 else 495.0 / (32.0 * math.pi * H ** 3)
            f = -(56.0 / 3.0) * B / (H * H) * om ** 5 * (1.0 + 5.0 * q)
        return torch.where(r2 > 0.0, f, torch.zeros_like(f)), torch.clamp(r2, min=1e-300)


def _tensor(v, aL, aT, Dm):
    s = float(np.linalg.norm(v))
    D = (aT * s + Dm) * np.eye(len(v))
    return D + (aL - aT) * np.outer(v, v) / s


def _weight(g, o, Ds):
    """Weights of Eq. 4-5 for the pair (site, site + o), one per uniform tensor of Ds."""
    p = g.plume
    gamma = p.dim + 2.0
    d = g.separation(g.x, o)
    f, r2 = g.radial(d)
    out = []
    for D in Ds:
        K = 2.0 * D
        Q = sum(K[i, j] * d[i] * d[j] for i in range(p.dim) for j in range(p.dim))
        out.append(0.5 * p.mass / p.rho * (gamma * Q / r2 - float(np.trace(K))) * f)
    return out


class _Operator:
    """C -> dC/dt for uniform tensors Ds (the geometry does not change in a uniform flow)."""

    def __init__(self, g, Ds):
        self.g, self.Ds = g, Ds
        self.kept = None
        if len(g.offsets) * g.plume.n * 8 * len(Ds) < 24e9:
            self.kept = [_weight(g, o, Ds) for o in g.offsets]

    def __call__(self, Cs, which=None):
        """Cs: one field per tensor; or one field with `which`, the tensor."""
        g = self.g
        out = [torch.zeros_like(c) for c in Cs]
        for k, o in enumerate(g.offsets):
            w = self.kept[k] if self.kept is not None else _weight(g, o, self.Ds)
            for i, c in enumerate(Cs):
                out[i] += w[i if which is None else which] * (c - g.at(c, o))
        return out


def _advance(op, Cs, dt, steps):
    for _ in range(steps):
        half = [c + 0.5 * dt * r for c, r in zip(Cs, op(Cs))]
        Cs = [c + dt * r for c, r in zip(Cs, op(half))]
    return Cs


def _too_much(plume, jitter, evaluations, per=1.0):
    return plume.n * _neighbours(plume, jitter) * evaluations * per > 1.5e11


def _field_rate(g, x, C, v, D):
    """Eq. 4 with a velocity and a tensor per particle: both sums."""
    p = g.plume
    dim, gamma = p.dim, p.dim + 2.0
    out = torch.zeros_like(C)
    for o in g.offsets:
        d = g.separation(x, o)
        f, r2 = g.radial(d)
        Q = tr = 0.0
        for (i, j), a in D.items():
            b = g.at(a, o)
            s = a + b
            K = torch.where(s != 0.0, 4.0 * a * b / torch.where(s != 0.0, s, torch.ones_like(s)), torch.zeros_like(s))
            Q = Q + (1.0 if i == j else 2.0) * K * d[i] * d[j]
            if i == j:
                tr = tr + K
        out += 0.5 * p.mass / p.rho * (gamma * Q / r2 - tr) * f * (C - g.at(C, o))
        conv = sum((v[i] - g.at(v[i], o)) * d[i] for i in range(dim))
        out += p.mass / p.rho * C * conv * f
    return out


def exact(case, seed):
    f = case["family"]
    if f == "batch":
        Cs, evaluations = [], 2 * case["steps"]
        plumes = _batch_plumes(case, seed)
        if sum(p.n * _neighbours(p, 0.0) for p in plumes) * evaluations > 1.5e11:
            return None
        for i, p in enumerate(plumes):
            xq, C, order = _particles(p, _BATCH_CASE, seed + 1000 * i)
            g = _Grid(p, xq, order)
            op = _Operator(g, [_tensor(p.velocity, p.alpha_L, p.alpha_T, p.D_m)])
            c = g.site(torch.from_numpy(C).cuda().double())
            Cs.append(g.caller(_advance(op, [c], _dt(p, p.speed), case["steps"])[0]))
        return {"C": torch.cat(Cs), "xq": None}
    plume = _paper_plume(case, seed) if f == "paper" else _plume(case)
    jitter = case["jitter"]
    if _too_much(plume, jitter, 2 * max(1, case["steps"]), 3.0 if f == "field" else 1.0):
        return None
    xq, C, order = _particles(plume, case, seed)
    # in a field particles move apart by a fraction of the spacing within the few steps of a case
    g = _Grid(plume, xq, order, slack=2.0 * jitter + (1.0 if f == "field" else 0.0))
    c = g.site(torch.from_numpy(C).cuda().double())
    steps = case["steps"]
    uniform = _tensor(plume.velocity, plume.alpha_L, plume.alpha_T, plume.D_m)
    if f == "field":
        dt = _dt(plume, VMAX)
        v32 = _velocities(plume, xq, seed)
        v = [g.site(torch.from_numpy(a).cuda().double()) for a in v32]
        s = torch.sqrt(sum(a * a for a in v))
        D = {}
        for i in range(plume.dim):
            for j in range(i, plume.dim):
                D[i, j] = (plume.alpha_L - plume.alpha_T) * v[i] * v[j] / s
                if i == j:
                    D[i, j] = D[i, j] + plume.alpha_T * s + plume.D_m
        x = g.x
        for _ in range(steps):
            r = _field_rate(g, x, c, v, D)
            xh = [a + torch.round(b * (0.5 * dt) * TWO32).long() for a, b in zip(x, v)]
            r = _field_rate(g, xh, c + 0.5 * dt * r, v, D)
            c = c + dt * r
            x = [a + torch.round(b * dt * TWO32).long() for a, b in zip(x, v)]
        return {"C": g.caller(c), "xq": None}
    if f == "sweep":
        th = _thetas(case["sets"])
        Ds = [_tensor(plume.velocity, *t) for t in th]
        dt = min(0.1 * plume.h ** 2 / (max(t[0], t[1]) * plume.speed + t[2]) for t in th)
        scale = (1.0 + 0.2 * _rng(seed, 1).uniform(size=(case["sets"], 1))).astype(np.float32)
        Cs = [g.site(torch.from_numpy(C * k).cuda().double()) for k in scale]
        out = []
        for k in range(0, len(Ds), 4):
            out += _advance(_Operator(g, Ds[k:k + 4]), Cs[k:k + 4], dt, steps)
        return {"C": torch.stack([g.caller(a) for a in out]), "xq": None}
    if f == "adjoint":
        return _exact_adjoint(case, seed, plume, g, c, xq)
    op = _Operator(g, [uniform])
    if case.get("call") == "rate":
        return {"rate": g.caller(op([c])[0])}
    dt = _dt(plume, plume.speed)
    out = {}
    tau = _tau(case, plume) if f == "single" else 0.0
    if tau > 0.0:
        dt = min(dt, tau)
        q = op([c])[0]
        for _ in range(steps):
            ch, qh = c + 0.5 * dt * q, q + 0.5 * dt * (op([c])[0] - q) / tau
            c, q = c + dt * qh, q + dt * (op([ch])[0] - qh) / tau
        out["flux"] = g.caller(q)
    else:
        c = _advance(op, [c], dt, steps)[0]
    if case.get("stats"):
        out["stats"] = [float(c.sum()) * plume.mass, float(c.min()), float(c.max())]
    out["C"], out["xq"] = g.caller(c), None
    return out


def _exact_adjoint(case, seed, plume, g, c, xq):
    v = plume.velocity
    s = float(np.linalg.norm(v))
    vv = np.outer(v, v) / s
    basis = [vv, s * np.eye(plume.dim) - vv, np.eye(plume.dim)]
    theta = [plume.alpha_L, plume.alpha_T, plume.D_m]
    op = _Operator(g, basis + [sum(t * b for t, b in zip(theta, basis))])
    dt, steps = _dt(plume, plume.speed), case["steps"]

    def L(u):
        return op([u], which=3)[0]

    states = [c]
    for _ in range(steps):
        u = states[-1]
        states.append(u + dt * L(u + 0.5 * dt * L(u)))
    p = states[-1] - g.site(torch.from_numpy(_target(plume, xq, seed)).cuda().double())
    J = 0.5 * float((p * p).sum())
    grad = [0.0, 0.0, 0.0]
    for u in reversed(states[:-1]):
        a, b = L(u), L(p)
        for k in range(3):
            r = op([u], which=k)[0]
            la = op([a], which=k)[0]
            grad[k] += dt * float((p * r).sum()) + 0.5 * dt * dt * float((p * la).sum() + (b * r).sum())
        p = p + dt * L(p + 0.5 * dt * b)
    return {"J": J, "dC0": g.caller(p), "dtheta": grad}
