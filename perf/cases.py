"""Timing cases: what programs have this library do, over the sizes, models, precisions and
options that they use, each through the public Python objects.

A case is a dict of plain values.  `kind` says which call is made:

* "run":      one System advanced `steps` integrator steps from a given state, the new state
              read back, all in device memory; with `energy` the kinetic and potential energy
              as well (an accuracy-monitored run samples them between blocks of steps).
* "grad":     System.grad, the gradient of the final kinetic energy with respect to the
              starting state and the softening (forward steps and the reverse sweep).
* "ensemble": an Ensemble of independent Ring and 2D systems of uneven sizes advanced
              together, all states read back.

`exact` recomputes every output in FP64 with plain torch from the definitions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1212_0262_gb300 import Ensemble, System

DIM = {"hmf": 1, "ring": 1, "grav2d": 2, "grav3d": 3, "sheet1d": 1}

# FP operations of one unordered pair's force term, added to both particles (HMF: of one
# particle's stage; sheets: of one comparison of a sort), and of its potential term
FORCE_OPS = {"hmf": 40, "ring": 16, "grav2d": 14, "grav3d": 20, "sheet1d": 4}
POTENTIAL_OPS = {"hmf": 20, "ring": 8, "grav2d": 7, "grav3d": 10, "sheet1d": 4}
GRAD_OPS = {"ring": 34, "grav2d": 40}  # force, Jacobian-vector product and d/d eps of a pair


def listed():
    return [
        # A small mean-field run (Lyapunov and accuracy studies use about 10^4 particles): 150
        # stages of a few microseconds each, so what counts is the latency of a stage.
        dict(name="hmf_small_mixed", kind="run", model="hmf", N=10_007, precision="mixed", steps=50, dt=0.1, eps=0.0,
             energy=True),
        # The benchmark's mean-field system: one streaming pass over 800 MB per stage.
        dict(name="hmf_large_mixed", kind="run", model="hmf", N=50_000_000, precision="mixed", steps=10, dt=0.1,
             eps=0.0, energy=False),
        # The same model in the library's default precision.
        dict(name="hmf_fp64", kind="run", model="hmf", N=10_000_000, precision="fp64", steps=10, dt=0.1, eps=0.0,
             energy=False),
        # The smallest Ring size in use (the smallest member of the ensembles, the Lyapunov runs).
        dict(name="ring_small_mixed", kind="run", model="ring", N=4_096, precision="mixed", steps=9, dt=0.01,
             eps=0.01, energy=False),
        # The benchmark's Ring system.
        dict(name="ring_large_mixed", kind="run", model="ring", N=131_072, precision="mixed", steps=2, dt=0.05,
             eps=0.01, energy=False),
        # The accuracy experiment's Ring system in the default precision, energies monitored.
        dict(name="ring_fp64_energy", kind="run", model="ring", N=16_384, precision="fp64", steps=1, dt=0.005,
             eps=1e-3, energy=True),
        # The benchmark's 2D system.
        dict(name="grav2d_large_mixed", kind="run", model="grav2d", N=262_144, precision="mixed", steps=1, dt=0.01,
             eps=1e-4, energy=False),
        # The accuracy experiment's 2D system, one particle more than whole tiles, default precision.
        dict(name="grav2d_fp64_energy", kind="run", model="grav2d", N=16_385, precision="fp64", steps=1, dt=0.005,
             eps=1e-3, energy=True),
        # A 3D system of an odd size in mixed precision.
        dict(name="grav3d_mixed", kind="run", model="grav3d", N=65_537, precision="mixed", steps=1, dt=0.01,
             eps=1e-3, energy=False),
        # Unsoftened sheets: every force an exact sign count.
        dict(name="sheets_mixed", kind="run", model="sheet1d", N=100_003, precision="mixed", steps=2, dt=0.01,
             eps=0.0, energy=False),
        # A gradient through the integrator in the default precision (autograd's size range).
        dict(name="grav2d_grad_fp64", kind="grad", model="grav2d", N=8_192, precision="fp64", steps=4, dt=0.01,
             eps=1e-3, checkpoint=2),
        # An ensemble with the benchmark's spread of sizes, log-uniform in [4096, 65536].
        dict(name="ensemble_mixed", kind="ensemble", nsys=24, precision="mixed", steps=2),
    ]


def _size(rng, lo, hi):
    """Log-uniform size in [lo, hi]; odd half of the time."""
    n = int(round(lo * (hi / lo) ** rng.random()))
    return n | 1 if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["hmf", "hmf", "pairs", "pairs", "pairs", "fp64", "fp64", "fp64", "sheet1d", "grad", "ensemble"])
    if kind == "hmf":
        prec = rng.choice(["mixed", "fp64"])
        return dict(kind="run", model="hmf", N=_size(rng, 2_000, 20_000_000 if prec == "mixed" else 8_000_000),
                    precision=prec, steps=rng.choice([1, 5, 10, 20]), dt=rng.choice([0.05, 0.1]), eps=0.0,
                    energy=rng.random() < 0.5)
    if kind == "pairs":
        model = rng.choice(["ring", "grav2d", "grav3d"])
        return dict(kind="run", model=model, N=_size(rng, 1_500, 65_536), precision="mixed",
                    steps=rng.choice([1, 2, 3]), dt=rng.choice([0.005, 0.01]), eps=rng.choice([1e-3, 0.01]),
                    energy=rng.random() < 0.3)
    if kind == "fp64":
        model = rng.choice(["ring", "grav2d", "grav3d"])
        return dict(kind="run", model=model, N=_size(rng, 1_000, 20_000), precision="fp64",
                    steps=rng.choice([1, 2]), dt=rng.choice([0.005, 0.01]), eps=rng.choice([1e-4, 1e-3, 0.01]),
                    energy=rng.random() < 0.5)
    if kind == "sheet1d":
        return dict(kind="run", model="sheet1d", N=_size(rng, 2_000, 262_144), precision=rng.choice(["mixed", "fp64"]),
                    steps=rng.choice([1, 2]), dt=0.01, eps=0.0, energy=False)
    if kind == "grad":
        return dict(kind="grad", model=rng.choice(["ring", "grav2d"]), N=_size(rng, 1_000, 8_192), precision="fp64",
                    steps=rng.choice([2, 3, 4]), dt=0.01, eps=rng.choice([1e-3, 0.01]), checkpoint=rng.choice([1, 2, 4]))
    return dict(kind="ensemble", nsys=rng.randint(4, 24), precision="mixed", steps=rng.choice([1, 2]))


# ---------------------------------------------------------------- inputs ---

def _gen(seed, device):
    return torch.Generator(device=device).manual_seed(int(seed) * 7919 + 17)


def _state(model, N, g):
    """(q, p), each dim * N doubles in the library's layout: the models' default recipes."""
    dev = g.device
    u = lambda: torch.rand(N, generator=g, device=dev, dtype=torch.float64)  # noqa: E731
    n = lambda: torch.randn(N, generator=g, device=dev, dtype=torch.float64)  # noqa: E731
    if model == "hmf":
        return 2.0 * u() - 1.0, 2.4 * u() - 1.2
    if model == "ring":
        return (2.0 * u() - 1.0) * math.pi, 0.5 * n()
    if model == "sheet1d":
        return 2.0 * u() - 1.0, u() - 0.5
    if model == "grav2d":
        r, phi = u().sqrt(), 2.0 * math.pi * u()
        return torch.cat([r * phi.cos(), r * phi.sin()]), 0.3 * torch.cat([n(), n()])
    r, c, phi = u() ** (1.0 / 3.0), 2.0 * u() - 1.0, 2.0 * math.pi * u()
    s = (1.0 - c * c).sqrt()
    return torch.cat([r * s * phi.cos(), r * s * phi.sin(), r * c]), 0.3 * torch.cat([n(), n(), n()])


def _members(case):
    """(model, N, eps, dt) of every system of an ensemble; the sizes spread over [4096, 65536]."""
    out = []
    for s in range(case["nsys"]):
        u = (s * 0.6180339887498949 + 0.3) % 1.0
        ring = s < case["nsys"] // 2
        out.append(("ring" if ring else "grav2d", int(4096 * 16**u), 0.01 if ring else 1e-4, 0.05 if ring else 0.01))
    return out


def _member_state(model, N, seed, s):
    return _state(model, N, _gen(1000 * seed + s, "cpu"))


# ------------------------------------------------------- the measured call --

def prepare(case, seed):
    if case["kind"] == "ensemble":
        m = _members(case)
        ens = Ensemble([x[0] for x in m], [x[1] for x in m], [x[2] for x in m], [x[3] for x in m],
                       [seed + s for s in range(len(m))], precision=case["precision"])
        for s, (model, N, _, _) in enumerate(m):
            q, p = _member_state(model, N, seed, s)
            ens.set_state(s, q.numpy(), p.numpy())
        return dict(case=case, ens=ens)
    model, N = case["model"], case["N"]
    q, p = _state(model, N, _gen(seed, "cuda"))
    torch.cuda.synchronize()  # the system works on a stream of its own
    system = System(model, N, case["eps"], case["dt"], seed, precision=case["precision"])
    if case["kind"] == "grad":
        system.set_state_device(q.data_ptr(), p.data_ptr())
        system.synchronize()
        return dict(case=case, system=system)
    return dict(case=case, system=system, q=q, p=p, q_out=torch.empty_like(q), p_out=torch.empty_like(p))


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        return {str(s): ens.get_state(s) for s in range(case["nsys"])}
    system = state["system"]
    if case["kind"] == "grad":
        value, gq, gp, geps = system.grad(case["steps"], checkpoint_every=case["checkpoint"])
        return {"value": value, "grad_q": gq, "grad_p": gp, "grad_eps": geps}
    system.set_state_device(state["q"].data_ptr(), state["p"].data_ptr())
    system.step(case["steps"])
    system.get_state_device(state["q_out"].data_ptr(), state["p_out"].data_ptr())
    out = {"q": state["q_out"], "p": state["p_out"]}
    if case["energy"]:
        out["K"], out["V"] = system.energy()
    return out


# -------------------------------------------------------------------- work --

def _evaluations(steps):
    return 3 * steps + 1  # three per step and the closing kick's


def work(case):
    if case["kind"] == "ensemble":
        flops = sum(_evaluations(case["steps"]) * FORCE_OPS[m] * N * (N - 1) / 2 for m, N, _, _ in _members(case))
        size = sum(DIM[m] * N for m, N, _, _ in _members(case))
        return dict(bytes=32.0 * size, flops=flops)
    model, N, steps = case["model"], case["N"], case["steps"]
    size = DIM[model] * N
    if model == "hmf":
        # the magnetization orders the stages: every one of them reads and writes the state
        return dict(bytes=32.0 * N * _evaluations(steps), flops=FORCE_OPS[model] * N * _evaluations(steps))
    if model == "sheet1d":
        return dict(bytes=32.0 * N, flops=_evaluations(steps) * FORCE_OPS[model] * N * math.log2(max(N, 2)))
    pairs = N * (N - 1) / 2
    if case["kind"] == "grad":
        return dict(bytes=32.0 * size, flops=_evaluations(steps) * (FORCE_OPS[model] + GRAD_OPS[model]) * pairs)
    flops = _evaluations(steps) * FORCE_OPS[model] * pairs
    if case["energy"]:
        flops += POTENTIAL_OPS[model] * pairs
    return dict(bytes=32.0 * size, flops=flops)


# ------------------------------------------------- 64-bit values in torch ---

def _yoshida():
    t = 2.0 ** (1.0 / 3.0)
    w1, w0 = 1.0 / (2.0 - t), -t / (2.0 - t)
    return 0.5 * w1, 0.5 * (w0 + w1), w1, w0


def _rows(N):
    """Blocks of rows whose N-wide FP64 temporaries stay in cache."""
    step = max(1, min(N, 4_000_000 // N))
    return ((a, min(N, a + step)) for a in range(0, N, step))


def _force(model, q, eps):
    """Minus the gradient of the potential; q: (dim, N)."""
    N = q.shape[1]
    if model == "hmf":
        c, s = q[0].cos(), q[0].sin()
        return (c * s.mean() - s * c.mean())[None]
    if model == "sheet1d" and eps == 0.0:
        order, _ = q[0].sort()
        left = torch.searchsorted(order, q[0])
        right = N - torch.searchsorted(order, q[0], right=True)
        return ((right - left).double() / N)[None]
    f = torch.empty_like(q)
    for a, b in _rows(N):
        if model == "ring":
            d = q[0, a:b, None] - q[0]
            w = (0.5 * d).sin_()
            w.mul_(w).mul_(2.0).add_(eps)  # 1 - cos d + eps
            y = w.rsqrt()
            f[0, a:b] = d.sin_().mul_(y).div_(w).sum(1) * (-1.0 / (2.0 * math.sqrt(2.0) * N))
            continue
        d = [q[k, a:b, None] - q[k] for k in range(q.shape[0])]
        s = d[0] * d[0]
        for x in d[1:]:
            s.addcmul_(x, x)
        s.add_(eps)
        if model == "grav2d":
            s.reciprocal_()
            scale = -2.0 / N
        elif model == "grav3d":
            s = s.rsqrt().div_(s)
            scale = -1.0 / N
        else:  # softened sheets
            s.rsqrt_()
            scale = -1.0 / N
        for k, x in enumerate(d):
            f[k, a:b] = x.mul_(s).sum(1) * scale
    return f


def _potential(model, q, eps):
    N = q.shape[1]
    if model == "hmf":
        mx, my = q[0].cos().mean(), q[0].sin().mean()
        return float(0.5 * N * (1.0 - mx * mx - my * my))
    if model == "sheet1d" and eps == 0.0:
        gaps = q[0].sort()[0].diff()
        k = torch.arange(1, N, device=q.device, dtype=torch.float64)
        return float((gaps * k * (N - k)).sum() / N)
    total = 0.0
    for a, b in _rows(N):
        if model == "ring":
            w = (0.5 * (q[0, a:b, None] - q[0])).sin_()
            v = w.mul_(w).mul_(2.0).add_(eps).rsqrt_().mul_(-1.0 / (math.sqrt(2.0) * N))
        else:
            s = sum((q[k, a:b, None] - q[k]) ** 2 for k in range(q.shape[0])).add_(eps)
            v = s.log_() if model == "grav2d" else s.rsqrt_().neg_() if model == "grav3d" else s.sqrt_()
            v.div_(N)
        v[torch.arange(b - a, device=q.device), torch.arange(a, b, device=q.device)] = 0.0
        total += float(v.sum())
    return 0.5 * total


def _integrate(model, q, p, eps, dt, steps, kicks=None):
    """Advances (q, p), (dim, N) each, in place; appends (coefficient, q) of every kick to `kicks`."""
    B0, B1, D0, D1 = _yoshida()
    for t in range(steps):
        for b, d in (((B0 if t == 0 else 2.0 * B0), D0), (B1, D1), (B1, D0)):
            if kicks is not None:
                kicks.append((b, q.clone(), d))
            p.add_(_force(model, q, eps), alpha=b * dt)
            q.add_(p, alpha=d * dt)
    if kicks is not None:
        kicks.append((B0, q.clone(), 0.0))
    p.add_(_force(model, q, eps), alpha=B0 * dt)


def _jacobian_terms(model, q, v, eps):
    """(J(q) v, df/d eps) with J = df/dq."""
    N = q.shape[1]
    jv, de = torch.empty_like(q), torch.empty_like(q)
    for a, b in _rows(N):
        if model == "ring":
            d = q[0, a:b, None] - q[0]
            w = 2.0 * (0.5 * d).sin() ** 2 + eps
            S, C, y = d.sin(), d.cos(), w.rsqrt()
            y3 = y / w
            c = -1.0 / (2.0 * math.sqrt(2.0) * N)
            jv[0, a:b] = ((C * y3 - 1.5 * S * S * y3 / w) * (v[0, a:b, None] - v[0])).sum(1) * c
            de[0, a:b] = (S * y3 / w).sum(1) * (-1.5 * c)
            continue
        d = [q[k, a:b, None] - q[k] for k in range(2)]
        u = [v[k, a:b, None] - v[k] for k in range(2)]
        inv = 1.0 / (d[0] * d[0] + d[1] * d[1] + eps)
        ru = (d[0] * u[0] + d[1] * u[1]) * inv * inv
        for k in range(2):
            jv[k, a:b] = (u[k] * inv - 2.0 * d[k] * ru).sum(1) * (-2.0 / N)
            de[k, a:b] = (d[k] * inv * inv).sum(1) * (2.0 / N)
    return jv, de


def _gradient(case, q, p):
    model, eps, dt = case["model"], case["eps"], case["dt"]
    kicks = []
    _integrate(model, q, p, eps, dt, case["steps"], kicks)
    value, lp, lq, ge = 0.5 * float((p * p).sum()), p.clone(), torch.zeros_like(p), 0.0
    for b, at, d in reversed(kicks):
        lp = lp + d * dt * lq
        jv, de = _jacobian_terms(model, at, lp, eps)
        ge += b * dt * float((lp * de).sum())
        lq = lq + b * dt * jv
    return {"value": value, "grad_q": lq.reshape(-1).cpu().numpy(), "grad_p": lp.reshape(-1).cpu().numpy(),
            "grad_eps": ge}


def exact(case, seed):
    if case["kind"] == "ensemble":
        out = {}
        for s, (model, N, eps, dt) in enumerate(_members(case)):
            q, p = (x.cuda().reshape(DIM[model], N) for x in _member_state(model, N, seed, s))
            _integrate(model, q, p, eps, dt, case["steps"])
            out[str(s)] = (q.reshape(-1).cpu().numpy(), p.reshape(-1).cpu().numpy())
        return out
    model, N = case["model"], case["N"]
    q, p = (x.reshape(DIM[model], N).clone() for x in _state(model, N, _gen(seed, "cuda")))
    if case["kind"] == "grad":
        return _gradient(case, q, p)
    _integrate(model, q, p, case["eps"], case["dt"], case["steps"])
    out = {"q": q.reshape(-1), "p": p.reshape(-1)}
    if case["energy"]:
        out["K"], out["V"] = 0.5 * float((p * p).sum()), _potential(model, q, case["eps"])
    return out
