"""Measured cases of the direct-summation gravity library.

Each case is one pass through a public entry point, at sizes from the
repository's own workloads, tests and benchmark or of the same ranges:

  force       nb_force: Eq. (gravity) of one system (FP32 x, m -> a, p)
  kdk         nb_leapfrog_step: kick-drift-kick steps on FP64 state, a fixed
              time step; with "energy" also nb_energy, the conservation check
              that a run makes between segments
  batched     nb_force_batched: many independent clusters of uneven size
  batched_kdk nb_leapfrog_batched_step on such a batch, on a side stream (so
              that the steps after the first are replayed from a graph)
  vjp         autograd.force forward and backward with upstream gradients on
              a and p: a training step on forces
  trajectory  autograd.leapfrog forward and backward: gradients of a loss of
              the final positions with respect to x0, v0 and the masses

Particles are Plummer spheres (or, in a batch, Plummer spheres and uniform
balls by turns), drawn on the GPU from the seed. One context is kept for the
whole program, as a user's program keeps it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_0904_3659_gb300 as nb
from paper_0904_3659_gb300 import autograd as nbgrad

PLAIN, COMPENSATED = nb.NB_PLAIN, nb.NB_COMPENSATED

_kept = {}


def _context():
    if "ctx" not in _kept:
        _kept["ctx"] = nb.Context(0)
    return _kept["ctx"]


def _stream():
    if "stream" not in _kept:
        _kept["stream"] = torch.cuda.Stream()
    return _kept["stream"]


# ---------------------------------------------------------------------------
# The cases.

def listed():
    return [
        # The smallest calls: a star cluster of a thousand bodies inside a
        # host program's own loop; the launch counts as much as the sum.
        dict(name="force_1000", kind="force", n=1000, eps=1 / 64, mode=0, mass="equal"),
        # The single-evaluation workload.
        dict(name="force_4096", kind="force", n=4096, eps=0.01, mode=0, mass="equal"),
        # An odd mid size in the accurate mode.
        dict(name="force_10007_comp", kind="force", n=10007, eps=1 / 64, mode=1, mass="spectrum"),
        # A galaxy model of the integrated workload's size.
        dict(name="force_65536", kind="force", n=65536, eps=1 / 128, mode=0, mass="equal"),
        # Large, odd, unequal masses, accurate mode.
        dict(name="force_200003_comp", kind="force", n=200003, eps=1 / 128, mode=1, mass="spectrum"),
        # The throughput workload.
        dict(name="force_1m", kind="force", n=1 << 20, eps=1 / 256, mode=0, mass="equal"),
        # The integrated workload: the integrator needs no potential.
        dict(name="kdk_65536", kind="kdk", n=65536, eps=1 / 128, dt=1 / 4096, steps=8, mode=0,
             pot=False, energy=False, mass="equal"),
        # A production segment in the accurate mode: steps with the
        # potential, then the energy check.
        dict(name="kdk_energy_20011_comp", kind="kdk", n=20011, eps=1 / 64, dt=1 / 2048, steps=4,
             mode=1, pot=True, energy=True, mass="spectrum"),
        # The many-cluster workload: 1024 clusters of 32 to 4096 bodies.
        dict(name="batched_1024", kind="batched", clusters=1024, nmin=32, nmax=4096, sizes=0, mode=0),
        # A smaller ensemble integrated in the accurate mode.
        dict(name="batched_kdk_300_comp", kind="batched_kdk", clusters=300, nmin=32, nmax=2048,
             sizes=7, dt=1 / 4096, steps=4, mode=1),
        # A training step on forces at the differentiation workload's size.
        dict(name="vjp_16384", kind="vjp", n=16384, eps=1 / 64, mass="equal"),
        # Gradients through a trajectory.
        dict(name="trajectory_4096", kind="trajectory", n=4096, eps=1 / 64, dt=1 / 2048, steps=8,
             every=4, mode=0, mass="equal"),
    ]


def _between(rng, lo, hi):
    """An odd-or-even size spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "kdk", "batched", "batched_kdk", "vjp", "trajectory"])
    mass = rng.choice(["equal", "spectrum"])
    eps = 1.0 / rng.choice([32, 64, 128])
    mode = rng.choice([0, 1])
    if kind == "force":
        return dict(kind=kind, n=_between(rng, 700, 600000), eps=eps, mode=mode, mass=mass)
    if kind == "kdk":
        return dict(kind=kind, n=_between(rng, 2000, 120000), eps=eps, dt=1 / 4096, steps=rng.randint(1, 6),
                    mode=mode, pot=rng.random() < 0.5, energy=rng.random() < 0.5, mass=mass)
    if kind in ("batched", "batched_kdk"):
        nmax = rng.choice([512, 1024, 2048, 4096])
        case = dict(kind=kind, clusters=_between(rng, 20, 1200 if kind == "batched" else 400), nmin=32,
                    nmax=nmax, sizes=rng.randrange(1 << 30), mode=mode)
        if kind == "batched_kdk":
            case.update(dt=1 / 8192, steps=rng.randint(2, 8))
        return case
    if kind == "vjp":
        return dict(kind=kind, n=_between(rng, 700, 90000), eps=eps, mass=mass)
    return dict(kind=kind, n=_between(rng, 500, 6000), eps=eps, dt=1 / 2048, steps=rng.randint(2, 8),
                every=rng.choice([0, 2, 4]), mode=mode, mass=mass)


# ---------------------------------------------------------------------------
# Inputs, drawn on the GPU from the seed.

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _directions(g, n):
    u = torch.rand((2, n), generator=g, device="cuda", dtype=torch.float64)
    cz, phi = 1 - 2 * u[0], 2 * math.pi * u[1]
    sz = torch.sqrt(torch.clamp(1 - cz * cz, min=0))
    return torch.stack([sz * torch.cos(phi), sz * torch.sin(phi), cz], dim=1)


def _speeds(g, n):
    """q = v / v_escape of a Plummer sphere, from g(q) ~ q^2 (1 - q^2)^{7/2}
    by the inverse of its tabulated cumulative distribution."""
    q = torch.linspace(0, 1, 4097, device="cuda", dtype=torch.float64)
    c = torch.cumsum(q * q * (1 - q * q) ** 3.5, 0)
    c = c / c[-1]
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    k = torch.clamp(torch.searchsorted(c, u), 1, 4096)
    return q[k - 1] + (q[k] - q[k - 1]) * (u - c[k - 1]) / torch.clamp(c[k] - c[k - 1], min=1e-300)


def _plummer(g, n):
    """x, v (FP64) of a Plummer sphere, G = M = scale radius = 1, r <= 100."""
    most = (100.0 ** 3) / (100.0 ** 2 + 1) ** 1.5
    X = torch.clamp(torch.rand(n, generator=g, device="cuda", dtype=torch.float64), min=1e-12) * most
    r = 1 / torch.sqrt(X ** (-2 / 3) - 1)
    x = r[:, None] * _directions(g, n)
    v = (_speeds(g, n) * math.sqrt(2) * (1 + r * r) ** -0.25)[:, None] * _directions(g, n)
    return x, v


def _masses(g, n, kind):
    """FP32 masses of total 1: equal, or a power-law spectrum over a factor of 30."""
    if kind == "equal":
        return torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float32)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    lo, hi, e = 1.0, 30.0, -1.35
    m = (lo ** e + u * (hi ** e - lo ** e)) ** (1 / e)
    return (m / m.sum()).to(torch.float32)


def _sizes(case):
    r = np.random.default_rng(case["sizes"])
    logn = r.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["clusters"])
    return np.clip(np.rint(np.exp(logn)).astype(np.int64), case["nmin"], case["nmax"])


def _clusters(g, case):
    """Concatenated clusters: Plummer spheres (even) and cold uniform balls
    (odd) of random radius in [0.5, 2], softening 0.02 of the radius."""
    sizes = torch.from_numpy(_sizes(case)).cuda()
    C, n = case["clusters"], int(sizes.sum())
    offsets = torch.zeros(C + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = torch.cumsum(sizes, 0)
    which = torch.repeat_interleave(torch.arange(C, device="cuda"), sizes, output_size=n)
    radius = 0.5 + 1.5 * torch.rand(C, generator=g, device="cuda", dtype=torch.float64)
    xp, vp = _plummer(g, n)
    ball = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) ** (1 / 3)
    xb = ball[:, None] * _directions(g, n)
    even = (which % 2 == 0)[:, None]
    R = radius[which][:, None]
    x = torch.where(even, xp, xb) * R
    v = torch.where(even, vp / torch.sqrt(R), torch.zeros_like(vp))
    m = (1.0 / sizes.to(torch.float64))[which].to(torch.float32)
    return x, v, m, offsets, (0.02 * radius).to(torch.float32), n


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    s = dict(case=dict(case), ctx=_context())
    if kind in ("batched", "batched_kdk"):
        x, v, m, offsets, eps, n = _clusters(g, case)
        s.update(n=n, m=m, offsets=offsets, eps=eps)
        s["a"] = torch.empty((n, 3), device="cuda", dtype=torch.float32)
        s["p"] = torch.empty((n,), device="cuda", dtype=torch.float32)
        if kind == "batched":
            s["x"] = x.to(torch.float32)
        else:
            s.update(x=x, v=v, stream=_stream())
        return s
    n = case["n"]
    x, v = _plummer(g, n)
    m = _masses(g, n, case["mass"])
    s.update(n=n, m=m, eps=float(np.float32(case["eps"])))
    if kind == "force":
        s.update(x=x.to(torch.float32), a=torch.empty((n, 3), device="cuda"), p=torch.empty(n, device="cuda"))
    elif kind == "kdk":
        s.update(x=x, v=v, a=torch.empty((n, 3), device="cuda"), p=torch.empty(n, device="cuda") if case["pot"] else None)
    elif kind == "vjp":
        s["x"] = x.to(torch.float32).requires_grad_(True)
        s["m"] = m.requires_grad_(True)
        s["ga"] = torch.randn((n, 3), generator=g, device="cuda")
        s["gp"] = torch.randn(n, generator=g, device="cuda")
    else:
        s.update(x=x.requires_grad_(True), v=v.requires_grad_(True), m=m.requires_grad_(True))
        s["y"] = x.detach() + 0.05 * torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    return s


# ---------------------------------------------------------------------------
# One pass.

def run(state):
    s, c = state, state["case"]
    ctx, n, kind = s["ctx"], s["n"], c["kind"]
    if kind == "force":
        nb.nb_force(ctx, s["x"], s["m"], n, s["eps"], s["a"], s["p"], c["mode"])
        return s["a"], s["p"]
    if kind == "kdk":
        nb.nb_leapfrog_step(ctx, s["x"], s["v"], s["m"], s["a"], s["p"], n, s["eps"], c["dt"], c["steps"], 0,
                            c["mode"])
        out = [s["x"], s["v"], s["a"]] + ([s["p"]] if c["pot"] else [])
        if c["energy"]:
            out += list(nb.nb_energy(ctx, s["x"], s["v"], s["m"], n, s["eps"], c["mode"]))
        return out
    if kind == "batched":
        nb.nb_force_batched(ctx, s["x"], s["m"], s["offsets"], c["clusters"], n, s["eps"], s["a"], s["p"], c["mode"])
        return s["a"], s["p"]
    if kind == "batched_kdk":
        nb.nb_leapfrog_batched_step(ctx, s["x"], s["v"], s["m"], s["offsets"], c["clusters"], n, s["eps"], s["a"],
                                    s["p"], c["dt"], c["steps"], 0, c["mode"], s["stream"])
        return s["x"], s["v"], s["a"], s["p"]
    if kind == "vjp":
        a, p = nbgrad.force(s["x"], s["m"], s["eps"], PLAIN, ctx)
        gx, gm = torch.autograd.grad((a, p), (s["x"], s["m"]), (s["ga"], s["gp"]))
        return a, p, gx, gm
    x, v = nbgrad.leapfrog(s["x"], s["v"], s["m"], s["eps"], c["dt"], c["steps"], c["every"], c["mode"], ctx)
    loss = ((x - s["y"]) ** 2).sum()
    gx, gv, gm = torch.autograd.grad(loss, (s["x"], s["v"], s["m"]))
    return x, v, gx, gv, gm


# ---------------------------------------------------------------------------
# What a pass cannot do without. An evaluation of n bodies has n (n - 1) / 2
# distinct pairs; each takes at least 3 subtractions, 5 operations for r^2 +
# eps^2 and one reciprocal square root, then per pair and output: the cube and
# both weights (4) and both sums of 3 products (12) for a, both products and
# sums (4) for p.

def _pair_flops(pot=True, acc=True):
    return 9 + (16 if acc else 0) + (4 if pot else 0)


def work(case):
    kind = case["kind"]
    if kind in ("batched", "batched_kdk"):
        z = _sizes(case).astype(np.float64)
        n, pairs = float(z.sum()), float((z * (z - 1) / 2).sum())
        if kind == "batched":
            return dict(bytes=32 * n + 12 * case["clusters"], flops=pairs * _pair_flops())
        steps = case["steps"]
        return dict(bytes=(96 + 4 + 16) * n, flops=(steps + 1) * pairs * _pair_flops())
    n = float(case["n"])
    pairs = n * (n - 1) / 2
    if kind == "force":
        return dict(bytes=32 * n, flops=pairs * _pair_flops())
    if kind == "kdk":
        flops = (case["steps"] + 1) * pairs * _pair_flops(False) + pairs * 4 * (1 if case["pot"] else 0)
        if case["energy"]:
            flops += pairs * _pair_flops(True, False)
        return dict(bytes=(96 + 4 + 12 + (4 if case["pot"] else 0)) * n, flops=flops)
    # The adjoint, per distinct pair: the difference, r^2 + eps^2 and its
    # reciprocal square root (9), both scalar products with ga (10), the
    # coefficient of r, shared by both (13 with gp, 8 without), both sums of r
    # (12), of m y^3 (4) and of y^3 ga (12), and the mass gradient's (8 or 4).
    if kind == "vjp":
        return dict(bytes=(16 + 16 + 16 + 16) * n, flops=pairs * (_pair_flops() + 68))
    k = case["steps"]
    return dict(bytes=(2 * 48 + 4 + 24 + 48 + 4) * n,
                flops=pairs * ((k + 1) * _pair_flops(False) + (k + 1) * 59))


# ---------------------------------------------------------------------------
# The same in plain FP64 torch.

def _force64(x, m, e2, rows=None, pot=True):
    """a, p of Eq. (gravity) in FP64, in blocks of rows; a has the printed sign."""
    n = x.shape[0]
    step = max(1, min(n, (1 << 26) // max(n, 1)))
    a, p = [], []
    for i in range(0, n, step):
        d = [x[i:i + step, k, None] - x[None, :, k] for k in range(3)]
        y = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + e2)
        k = torch.arange(y.shape[0], device=x.device)
        y[k, k + i] = 0
        if pot:
            p.append(y @ m)
        w = y * y * y * m
        a.append(torch.stack([(w * dk).sum(1) for dk in d], dim=1))
    return torch.cat(a), torch.cat(p) if pot else None


def _energy64(x, v, m, e2):
    _, p = _force64(x, m, e2)
    return float(0.5 * (m * (v * v).sum(1)).sum()), float(-0.5 * (m * p).sum())


def _kdk64(x, v, m, e2, dt, steps):
    a, p = _force64(x, m, e2)
    for _ in range(steps):
        v = v - 0.5 * dt * a
        x = x + dt * v
        a, p = _force64(x, m, e2)
        v = v - 0.5 * dt * a
    return x, v, a, p


def _vjp64(x, m, e2, ga, gp):
    """Gradients of sum ga.a + gp p with respect to x and m, in blocks of rows."""
    n = x.shape[0]
    step = max(1, min(n, (1 << 26) // max(n, 1)))
    gx, gm = torch.empty_like(x), torch.empty_like(m)
    for i in range(0, n, step):
        d = [x[i:i + step, k, None] - x[None, :, k] for k in range(3)]
        y = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + e2)
        k = torch.arange(y.shape[0], device=x.device)
        y[k, k + i] = 0
        y3 = y * y * y
        gi, gl = ga[i:i + step], ga
        ri = sum(d[c] * gi[:, c, None] for c in range(3))
        rl = sum(d[c] * gl[None, :, c] for c in range(3))
        mi = m[i:i + step]
        coef = 3 * y3 * y * y * (mi[:, None] * rl - m[None, :] * ri) - y3 * (
            gp[i:i + step, None] * m[None, :] + mi[:, None] * gp[None, :])
        S = y3 @ m
        V = y3 @ ga
        R = torch.stack([(coef * dk).sum(1) for dk in d], dim=1)
        gx[i:i + step] = R + gi * S[:, None] - mi[:, None] * V
        gm[i:i + step] = (y @ gp) - (y3 * rl).sum(1)
    return gx, gm


def _trajectory64(x0, v0, m, e2, dt, steps, y):
    """Final state and gradients of sum |x - y|^2: the reverse sweep of the steps."""
    xs, x, v = [x0], x0, v0
    a, _ = _force64(x, m, e2, pot=False)
    for _ in range(steps):
        v = v - 0.5 * dt * a
        x = x + dt * v
        a, _ = _force64(x, m, e2, pot=False)
        v = v - 0.5 * dt * a
        xs.append(x)
    zero = torch.zeros_like(m)
    lx, lv, la, lm = 2 * (x - y), torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(m)
    for t in range(steps - 1, -1, -1):
        la = la - 0.5 * dt * lv
        gx, gm = _vjp64(xs[t + 1], m, e2, la, zero)
        lx, lm = lx + gx, lm + gm
        lv = lv + dt * lx
        la = -0.5 * dt * lv
    gx, gm = _vjp64(xs[0], m, e2, la, zero)
    return x, v, lx + gx, lv, lm + gm


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("batched", "batched_kdk"):
        evals = {"force": 1, "vjp": 3}.get(kind, case.get("steps", 0) * (1 if kind == "kdk" else 4) + 3)
        if evals * float(case["n"]) ** 2 > 1.5e11:
            return None
    s = prepare(case, seed)
    m = s["m"].detach().to(torch.float64)
    x = s["x"].detach().to(torch.float64)
    if kind in ("batched", "batched_kdk"):
        off, eps = s["offsets"].tolist(), s["eps"].to(torch.float64).tolist()
        parts = []
        for c in range(case["clusters"]):
            r, e2 = slice(off[c], off[c + 1]), eps[c] ** 2
            parts.append(_force64(x[r], m[r], e2) if kind == "batched"
                         else _kdk64(x[r], s["v"][r], m[r], e2, case["dt"], case["steps"]))
        return tuple(torch.cat(v) for v in zip(*parts))
    e2 = s["eps"] ** 2
    if kind == "force":
        return _force64(x, m, e2)
    if kind == "kdk":
        x, v, a, p = _kdk64(x, s["v"], m, e2, case["dt"], case["steps"])
        return [x, v, a] + ([p] if case["pot"] else []) + (list(_energy64(x, v, m, e2)) if case["energy"] else [])
    if kind == "vjp":
        return _force64(x, m, e2) + _vjp64(x, m, e2, s["ga"].to(torch.float64), s["gp"].to(torch.float64))
    return _trajectory64(x, s["v"].detach(), m, e2, case["dt"], case["steps"], s["y"])
