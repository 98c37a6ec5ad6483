"""The work this library does for its users, as cases to time: what a time-stepping gravity code calls
through the binding, from a 4096-particle box to a 384^3 one.

Kinds of case (the "kind" field):
  solve    one force solve of an isolated or periodic box (fmm_compute_forces), every particle active
  i32      the same on 32-bit fixed-point positions (fmm_compute_forces_i32)
  host     the same through host buffers, copies included (fmm_compute_forces_host)
  batch    many independent boxes in one pass (fmm_compute_forces_batch)
  substep  the solve of one rung substep, a small part of the particles active
  dual     an interval of the dual-tree scheme: the fixed tree, then the substeps inside it
  learned  a solve with the learned opening criterion, the last step's accelerations as estimate
  kick     the kick-drift of one rung substep
  train    training the learned criterion's network on labelled pairs

Particle sets are seeded stand-ins for clustered cosmological boxes: "plummer" is half uniform and half in
four Plummer spheres, "nfw" 30% uniform and the rest in 200 NFW halos of masses over three decades.
Softening is 1/50 of the mean separation unless a case names it.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1609_08621_gb300 import binding

DEV = "cuda:0"


def listed():
    return [
        # the smallest box a user solves, step after step on the same buffers: launches and latency
        dict(name="solve_4096", kind="solve", set="plummer", n=4096, eps=1e-3, theta=0.7, graph=True),
        # a single solve with the library's defaults, nothing kept between calls but the context
        dict(name="solve_nfw_63cubed", kind="solve", set="nfw", n=63 ** 3, theta=0.55, graph=False),
        # the ordinary time step: 128^3 clustered box, replayed, sums in FP64, the tuner's chunk
        dict(name="solve_nfw_128cubed", kind="solve", set="nfw", n=128 ** 3, theta=0.55, graph=True, accumulate=1,
             chunk=128),
        # the same box with periodic boundaries (replica shell of 1 and the Ewald correction)
        dict(name="periodic_nfw_128cubed", kind="solve", set="nfw", n=128 ** 3, theta=0.55, graph=True, nrep=1,
             accumulate=1, chunk=128),
        # a large box whose positions are stored compressed: the largest call here
        dict(name="compressed_384cubed", kind="i32", set="plummer", n=384 ** 3, theta=0.55, graph=False,
             accumulate=1, chunk=128),
        # a program that keeps its particles in host memory
        dict(name="host_200k", kind="host", set="plummer", n=200_003, theta=0.6, graph=False),
        # an ensemble of independent boxes of unequal sizes
        dict(name="batch_64_boxes", kind="batch", boxes=64, lo=32 ** 3, hi=96 ** 3, eps=1e-3, theta=0.7, graph=False,
             accumulate=1, chunk=128),
        # one substep of the rung hierarchy: about a tenth of a 256^3 box is active
        dict(name="substep_256cubed", kind="substep", set="plummer", n=256 ** 3, theta=0.55, active=0.1, graph=False,
             accumulate=1, chunk=128),
        # the rest of that substep: kicks of the active particles, drift of all
        dict(name="kick_drift_256cubed", kind="kick", n=256 ** 3, max_rung=5, active=0.1),
        # multiple time steps with dual trees: the fixed tree and three substeps of an interval
        dict(name="dual_60cubed", kind="dual", set="nfw", n=60 ** 3, theta=0.55, fast=0.2),
        # a step with the learned opening criterion
        dict(name="learned_200cubed", kind="learned", set="plummer", n=200 ** 3, theta=0.55, tau=-4.8, graph=True,
             accumulate=1, chunk=128),
        # training that criterion's network on audited pairs
        dict(name="train_200k_rows", kind="train", rows=200_000, epochs=2, batch=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "i32", "host", "batch", "substep", "dual", "learned", "kick", "train"])
    if kind == "kick":
        return dict(kind=kind, n=_log_int(rng, 20_000, 40_000_000), max_rung=rng.randint(1, 8),
                    active=round(rng.uniform(0.05, 0.5), 3))
    if kind == "train":
        return dict(kind=kind, rows=_log_int(rng, 20_000, 400_000), epochs=rng.randint(1, 3),
                    batch=rng.choice([256, 1000, 4096]))
    c = dict(kind=kind, theta=round(rng.uniform(0.5, 0.75), 3), bucket=rng.choice([8, 12, 16, 16]),
             group=rng.choice([32, 48, 64, 64]), chunk=rng.choice([32, 64, 128]), accumulate=rng.randint(0, 1))
    if kind == "batch":
        hi = _log_int(rng, 3_000, 500_000)
        c.update(boxes=rng.randint(2, 64), lo=max(500, hi // rng.randint(2, 27)), hi=hi, eps=1e-3,
                 graph=rng.random() < 0.5)
        return c
    c.update(set=rng.choice(["plummer", "nfw"]))
    top = {"solve": 16_000_000, "i32": 30_000_000, "host": 2_000_000, "substep": 16_000_000, "dual": 2_000_000,
           "learned": 8_000_000}[kind]
    c.update(n=_log_int(rng, 2_000, top))
    if kind == "solve":
        c.update(graph=rng.random() < 0.5, nrep=rng.choice([0, 0, 0, 1, 2]))
        if c["nrep"]:
            c["n"] = min(c["n"], 4_000_000)
    elif kind == "dual":
        c.update(fast=round(rng.uniform(0.05, 0.4), 3))
    else:
        c.update(graph=kind != "host" and rng.random() < 0.5)
    if kind == "substep":
        c.update(active=round(rng.uniform(0.03, 0.5), 3))
    if kind == "learned":
        c.update(tau=round(rng.uniform(-5.3, -4.4), 2))
    return c


# ---------------------------------------------------------------- particle sets (seeded, made on the GPU)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _sphere(g, r):
    """Points at the radii r in isotropic directions, 3 x len(r)."""
    cz = 2.0 * _rand(g, r.numel()) - 1.0
    ph = (2.0 * math.pi) * _rand(g, r.numel())
    sz = (1.0 - cz * cz).clamp_(min=0.0).sqrt_()
    return torch.stack([r * sz * ph.cos(), r * sz * ph.sin(), r * cz])


def _into_box(g, p):
    """Points outside [0, 1)^3 are drawn again, uniformly."""
    out = ~((p >= 0.0) & (p < 1.0)).all(0)
    return torch.where(out, _rand(g, 3, p.shape[1]), p)


def _shuffled(g, parts, n):
    p = torch.cat(parts, 1)
    return p[:, torch.randperm(n, generator=g, device=DEV)].contiguous()


def _plummer(g, n):
    n_uni = n // 2
    n_cl = n - n_uni
    centre = 0.2 + 0.6 * _rand(g, 3, 4)
    u = _rand(g, n_cl).clamp_(1e-12, 1.0 - 1e-12)
    p = _sphere(g, 0.02 / (u.pow(-2.0 / 3.0) - 1.0).sqrt())
    p += centre[:, torch.arange(n_cl, device=DEV) * 4 // max(n_cl, 1)]
    return _shuffled(g, [_rand(g, 3, n_uni), _into_box(g, p)], n)


def _nfw(g, n, halos=200, slope=1.9, decades=3.0, rvir=0.05):
    n_uni = int(0.3 * n)
    n_cl = n - n_uni
    k, t = 1.0 - slope, 10.0 ** (-decades * (1.0 - slope))
    m = (t + _rand(g, halos) * (1.0 - t)).pow(1.0 / k)  # dN/dM ~ M^-slope over the decades
    m = m / m.max()
    c = 5.0 + 10.0 * _rand(g, halos)
    centre = 0.1 + 0.8 * _rand(g, 3, halos)
    h = torch.bucketize(_rand(g, n_cl), (m.cumsum(0) / m.sum())[:-1].contiguous())
    # radius from the enclosed mass mu(x) = ln(1 + x) - x / (1 + x), by bisection
    mu = lambda x: torch.log1p(x) - x / (1.0 + x)  # noqa: E731
    ch = c[h]
    want = _rand(g, n_cl) * mu(ch)
    a, b = torch.zeros_like(ch), ch.clone()
    for _ in range(40):
        mid = 0.5 * (a + b)
        low = mu(mid) < want
        a, b = torch.where(low, mid, a), torch.where(low, b, mid)
    p = _sphere(g, 0.5 * (a + b) / ch * (rvir * m.pow(1.0 / 3.0))[h]) + centre[:, h]
    return _shuffled(g, [_rand(g, 3, n_uni), _into_box(g, p)], n)


def _positions(case, g, n=None):
    n = case["n"] if n is None else n
    return (_nfw if case.get("set") == "nfw" else _plummer)(g, n)


def _eps(case):
    return case.get("eps") or 1.0 / (50.0 * case["n"] ** (1.0 / 3.0))


def _box_sizes(case):
    """Particles per box, uniform in [lo, hi]: an ensemble keeps its boxes from step to step."""
    r = np.random.Generator(np.random.PCG64(case["boxes"] + case["hi"]))
    return r.integers(case["lo"], case["hi"] + 1, case["boxes"])


def _fixed_point(pos):
    """Positions in [0, 1) as 32-bit fixed-point coordinates, in the int32 that holds the bits."""
    u = (pos * 4294967296.0).round_().clamp_(max=4294967295.0).to(torch.int64)
    return torch.where(u >= 1 << 31, u - (1 << 32), u).to(torch.int32)


# ---------------------------------------------------------------- the learned criterion's network


def _pair_rows(r, n):
    """Feature rows (sizes of sink and source over distance, softening, pull relative to the sink's own
    acceleration, particle counts, moment norms) and labels (log10 of the relative error of accepting the
    pair, which falls with the sixth power of the opening angle) as an audit of clustered boxes gives them."""
    te = np.exp(r.uniform(math.log(0.35), 0.0, n))
    share = r.uniform(0.15, 0.75, n)
    f = np.empty((n, 8))
    f[:, 0] = te * share
    f[:, 1] = te * (1.0 - share) / 1.5
    f[:, 2] = 10.0 ** r.uniform(-4.5, -1.5, n)
    f[:, 3] = r.uniform(-5.5, -0.5, n)
    f[:, 4] = r.uniform(1.0, 18.0, n)
    f[:, 5] = r.uniform(1.0, 18.0, n)
    f[:, 6] = r.uniform(0.15, 0.9, n)
    f[:, 7] = f[:, 6] ** 2 * r.uniform(0.5, 1.0, n)
    y = f[:, 3] + 6.0 * np.log10(te) + 0.5 * (f[:, 6] - 0.5) - 0.02 * f[:, 4]
    y += 1.5 * (share - 0.45) ** 2 - 0.3 * (f[:, 6] - 0.5) * (f[:, 4] - 9.0) / 9.0 + 0.15 * r.standard_normal(n)
    return f, y


@functools.lru_cache(maxsize=1)
def _network():
    """A trained network's parameters, the same for every seed as a program's file of weights would be:
    hidden units that carry the features, hinges along the opening angle and random directions, the output
    layer fitted to the rows above, then the surrogate bound."""
    r = np.random.Generator(np.random.PCG64(20160908))
    f, y = _pair_rows(r, 20_000)
    mean, istd = f.mean(0), 1.0 / f.std(0)
    h = (f - mean) * istd
    w1, b1 = r.standard_normal((64, 8)) / math.sqrt(8.0), r.uniform(-1.0, 1.0, 64)
    w1[:8], b1[:8] = np.eye(8), 4.0
    te = np.zeros(8)
    te[0], te[1] = 1.0 / istd[0], 1.5 / istd[1]
    knots = np.exp(np.linspace(math.log(0.34), math.log(0.95), 24))
    w1[8:32] = 4.0 * te
    b1[8:32] = 4.0 * (mean[0] + 1.5 * mean[1] - knots)
    h = np.maximum(h @ w1.T + b1, 0.0)
    parts = [w1.ravel(), b1]
    for _ in range(2):
        w, b = np.eye(64), np.zeros(64)
        w[32:, 32:] += r.standard_normal((32, 32)) * 0.1
        h = np.maximum(h @ w.T + b, 0.0)
        parts += [w.ravel(), b]
    a = np.c_[h, np.ones(len(y))]
    w4 = np.linalg.solve(a.T @ a + 1e-5 * len(y) * np.eye(65), a.T @ y)
    x = np.c_[np.log10(1.5 * f[:, 1] + f[:, 0]), np.ones(len(y)), f]
    s = np.sqrt((x * x).mean(0))
    co = np.linalg.solve((x / s).T @ (x / s) + 1e-6 * len(y) * np.eye(10), (x / s).T @ (y - f[:, 3])) / s
    lo, hi = np.quantile(a @ w4 - (f[:, 3] + x @ co), [0.0005, 0.9995])
    return np.concatenate(parts + [w4, mean, istd, [co[0], co[1], lo, hi], co[2:]]).astype(np.float32)


# ---------------------------------------------------------------- prepare and run


class State:
    pass


def _context(case):
    p = {k: case[q] for k, q in (("bucket", "bucket"), ("group", "group"), ("list_chunk", "chunk"),
                                 ("accumulate", "accumulate"), ("nrep", "nrep")) if q in case}
    ctx = binding.Context(0, **p)
    if case.get("graph"):
        ctx.set_graphs(True)
    return ctx


def prepare(case, seed):
    s, g, kind = State(), _gen(seed), case["kind"]
    s.case = case
    if kind == "train":
        f, y = _pair_rows(np.random.Generator(np.random.PCG64(int(seed))), case["rows"])
        s.feats = torch.from_numpy(f.astype(np.float32)).to(DEV)
        s.labels = torch.from_numpy(y.astype(np.float32)).to(DEV)
        s.ctx = binding.Context(0)
        return s
    if kind == "batch":
        s.off = np.concatenate([[0], np.cumsum(_box_sizes(case))]).astype(np.int64)
        s.n = int(s.off[-1])
        s.pos = torch.cat([_plummer(g, int(k)) for k in np.diff(s.off)], 1).contiguous().view(-1)
        s.mass = torch.cat([torch.full((int(k),), 1.0 / int(k), device=DEV) for k in np.diff(s.off)])
    else:
        s.n = case["n"]
        s.mass = torch.full((s.n,), 1.0 / s.n, device=DEV)
        if kind == "kick":
            s.pos = _rand(g, 3 * s.n) * 0.98 + 0.01
        else:
            s.pos = _positions(case, g).view(-1)
    n = s.n
    s.acc = torch.zeros(3 * n, device=DEV)
    s.pot = torch.zeros(n, device=DEV)
    s.active = None
    s.ctx = _context(case)
    if kind == "i32":
        s.pos = _fixed_point(s.pos)
    elif kind == "host":
        s.pinned = [t.cpu().pin_memory() for t in (s.pos, s.mass, s.acc, s.pot)]
        s.pos, s.mass, s.acc, s.pot = [t.numpy() for t in s.pinned]
    elif kind == "substep":
        s.active = (_rand(g, n) < case["active"]).to(torch.uint8)
        s.active[0] = 1
    elif kind == "dual":
        # rungs 0-3; the particles of rungs 2 and 3 are the fast ones
        u = _rand(g, n)
        s.rung = ((u < case["fast"]).to(torch.uint8) * 2) + (u < 0.5 * case["fast"]).to(torch.uint8)
        s.rung[0] = 3
        v = 1e-3 * (_rand(g, 3 * n) - 0.5)
        s.dt = 1e-3
        end = s.pos + v * s.dt  # the slow particles' middle of the interval stays in the box
        s.vel = torch.where((end >= 0.0) & (end < 1.0), v, torch.zeros_like(v))
        s.sinks = [(s.rung >= 3).to(torch.uint8), (s.rung >= 2).to(torch.uint8)]
    elif kind == "learned":
        s.ctx.mlp_load(_network())
        s.ctx.compute_forces(s.pos, s.mass, _eps(case), case["theta"], s.acc, s.pot)  # the last step's
        s.ctx.set_params(criterion=1, mlp_tau=case["tau"])
    elif kind == "kick":
        s.vel = 1e-3 * (_rand(g, 3 * n) - 0.5)
        s.acc = (20.0 * (_rand(g, 3 * n) - 0.5)).float()
        R = case["max_rung"]
        lower = (_rand(g, n) * R).floor_().clamp_(max=R - 1)
        s.rung = torch.where(_rand(g, n) < case["active"], torch.full_like(lower, R), lower).to(torch.uint8)
        s.next = torch.zeros(n, dtype=torch.uint8, device=DEV)
    return s


def run(s):
    case, ctx, kind = s.case, s.ctx, s.case["kind"]
    if kind == "train":
        loss = ctx.mlp_train(s.feats, s.labels, epochs=case["epochs"], batch=case["batch"], lr=4e-3, seed=1)
        return {"weights": ctx.mlp_get(), "loss": np.float32(loss)}
    if kind == "kick":
        # an odd substep: the finest rung's particles are active; a base step far below their own time step
        ctx.kick_drift(s.pos, s.vel, s.acc, s.rung, s.next, _eps(case), 1e-6, case["max_rung"], 1, 1)
        return {"pos": s.pos, "vel": s.vel, "rung": s.rung, "next": s.next}
    eps, theta = _eps(case), case["theta"]
    if kind == "batch":
        ctx.compute_forces_batch(s.pos, s.mass, s.off, eps, theta, s.acc, s.pot)
    elif kind == "i32":
        ctx.compute_forces_i32(s.pos, s.mass, eps, theta, s.acc, s.pot)
    elif kind == "host":
        ctx.compute_forces_host(s.pos, s.mass, eps, theta, s.acc, s.pot)
    elif kind == "dual":
        ctx.set_fixed_sources(s.pos, s.mass, s.rung, 1, s.vel, s.dt)
        for k in (0, 1, 0):
            ctx.compute_forces_dual(s.pos, s.mass, eps, theta, s.acc, s.pot, s.sinks[k])
    else:
        ctx.compute_forces(s.pos, s.mass, eps, theta, s.acc, s.pot, s.active)
    return {"acc": s.acc, "pot": s.pot}


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    """Bytes: every input read once, every output written once.  Flops: of a solve, the FP32 interactions of
    the method at its opening angle (about 1000 particle pairs of 19 flops, 220 particle-cell pairs of 293 and
    8 cell-cell pairs of 1110 per active particle at 0.55, the last two falling with its cube)."""
    kind = case["kind"]
    if kind == "train":
        rows = case["rows"] * case["epochs"]
        return {"bytes": rows * 36, "flops": rows * 6 * 8960}
    if kind == "kick":
        # drift: pos in and out, vel in; rung in, flag out; kicks of the active: acc in, vel out
        return {"bytes": case["n"] * (24 + 24 + 24 + 2 + case["active"] * (12 + 24)), "flops": case["n"] * 12}
    if kind == "batch":
        n = int(_box_sizes(case).sum())
    else:
        n = case["n"]
    frac = case.get("active", 1.0) if kind == "substep" else 1.0
    if kind == "dual":
        frac = case["fast"] * 2.0  # three solves: half, all and half of the fast particles
    far = (0.55 / case["theta"]) ** 3
    return {"bytes": n * (16.0 if kind == "i32" else 28.0) + n * frac * 16.0,
            "flops": n * frac * (1000 * 19 + far * (220 * 293 + 8 * 1110))}


# ---------------------------------------------------------------- the same in 64 bits


def _direct(src, mass, eps, sinks, at):
    """The softened direct sum in FP64: acceleration (3 x k) and potential (k) of the sinks (3 x k), each of
    which is source number at[i] and does not feel itself."""
    k, n = sinks.shape[1], src.shape[1]
    acc, pot = torch.empty(3, k, device=DEV, dtype=torch.float64), torch.empty(k, device=DEV, dtype=torch.float64)
    step = max(1, 60_000_000 // n)
    for b in range(0, k, step):
        e = min(k, b + step)
        d = [src[a][None, :] - sinks[a, b:e, None] for a in range(3)]
        w = torch.addcmul(torch.full_like(d[0], eps * eps), d[0], d[0])
        w.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        ir = w.rsqrt_()
        m = ir * mass
        m.scatter_(1, at[b:e, None], 0.0)
        pot[b:e] = -m.sum(1)
        m.mul_(ir).mul_(ir)
        for a in range(3):
            acc[a, b:e] = (d[a].mul_(m)).sum(1)
    return acc, pot


def exact(case, seed):
    kind = case["kind"]
    if kind == "kick":
        s = prepare(case, seed)
        R, n = case["max_rung"], s.n
        on = (s.rung == R).repeat(3)
        a = s.acc.double()
        # closing and opening half kicks of the finest rung, whose particles stay there on an odd substep
        hk = 1e-6 * 2.0 ** -(R + 1)
        vel = torch.where(on, (s.vel + a * hk) + a * hk, s.vel)
        return {"pos": s.pos + vel * (1e-6 * 2.0 ** -R), "vel": vel, "rung": None, "next": None}
    if kind in ("train", "batch", "learned") or case.get("nrep") or case["n"] > 260_000:
        return None
    s = prepare(case, seed)
    if kind == "host":
        s.pos, s.mass = [torch.from_numpy(x).to(DEV) for x in (s.pos, s.mass)]
    if kind == "i32":
        s.pos = (s.pos.to(torch.int64) & 0xFFFFFFFF).double() * 2.0 ** -32
    n, eps = s.n, _eps(case)
    pos, mass = s.pos.view(3, n), s.mass.double()
    acc, pot = torch.zeros(3, n, device=DEV, dtype=torch.float64), torch.zeros(n, device=DEV, dtype=torch.float64)
    src, on = pos, torch.arange(n, device=DEV)
    if kind == "substep":
        on = s.active.nonzero().view(-1)
    elif kind == "dual":
        src = torch.where(s.rung <= 1, pos + s.vel.view(3, n) * s.dt, pos)
        on = (s.rung >= 2).nonzero().view(-1)
    acc[:, on], pot[on] = _direct(src, mass, eps, pos[:, on].contiguous(), on)
    return {"acc": acc.view(-1), "pot": pot}
