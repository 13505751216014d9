"""The workloads this library's speed is measured on, each through its public entry points.

A case is a dict of plain values; ``listed`` gives the fixed ones, ``draw`` one more of the same
ranges.  ``prepare`` makes what a program holds before the call (seeded inputs on the GPU, a
context), ``run`` makes one pass, ``work`` counts what a pass cannot do without, ``exact`` gives
the results of the same inputs in plain 64-bit torch.

The particles are Plummer spheres in virial N-body units with the accelerations and jerks of the
smooth model, the state a block-step integration holds.  The mixed path computes its forces in
FP32 pair arithmetic, so its results are handed on as FP32; the FP64 path's as FP64.  Block steps
are powers of two picked from the forces: on the mixed path a different rounding of one force can
turn one of them, so its runs return the particles and forces, not the steps.
"""
import math

import numpy as np
import torch

from paper_0709_4552_gb300 import nbody as nb

ETA = 0.01
DT_MIN = 2.0 ** -22
T0 = 0.5             # the particles' times lie at or before this ...
H = 2.0 ** -9        # ... and the forces are taken this much later
# arithmetic of one pair: 6 differences, r.r + eps^2 (6), r.v (5), 1/s (1), 1/s^2, m/s, m/s^3 (3),
# -3 (r.v)/s^2 (2), the potential's sum (1), the acceleration's (6), the jerk term and its sum (12)
FLOPS_PER_PAIR = 42


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # a full force evaluation of a small cluster: the latency of a predict + force call
        dict(name="mixed_small", kind="forces", precision="mixed", N=1024, n=1024, eps=2.0 ** -8, masses="equal"),
        # a caller's list of every particle of an odd-sized system of ordinary size
        dict(name="mixed_ragged", kind="forces", precision="mixed", N=20011, n=20011, eps=2.0 ** -9,
             masses="salpeter"),
        # an active block of a large system: the block-step force call of a production run
        dict(name="mixed_block", kind="forces", precision="mixed", N=1 << 20, n=4096, eps=2.0 ** -12,
             masses="equal"),
        # every particle of that system: the start of a run, shared steps, the benchmark's step
        dict(name="mixed_full", kind="forces", precision="mixed", N=1 << 20, n=1 << 20, eps=2.0 ** -12,
             masses="equal"),
        # the smallest blocks of that system, the other particles predicted inside the force call
        dict(name="mixed_at_block", kind="forces_at", precision="mixed", N=1 << 20, n=256, eps=2.0 ** -12,
             masses="equal"),
        # the FP64 path on a block of average size (0.20 N^0.81) of a large system
        dict(name="fp64_block", kind="forces", precision="fp64", N=196608, n=3883, eps=2.0 ** -10,
             masses="salpeter"),
        # FP64 forces in the caller's own memory, an odd block of an odd-sized system
        dict(name="noalloc_block", kind="noalloc", precision="fp64", N=30011, n=1001, eps=2.0 ** -9,
             masses="salpeter"),
        # FP64 integration with one shared step: every step a full force evaluation of a small system
        dict(name="fp64_shared_steps", kind="integrate", precision="fp64", N=1024, eps=2.0 ** -8, masses="equal",
             t_span=2.0 ** -4, dt_min=2.0 ** -10, dt_max=2.0 ** -10),
        # block-step integration of a small cluster, the loop chosen by the library
        dict(name="mixed_run_small", kind="integrate", precision="mixed", N=1024, eps=2.0 ** -8, masses="equal",
             t_span=2.0 ** -3, dt_min=DT_MIN, dt_max=2.0 ** -3),
        # block-step integration of a mid-sized cluster, the loop chosen by the library
        dict(name="mixed_run", kind="integrate", precision="mixed", N=12000, eps=2.0 ** -8, masses="equal",
             t_span=2.0 ** -5, dt_min=DT_MIN, dt_max=2.0 ** -5),
        # many independent clusters of uneven size integrated together
        dict(name="mixed_ensemble", kind="ensemble", precision="mixed", clusters=96, lo=256, hi=8192,
             masses="salpeter", t_span=2.0 ** -6),
        # the start of a run from a host snapshot: read in, first forces and steps, energy, written out
        dict(name="mixed_start", kind="start", precision="mixed", N=32768, eps=2.0 ** -8, masses="salpeter"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forces", "forces", "forces64", "forces_at", "noalloc", "integrate", "integrate64", "ensemble",
                       "start"])
    masses = rng.choice(["equal", "salpeter"])
    if kind == "forces":
        N = _log_int(rng, 1000, 600000)
        n = N if rng.random() < 0.4 else _log_int(rng, 1, N)
        return dict(kind="forces", precision="mixed", N=N, n=n, eps=2.0 ** -rng.randint(7, 13), masses=masses)
    if kind == "forces64":
        N = _log_int(rng, 1000, 200000)
        n = _log_int(rng, 1, min(N, 10 ** 9 // N))
        return dict(kind="forces", precision="fp64", N=N, n=n, eps=2.0 ** -rng.randint(7, 12), masses=masses)
    if kind == "forces_at":
        N = _log_int(rng, 20000, 1 << 20)
        return dict(kind="forces_at", precision="mixed", N=N, n=_log_int(rng, 1, 2000),
                    eps=2.0 ** -rng.randint(8, 13), masses=masses)
    if kind == "noalloc":
        N = _log_int(rng, 1000, 100000)
        return dict(kind="noalloc", precision="fp64", N=N, n=_log_int(rng, 1, min(N, 5 * 10 ** 8 // N)),
                    eps=2.0 ** -rng.randint(7, 12), masses=masses)
    if kind == "integrate":
        N = _log_int(rng, 256, 24000)
        t = 2.0 ** -rng.randint(5, 6)
        return dict(kind="integrate", precision="mixed", N=N, eps=2.0 ** -8, masses=masses, t_span=t, dt_min=DT_MIN,
                    dt_max=t)
    if kind == "integrate64":
        N = _log_int(rng, 256, 3000)
        return dict(kind="integrate", precision="fp64", N=N, eps=2.0 ** -8, masses=masses, t_span=2.0 ** -6,
                    dt_min=DT_MIN, dt_max=2.0 ** -6)
    if kind == "ensemble":
        return dict(kind="ensemble", precision="mixed", clusters=_log_int(rng, 8, 128), lo=256,
                    hi=_log_int(rng, 512, 8192), masses=masses, t_span=2.0 ** -rng.randint(6, 7))
    return dict(kind="start", precision="mixed", N=_log_int(rng, 1000, 60000), eps=2.0 ** -8, masses=masses)


# ------------------------------------------------------------------ the inputs
def _sphere(N, gen, masses):
    """m, x, v of a Plummer sphere of N particles (G = M = 1, E = -1/4) and the a and jerk of its
    smooth field, on the generator's device."""
    dev = gen.device

    def uniform(*shape):
        return torch.rand(*shape, generator=gen, device=dev, dtype=torch.float64)

    def isotropic(length):
        z = 1.0 - 2.0 * uniform(N)
        phi = 2.0 * math.pi * uniform(N)
        s = torch.sqrt(1.0 - z * z)
        return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], 1) * length[:, None]

    if masses == "salpeter":  # dN/dm ~ m^-2.35 between 0.1 and 100
        lo, hi = 0.1 ** -1.35, 100.0 ** -1.35
        m = (lo + uniform(N) * (hi - lo)) ** (-1.0 / 1.35)
        m = m / m.sum()
    else:
        m = torch.full((N,), 1.0 / N, device=dev, dtype=torch.float64)
    cut = (1.0 + 10.0 ** -2.0) ** -1.5  # the mass within ten scale lengths
    r = ((cut * uniform(N).clamp_min(1e-12)) ** (-2.0 / 3.0) - 1.0) ** -0.5
    x = isotropic(r)
    # speed / escape speed from g(q) = q^2 (1 - q^2)^3.5, by its tabulated distribution
    q = torch.linspace(0.0, 1.0, 4097, device=dev, dtype=torch.float64)
    cdf = torch.cumsum(q * q * (1.0 - q * q).clamp_min(0.0) ** 3.5, 0)
    cdf = cdf / cdf[-1]
    at = torch.searchsorted(cdf, uniform(N)).clamp(1, 4096)
    v = isotropic((q[at] - uniform(N) / 4096.0) * math.sqrt(2.0) * (1.0 + r * r) ** -0.25)
    x = x - (m[:, None] * x).sum(0)
    v = v - (m[:, None] * v).sum(0)
    b = 3.0 * math.pi / 16.0
    x = (x * b).contiguous()
    v = (v / math.sqrt(b)).contiguous()
    s2 = (x * x).sum(1, keepdim=True) + b * b
    a = -x * s2 ** -1.5
    jerk = -v * s2 ** -1.5 + 3.0 * (x * v).sum(1, keepdim=True) * x * s2 ** -2.5
    return m, x, v, a.contiguous(), jerk.contiguous()


def _state(case, seed):
    """The particles of a single-system case: m, x, v, a, jerk, t, dt (times in block steps)."""
    gen = torch.Generator("cuda").manual_seed(int(seed))
    N = case["N"]
    m, x, v, a, jerk = _sphere(N, gen, case["masses"])
    k = torch.randint(4, 10, (N,), generator=gen, device="cuda")
    dt = torch.ldexp(torch.ones(N, device="cuda", dtype=torch.float64), -k)
    half = torch.randint(0, 2, (N,), generator=gen, device="cuda")
    t = torch.where(k < 9, T0 - 0.5 * dt * half, torch.full_like(dt, T0))
    return gen, (m, x, v, a, jerk, t, dt)


def _block(case, gen):
    """n distinct particles, ascending."""
    N, n = case["N"], case["n"]
    if n == N:
        return torch.arange(N, device="cuda", dtype=torch.int32)
    return torch.randperm(N, generator=gen, device="cuda")[:n].sort().values.to(torch.int32)


def _pair_sums(m, x, v, eps, idx):
    """acc, jerk, pot of the particles idx from all others: the direct sum in 64 bits."""
    n, N = idx.shape[0], m.shape[0]
    acc = torch.empty(n, 3, device=x.device, dtype=torch.float64)
    jerk = torch.empty_like(acc)
    pot = torch.empty(n, device=x.device, dtype=torch.float64)
    xj, vj = x.t().contiguous(), v.t().contiguous()
    rows = max(1, min(n, (1 << 25) // N))
    for lo in range(0, n, rows):
        i = idx[lo:lo + rows].long()
        d = [xj[c][None, :] - xj[c][i][:, None] for c in range(3)]
        w = [vj[c][None, :] - vj[c][i][:, None] for c in range(3)]
        y = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps).rsqrt()
        y[torch.arange(i.shape[0], device=x.device), i] = 0.0
        rv = (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * (-3.0) * y * y
        g = y * m[None, :]
        pot[lo:lo + rows] = -g.sum(1)
        g = g * y * y
        for c in range(3):
            acc[lo:lo + rows, c] = (g * d[c]).sum(1)
            jerk[lo:lo + rows, c] = (g * (w[c] + rv * d[c])).sum(1)
    return acc, jerk, pot


def _predicted(s, t):
    m, x, v, a, jerk, ti, _ = s
    h = (t - ti)[:, None]
    return x + h * (v + h * (a / 2 + h * (jerk / 6))), v + h * (a + h * (jerk / 2))


def _first_steps(acc, jerk, dt_min, dt_max):
    """Largest power of two at most eta |a| / |j|, within the step range."""
    c = ETA * acc.norm(dim=1) / jerk.norm(dim=1)
    return torch.exp2(torch.floor(torch.log2(c))).clamp(dt_min, dt_max)


def _run_state(case, seed, N=None, gen=None, eps=None):
    """A particle set at t = 0 with its own forces and first steps, made without the library: what a
    snapshot of a running integration holds."""
    gen = gen or torch.Generator("cuda").manual_seed(int(seed))
    N = N or case["N"]
    m, x, v, _, _ = _sphere(N, gen, case["masses"])
    idx = torch.arange(N, device="cuda")
    acc, jerk, _ = _pair_sums(m, x, v, eps or case["eps"], idx)
    dt_max = case.get("dt_max", case["t_span"])
    dt = _first_steps(acc, jerk, case.get("dt_min", DT_MIN), dt_max)
    return m, x, v, acc.contiguous(), jerk.contiguous(), torch.zeros_like(m), dt


def _ensemble_sizes(case):
    """Sizes log-uniform in [lo, hi]; they belong to the case, the particles to the seed."""
    rng = np.random.default_rng(case["clusters"])
    u = rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["clusters"])
    return [int(s) for s in np.rint(np.exp(u))]


def _ensemble_state(case, seed):
    sizes = _ensemble_sizes(case)
    eps = [1.0 / (4.0 * s ** (1.0 / 3.0)) for s in sizes]
    gen = torch.Generator("cuda").manual_seed(int(seed))
    parts = [_run_state(case, seed, N=s, gen=gen, eps=e) for s, e in zip(sizes, eps)]
    return sizes, eps, [torch.cat([p[k] for p in parts]) for k in range(7)]


# -------------------------------------------------------- prepare and run a pass
def _empty(count, keys):
    shape = dict(m=(), x=(3,), v=(3,), a=(3,), jerk=(3,), pot=(), t=(), dt=())
    return {k: torch.empty((count,) + shape[k], device="cuda", dtype=torch.float64) for k in keys}


def prepare(case, seed):
    kind = case["kind"]
    prec = nb.NB_MIXED if case["precision"] == "mixed" else nb.NB_FP64
    stream = torch.cuda.current_stream()
    st = dict(case=case)
    if kind == "noalloc":
        gen, (m, x, v, *_) = _state(case, seed)
        n = case["n"]
        st.update(m=m, x=x, v=v, idx=_block(case, gen), out=_empty(n, ("a", "jerk", "pot")))
        return st
    if kind == "start":
        gen = torch.Generator("cuda").manual_seed(int(seed))
        st["host"] = [q.cpu().numpy() for q in _sphere(case["N"], gen, case["masses"])[:3]]
        st["sim"] = nb.NBody(case["N"], prec, 0, stream=stream)
        st["sim"].set_params(case["eps"], ETA, DT_MIN, 2.0 ** -3)
        return st
    if kind == "ensemble":
        sizes, eps, st["state"] = _ensemble_state(case, seed)
        off = np.concatenate([[0], np.cumsum(sizes)])
        st["sim"] = nb.Ensemble(off, np.array(eps), prec, 0, stream=stream)
        st["sim"].set_params(2.0 ** -8, ETA, DT_MIN, case["t_span"])
        st["out"] = _empty(int(off[-1]), ("x", "v", "a", "jerk", "pot"))
        return st
    sim = nb.NBody(case["N"], prec, 0, stream=stream)
    st["sim"] = sim
    if kind == "integrate":
        sim.set_params(case["eps"], ETA, case["dt_min"], case["dt_max"])
        st["state"] = _run_state(case, seed)
        keys = ("x", "v", "a", "jerk", "pot") + (("t", "dt") if prec == nb.NB_FP64 else ())
        st["out"] = _empty(case["N"], keys)
        return st
    sim.set_params(case["eps"], ETA, DT_MIN, 2.0 ** -3)
    gen, s = _state(case, seed)
    st["idx"] = _block(case, gen)
    sim.set_j_particles(0, *s)
    st["out"] = _empty(case["n"], ("a", "jerk", "pot"))
    return st


def _handed_on(case, out):
    """The results in the precision of the path that computed them."""
    return {k: q.float() for k, q in out.items()} if case["precision"] == "mixed" else out


def run(st):
    case = st["case"]
    kind = case["kind"]
    out = st.get("out")
    if kind == "noalloc":
        nb.nb_forces_fp64_noalloc(st["m"], st["x"], st["v"], case["eps"], st["idx"], out["a"], out["jerk"],
                                  out["pot"], stream=torch.cuda.current_stream())
        return out
    sim = st["sim"]
    if kind == "forces":
        sim.predict(T0 + H)
        sim.compute_forces(st["idx"], out["a"], out["jerk"], out["pot"])
        return _handed_on(case, out)
    if kind == "forces_at":
        sim.compute_forces_at(T0 + H, st["idx"], out["a"], out["jerk"], out["pot"])
        return _handed_on(case, out)
    if kind == "integrate":
        sim.set_j_particles(0, *st["state"])
        sim.integrate(case["t_span"], loop=nb.NB_LOOP_AUTO)
        sim.get_particles(0, case["N"], out)
        return _handed_on(case, out)
    if kind == "ensemble":
        sim.set_j_particles(0, *st["state"])
        nb.nb_ensemble_integrate(sim.ctx, case["t_span"])
        sim.get_particles(0, out["x"].shape[0], out)
        return _handed_on(case, out)
    sim.set_j_particles(0, *st["host"])
    sim.initial_forces_and_dt()
    kinetic, potential = sim.energy()
    p = sim.get_particles(0, case["N"])
    return {"kinetic": kinetic, "potential": np.float32(potential), "x": p["x"], "v": p["v"],
            "a": p["a"].astype(np.float32), "jerk": p["jerk"].astype(np.float32), "pot": p["pot"].astype(np.float32)}


def _pairs(case):
    """Pair interactions of a pass; for a block-step run the corrections a particle needs per time unit
    are those of Plummer spheres at eta = 0.01 (about 260 at N = 1024, growing slowly with N)."""
    kind = case["kind"]
    if kind == "ensemble":
        mean = (case["lo"] * case["hi"]) ** 0.5
        return case["clusters"] * 260.0 * (mean / 1024.0) ** 0.15 * mean * mean * case["t_span"]
    N = case["N"]
    if kind == "integrate":
        per_unit = 1.0 / case["dt_max"] if case["dt_min"] == case["dt_max"] else 260.0 * (N / 1024.0) ** 0.15
        return per_unit * case["t_span"] * N * N
    if kind == "start":
        return 2.0 * N * N
    return float(case["n"]) * N


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        N = case["clusters"] * (case["lo"] * case["hi"]) ** 0.5
    else:
        N = case["N"]
    if kind in ("forces", "forces_at"):
        moved = 8.0 * 14 * N + (4 + 56.0) * case["n"]   # the state in; the list in, the forces out
    elif kind == "noalloc":
        moved = 56.0 * N + (4 + 56.0) * case["n"]
    elif kind == "start":
        moved = 56.0 * N + 128.0 * N
    else:
        moved = 8.0 * 15 * N + 8.0 * 13 * N
    return {"bytes": moved, "flops": FLOPS_PER_PAIR * _pairs(case)}


# ------------------------------------------------------------------ in 64 bits
def _integrated(s, eps, t_end, dt_min, dt_max):
    """Hermite block steps to t_end in plain torch: x, v, a, jerk, pot, t, dt."""
    m, x, v, a, jerk, t, dt = [q.clone() for q in s]
    pot = torch.zeros_like(m)
    while True:
        due = t + dt
        now = float(due.min())
        if now > t_end:
            return dict(x=x, v=v, a=a, jerk=jerk, pot=pot, t=t, dt=dt)
        i = torch.nonzero(due == now).flatten()
        xp, vp = _predicted((m, x, v, a, jerk, t, dt), now)
        a1, j1, p1 = _pair_sums(m, xp, vp, eps, i)
        h = (now - t[i])[:, None]
        a0, j0 = a[i], jerk[i]
        a2 = (-6 * (a0 - a1) - h * (4 * j0 + 2 * j1)) / h ** 2
        a3 = (12 * (a0 - a1) + 6 * h * (j0 + j1)) / h ** 3
        x[i] = xp[i] + a2 * h ** 4 / 24 + a3 * h ** 5 / 120
        v[i] = vp[i] + a2 * h ** 3 / 6 + a3 * h ** 4 / 24
        a[i], jerk[i], pot[i] = a1, j1, p1
        na, nj, n2, n3 = a1.norm(dim=1), j1.norm(dim=1), (a2 + a3 * h).norm(dim=1), a3.norm(dim=1)
        c = torch.sqrt(ETA * (na * n2 + nj * nj) / (nj * n3 + n2 * n2))
        c = torch.exp2(torch.floor(torch.log2(c))).clamp(dt_min, dt_max)
        old = dt[i]
        grow = (c >= 2 * old) & (2 * old <= dt_max) & (torch.remainder(torch.full_like(old, now), 2 * old) == 0)
        dt[i] = torch.where(c < old, c, torch.where(grow, 2 * old, old))
        t[i] = now


def exact(case, seed):
    if _pairs(case) > 6e9:  # beyond what plain torch sums in a few seconds
        return None
    kind = case["kind"]
    if kind in ("forces", "forces_at"):
        gen, s = _state(case, seed)
        xp, vp = _predicted(s, T0 + H)
        acc, jerk, pot = _pair_sums(s[0], xp, vp, case["eps"], _block(case, gen))
        return dict(a=acc, jerk=jerk, pot=pot)
    if kind == "noalloc":
        gen, (m, x, v, *_) = _state(case, seed)
        acc, jerk, pot = _pair_sums(m, x, v, case["eps"], _block(case, gen))
        return dict(a=acc, jerk=jerk, pot=pot)
    if kind == "integrate":
        end = _integrated(_run_state(case, seed), case["eps"], case["t_span"], case["dt_min"], case["dt_max"])
        return {k: end[k] for k in ("x", "v", "a", "jerk", "pot") + (("t", "dt") if case["precision"] == "fp64" else ())}
    if kind == "ensemble":
        if case["clusters"] > 128:  # one Python loop per cluster
            return None
        sizes, eps, s = _ensemble_state(case, seed)
        ends, lo = [], 0
        for n, e in zip(sizes, eps):
            ends.append(_integrated([q[lo:lo + n] for q in s], e, case["t_span"], DT_MIN, case["t_span"]))
            lo += n
        return {k: torch.cat([e[k] for e in ends]) for k in ("x", "v", "a", "jerk", "pot")}
    gen = torch.Generator("cuda").manual_seed(int(seed))
    m, x, v = _sphere(case["N"], gen, case["masses"])[:3]
    acc, jerk, pot = _pair_sums(m, x, v, case["eps"], torch.arange(case["N"], device="cuda"))
    return {"kinetic": float(0.5 * (m * (v * v).sum(1)).sum()), "potential": float(0.5 * (m * pot).sum()), "x": x,
            "v": v, "a": acc, "jerk": jerk, "pot": pot}
