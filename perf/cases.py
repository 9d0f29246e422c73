"""What the performance of this library is measured on: its public entry points, as programs that use it call them.

Five kinds of case:

``force``     ``Simulation.predict`` and ``Simulation.force`` on a list of active particles: the call of a host
              program that keeps its own scheduler (one particle of a small block, the mean block of a
              65536-particle run, a large partial block, all particles of a shared step).
``step``      ``Simulation.set_state``, ``step``, ``get_state``: a run resumed from a saved state and taken some
              block steps further, from systems that are all latency to systems whose large blocks count.
``ensemble``  ``Ensemble``, ``run``, ``get_state``: many independent clusters of a seeded size distribution from
              start to end, the set-up included (every batch of clusters pays for it).
``gradient``  ``rollout_loss`` or ``rollout`` under torch autograd: forward and reverse of a shared-step run.
``energy``    ``Simulation.energy``: the conserved-quantity check after a run, in FP64 or with the double-single
              potential.

Inputs are seeded Plummer spheres in Henon units with equal masses, or with masses drawn from a power-law spectrum;
softening 1/256 (1e-3 for the million-particle shared step, 1/128 for gradients).  ``exact`` restates the method in
plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_astro_ph_0702058_gb300 import Ensemble, Simulation
from paper_astro_ph_0702058_gb300.autodiff import rollout, rollout_loss
from synthetic import active_subset, ensemble_sizes, plummer_sphere

EPS = 1.0 / 256
LMAX = 26  # dt_min = 2^-26


def listed():
    return [
        # one due particle of a 65536-particle system: the call is all latency
        dict(name="force_one", kind="force", n=65536, rows=1, mode="plain", eps=EPS, masses="equal"),
        # the mean block of a 65536-particle run
        dict(name="force_mean_block", kind="force", n=65536, rows=1594, mode="comp", eps=EPS, masses="equal"),
        # a large partial block of an odd-sized system with a mass spectrum
        dict(name="force_large_block", kind="force", n=100003, rows=40001, mode="plain", eps=EPS, masses="spectrum"),
        # the full force of a shared step at 2^20 particles, the benchmark's shape
        dict(name="force_all", kind="force", n=1 << 20, rows=1 << 20, mode="comp", eps=1e-3, masses="equal"),
        # a full force in the double-single precision tier
        dict(name="force_all_ds", kind="force", n=16384, rows=16384, mode="ds", eps=EPS, masses="equal"),
        # a small system's run of about 400 block steps
        dict(name="step_small", kind="step", n=1024, span=8, mode="plain", eta=0.01, masses="equal"),
        # an odd-sized system with a mass spectrum
        dict(name="step_odd", kind="step", n=5001, span=2, mode="comp", eta=0.02, masses="spectrum"),
        # a 65536-particle run: many small blocks beside a few large ones that hold most pairs
        dict(name="step_large", kind="step", n=65536, span=1, mode="comp", eta=0.02, masses="equal"),
        # 128 clusters of 256 to 8191 particles, from start to end
        dict(name="ensemble", kind="ensemble", clusters=128, sizes=4, span=1, mode="comp", eta=0.02),
        # the loss and gradient of a 4096-particle shared-step run
        dict(name="gradient_loss", kind="gradient", n=4096, steps=64, mode="plain", loss="fixed"),
        # a smaller run inside a larger differentiable program
        dict(name="gradient_general", kind="gradient", n=1500, steps=32, mode="comp", loss="general"),
        # the energy check after a 65536-particle run
        dict(name="energy", kind="energy", n=65536, double_single=False, masses="equal"),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]; one in three is a multiple of 1024 where there is one."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if n >= 2048 and rng.random() < 1 / 3:
        n = n // 1024 * 1024
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "step", "step", "ensemble", "gradient", "energy"])
    masses = rng.choice(["equal", "spectrum"])
    if kind == "force":
        mode = rng.choice(["plain", "plain", "comp", "comp", "ds"])
        n = _size(rng, 500, 30000 if mode == "ds" else 400000)
        rows = n if rng.random() < 1 / 3 else _size(rng, 1, n)
        return dict(kind=kind, n=n, rows=rows, mode=mode, eps=rng.choice([EPS, 1e-3]), masses=masses)
    if kind == "step":
        mode = rng.choice(["plain", "comp", "comp", "ds"])
        n = _size(rng, 256, 2048 if mode == "ds" else 65536)
        span = rng.choice([2, 4, 8] if n <= 4096 else [1, 2])
        return dict(kind=kind, n=n, span=span, mode=mode, eta=rng.choice([0.01, 0.02]), masses=masses)
    if kind == "ensemble":
        return dict(kind=kind, clusters=_size(rng, 4, 256), sizes=rng.randint(1, 999), span=rng.choice([1, 2]),
                    mode=rng.choice(["plain", "comp"]), eta=0.02)
    if kind == "gradient":
        return dict(kind=kind, n=_size(rng, 64, 8192), steps=rng.randint(8, 64), mode=rng.choice(["plain", "comp"]),
                    loss=rng.choice(["fixed", "general"]))
    ds = rng.random() < 0.5
    return dict(kind=kind, n=_size(rng, 1000, 262144 if ds else 90000), double_single=ds, masses=masses)


# ---- inputs ----

def _particles(n, seed, masses):
    m, x, v = plummer_sphere(n, seed)
    if masses == "spectrum":  # dN/dm ~ m^-2.35 over a factor of 100, normalised to unit total mass
        u = np.random.default_rng(seed).random(n)
        m = (1.0 + u * (100.0 ** -1.35 - 1.0)) ** (-1.0 / 1.35)
        m = m / m.sum()
    return m, x, v


def _t_force(case):
    """The time predicted to before a force: 2^-10, the shared step of the full-force run."""
    return 2.0 ** -10


def _span(case):
    return case["span"] / 64.0  # in units of dt_max = 1/64


def _clusters(case, seed):
    sizes = ensemble_sizes(case["clusters"], case["sizes"])  # log-uniform in [256, 8192)
    parts = [plummer_sphere(int(n), 1000 * seed + c) for c, n in enumerate(sizes)]
    return sizes, *(np.concatenate([p[k] for p in parts]) for k in range(3))


def _rollout_inputs(case, seed):
    m, x, v = plummer_sphere(case["n"], seed)
    g = np.random.default_rng(seed)
    return m, x, v, g.standard_normal((case["n"], 3)), g.standard_normal((case["n"], 3))


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        sizes, m, x, v = _clusters(case, seed)
        return dict(case=case, sizes=sizes, m=_dev(m), x=_dev(x), v=_dev(v), out=[_empty(len(m), 3) for _ in range(4)])
    if kind == "gradient":
        m, x, v, gx, gv = (_dev(a) for a in _rollout_inputs(case, seed))
        for a in (m, x, v):
            a.requires_grad_(True)
        return dict(case=case, m=m, x=x, v=v, gx=gx, gv=gv)
    n = case["n"]
    m, x, v = _particles(n, seed, case["masses"])
    if kind == "energy":
        return dict(case=case, sim=Simulation(m, x, v, EPS ** 2))
    if kind == "force":
        sim = Simulation(m, x, v, case["eps"] ** 2, mode=case["mode"], lmax=LMAX)
        rows = case["rows"]
        return dict(case=case, sim=sim, rows=_dev(active_subset(n, rows, seed)), acc=_empty(rows, 3),
                    jerk=_empty(rows, 3), pot=_empty(rows))
    sim = Simulation(m, x, v, EPS ** 2, mode=case["mode"], eta=case["eta"], lmax=LMAX)
    start = {k: _empty(n, 3) for k in ("x", "v", "a", "k")}
    start["t_tick"] = torch.zeros(n, dtype=torch.int64, device="cuda")
    start["level"] = torch.zeros(n, dtype=torch.int8, device="cuda")
    sim.get_state(**start)
    return dict(case=case, sim=sim, start=start, out={k: torch.empty_like(t) for k, t in start.items()})


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "force":
        sim = state["sim"]
        sim.predict(_t_force(case))
        sim.force(state["rows"], acc=state["acc"], jerk=state["jerk"], pot=state["pot"])
        return state["acc"], state["jerk"], state["pot"]
    if kind == "step":
        sim, out = state["sim"], state["out"]
        sim.set_state(**state["start"])
        sim.step(_span(case))
        sim.get_state(**out)
        return [out[k] for k in ("x", "v", "a", "k")]
    if kind == "ensemble":
        with Ensemble(state["sizes"], state["m"], state["x"], state["v"], EPS ** 2, eta=case["eta"],
                      mode=case["mode"]) as ens:
            ens.run(_span(case))
            x, v, a, k = state["out"]
            ens.get_state(x=x, v=v, a=a, k=k)
        return x, v, a, k
    if kind == "gradient":
        m, x, v = state["m"], state["x"], state["v"]
        if case["loss"] == "fixed":
            loss = rollout_loss(x, v, m, steps=case["steps"], mode=case["mode"])
            return (loss.detach(),) + torch.autograd.grad(loss, (x, v, m))
        xT, vT = rollout(x, v, m, steps=case["steps"], mode=case["mode"])
        return (xT.detach(), vT.detach()) + torch.autograd.grad((xT, vT), (x, v, m), (state["gx"], state["gv"]))
    return np.array(state["sim"].energy(ds_potential=case["double_single"]))


# ---- the least work of a pass ----

# Floating-point operations of an unordered pair (differences 6, r^2 6, dx.dv 5, r^-1, r^-2, r^-3, 3 (dx.dv) r^-2 2,
# dv - w dx 6) and of each particle that receives its force (m r^-3 1, acceleration 6, jerk 6, potential 2).
_PAIR, _RECEIVE = 28, 15
# The same in double-single arithmetic: 11 sums, 12 products and the reciprocal square root, and 7 products and sums,
# at about 10 operations each.
_PAIR_DS, _RECEIVE_DS = 250, 140
# The gradient of a pair: the force's geometry and the products of the two upstream vectors with it.
_PAIR_VJP = 80


def _force_flops(n, rows, mode):
    both = rows * (rows - 1) / 2  # pairs that give both members their force
    one = rows * (n - rows)
    pair, receive = (_PAIR_DS, _RECEIVE_DS) if mode == "ds" else (_PAIR + (6 if mode == "comp" else 0), _RECEIVE)
    return (both + one) * pair + (2 * both + one) * receive


def _run_flops(n, span, eta, mode):
    """A run: about 172 (n / 1024)^0.14 (0.02 / eta)^0.5 steps per particle and unit time (measured: 244 at n = 1024
    and eta = 0.01, 312 at n = 65536 and eta = 0.02), most pairs in large blocks."""
    steps = n * 172 * (n / 1024) ** 0.14 * math.sqrt(0.02 / eta) * span
    return steps / n * _force_flops(n, n, mode)


def work(case):
    kind = case["kind"]
    if kind == "force":  # the state in (t, x, v, a, k, m), the listed rows' forces out
        return dict(bytes=112.0 * case["n"] + 60.0 * case["rows"], flops=_force_flops(case["n"], case["rows"], case["mode"]))
    if kind == "step":  # the state in and out
        return dict(bytes=2 * 105.0 * case["n"], flops=_run_flops(case["n"], _span(case), case["eta"], case["mode"]))
    if kind == "ensemble":
        # sizes are log-uniform in [256, 8192): mean 2290 particles, mean square 9.7e6
        flops = case["clusters"] * _run_flops(3100, _span(case), case["eta"], case["mode"])
        return dict(bytes=2 * 105.0 * 2290 * case["clusters"], flops=flops)
    if kind == "gradient":
        n, steps = case["n"], case["steps"]
        once = _force_flops(n, n, case["mode"])
        return dict(bytes=56.0 * n * 2, flops=(steps + 1) * (once + n * (n - 1) / 2 * _PAIR_VJP))
    n = case["n"]
    pair = 100 if case["double_single"] else 11  # differences, r^2, reciprocal square root, product and sum
    return dict(bytes=56.0 * n, flops=n * (n - 1) / 2 * pair)


def tolerance(case):
    """About four times the largest distance from ``exact`` seen over these ranges.  Plain mode: its FP32 positions
    resolve a separation r to 2^-24 |x| / r, which close pairs feel more at the smaller softening."""
    kind, mode = case["kind"], case.get("mode")
    if kind == "force":
        if mode == "plain":
            return dict(rel=1.5e-5, max=5e-4) if case["eps"] == EPS else dict(rel=6e-5, max=1.5e-3)
        return dict(rel=1e-6, max=1.5e-5) if mode == "comp" else dict(rel=3e-12, max=3e-10)
    if kind in ("step", "ensemble"):
        return {"plain": dict(rel=2e-5, max=1.6e-3), "comp": dict(rel=4e-6, max=4e-5), "ds": dict(rel=1e-12, max=1e-11)}[mode]
    if kind == "gradient":
        return dict(rel=1.5e-5, max=1e-4)
    return dict(rel=1e-13, max=1e-13) if case["double_single"] else dict(rel=1e-14, max=1e-14)


# ---- the same outputs in plain FP64 torch ----

def _sums(xi, vi, x, v, m, eps2):
    """acc, jerk and pot of particles xi, vi over all of x, v, m; a particle's own term is zero where eps2 > 0
    (but for the potential, whose own term -m / eps is left to the caller)."""
    dx, dv = x[None] - xi[:, None], v[None] - vi[:, None]
    y = torch.rsqrt((dx * dx).sum(2) + eps2)
    y2 = y * y
    my = m * y
    w = my * y2
    q = 3.0 * (dx * dv).sum(2) * y2
    acc = (w[:, :, None] * dx).sum(1)
    return acc, (w[:, :, None] * dv).sum(1) - ((w * q)[:, :, None] * dx).sum(1), -my.sum(1)


def _force64(idx, x, v, m, eps2):
    out = [[], [], []]
    step = max(1, (1 << 24) // x.shape[0])
    for part in idx.split(step):
        for o, s in zip(out, _sums(x[part], v[part], x, v, m, eps2)):
            o.append(s)
    acc, jerk, pot = (torch.cat(o) for o in out)
    return acc, jerk, pot + m[idx] / math.sqrt(eps2)


def _floor_level(dt, lmin, lmax):
    return (1 - torch.frexp(dt)[1]).clamp(lmin, lmax).long()


def _norm(u):
    return u.square().sum(1).sqrt()


def _run64(x, v, m, eps2, eta, span, lmin=6, lmax=LMAX):
    """Block steps of the Hermite scheme from t = 0 to span (a multiple of 2^-lmin)."""
    n = x.shape[0]
    x, v = x.clone(), v.clone()
    a, k, _ = _force64(torch.arange(n, device=x.device), x, v, m, eps2)
    t = torch.zeros(n, dtype=torch.int64, device=x.device)
    level = _floor_level(eta * _norm(a) / _norm(k), lmin, lmax)
    end = int(span * 2 ** lmax)
    while True:
        due = t + (1 << (lmax - level))
        now = int(due.min())
        if now > end:
            return x, v, a, k
        dt = ((now - t).double() * 2.0 ** -lmax)[:, None]
        xp = x + v * dt + a * dt ** 2 / 2 + k * dt ** 3 / 6
        vp = v + a * dt + k * dt ** 2 / 2
        i = (due == now).nonzero()[:, 0]
        an, kn, _ = _force64(i, xp, vp, m, eps2)
        h, da = dt[i], a[i] - an
        a2 = -6 * da / h ** 2 - (4 * k[i] + 2 * kn) / h
        a3 = 12 * da / h ** 3 + 6 * (k[i] + kn) / h ** 2
        x[i] = xp[i] + a2 * h ** 4 / 24 + a3 * h ** 5 / 120
        v[i] = vp[i] + a2 * h ** 3 / 6 + a3 * h ** 4 / 24
        a[i], k[i], t[i] = an, kn, now
        e2 = a2 + a3 * h
        na, nk, n2, n3 = _norm(an), _norm(kn), _norm(e2), _norm(a3)
        crit = _floor_level((eta * (na * n2 + nk * nk) / (nk * n3 + n2 * n2)).sqrt(), lmin, lmax)
        old = level[i]
        grow = (crit < old) & (old > lmin) & (now % (2 << (lmax - old)) == 0)
        level[i] = torch.where(crit >= old, crit, torch.where(grow, old - 1, old))


def _shared64(x, v, m, eps2, dt, steps):
    """Shared steps of dt, differentiable, the pair terms of each step formed again in the backward pass."""
    from torch.utils.checkpoint import checkpoint

    def force(x, v, m):
        return _sums(x, v, x, v, m, eps2)[:2]

    def step(x, v, a, k, m):
        xp = x + v * dt + a * dt ** 2 / 2 + k * dt ** 3 / 6
        vp = v + a * dt + k * dt ** 2 / 2
        an, kn = force(xp, vp, m)
        a2 = -6 * (a - an) / dt ** 2 - (4 * k + 2 * kn) / dt
        a3 = 12 * (a - an) / dt ** 3 + 6 * (k + kn) / dt ** 2
        return xp + a2 * dt ** 4 / 24 + a3 * dt ** 5 / 120, vp + a2 * dt ** 3 / 6 + a3 * dt ** 4 / 24, an, kn

    a, k = checkpoint(force, x, v, m, use_reentrant=False)
    for _ in range(steps):
        x, v, a, k = checkpoint(step, x, v, a, k, m, use_reentrant=False)
    return x, v


def _potential64(x, m, eps2):
    """sum_i<j -m_i m_j / (r_ij^2 + eps2)^1/2."""
    total = torch.zeros((), dtype=torch.float64, device=x.device)
    step = max(1, (1 << 25) // x.shape[0])
    for b in range(0, x.shape[0], step):
        d = x[b:b + step]
        r2 = eps2 + sum((x[None, :, c] - d[:, None, c]).square() for c in range(3))
        total -= (m[b:b + step, None] * m * torch.rsqrt(r2)).sum()
    return 0.5 * (total + (m * m).sum() / math.sqrt(eps2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        if case["clusters"] * case["span"] > 80:
            return None
        sizes, m, x, v = _clusters(case, seed)
        m, x, v = _dev(m), _dev(x), _dev(v)
        parts = [_run64(xc, vc, mc, EPS ** 2, case["eta"], _span(case)) for xc, vc, mc in
                 zip(*(u.split([int(n) for n in sizes]) for u in (x, v, m)))]
        return [torch.cat([p[k] for p in parts]) for k in range(4)]
    if kind == "gradient":
        m, x, v, gx, gv = (_dev(a) for a in _rollout_inputs(case, seed))
        for a in (m, x, v):
            a.requires_grad_(True)
        eps2 = (1.0 / 128) ** 2
        xT, vT = _shared64(x, v, m, eps2, 2.0 ** -9, case["steps"])
        if case["loss"] == "fixed":
            loss = (xT * xT).sum() + 0.5 * ((m * _sums(xT, vT, xT, vT, m, eps2)[2]).sum() + (m * m).sum() / math.sqrt(eps2))
            return (loss.detach(),) + torch.autograd.grad(loss, (x, v, m))
        return (xT.detach(), vT.detach()) + torch.autograd.grad((xT, vT), (x, v, m), (gx, gv))
    n = case["n"]
    m, x, v = (_dev(a) for a in _particles(n, seed, case["masses"]))
    if kind == "energy":
        return torch.stack([0.5 * (m * v.square().sum(1)).sum(), _potential64(x, m, EPS ** 2)])
    if kind == "step":
        steps = 172 * (n / 1024) ** 0.14 * math.sqrt(0.02 / case["eta"]) * _span(case)
        if n * n * steps > 4e10:
            return None
        return _run64(x, v, m, EPS ** 2, case["eta"], _span(case))
    if n > 150000:
        return None
    a, k, _ = _force64(torch.arange(n, device=x.device), x, v, m, case["eps"] ** 2)
    t = _t_force(case)
    x, v = x + v * t + a * t ** 2 / 2 + k * t ** 3 / 6, v + a * t + k * t ** 2 / 2
    return _force64(_dev(active_subset(n, case["rows"], seed)).long(), x, v, m, case["eps"] ** 2)
