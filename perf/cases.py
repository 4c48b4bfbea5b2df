"""Measured cases of the hybrid symplectic N-body step, through its public calls.

A pass is what a run does between two of its outputs: `Simulation.step(n)`, then
`Simulation.state()` of every system (ids, masses, positions, velocities, radii on
the host), on a simulation created beforehand; the simulation goes on from where the
last pass left it, as a run does.  Two more cases are the diagnostic a run logs
beside its outputs: energy, angular momentum and momentum, of a simulation and of
caller-owned device arrays.

The systems are the seeded synthetic workloads of `opal_ic`.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import opal_ic as ic
from paper_2601_19654_gb300 import opal

MIXED, FP64 = 1, 0
RATIONAL, QUINTIC = 0, 1


def listed():
    return [
        # A terrestrial-planet system of ten bodies: the smallest run, all latency.
        {"name": "few_bodies", "kind": "tiny", "n": 10, "precision": MIXED, "changeover": RATIONAL, "steps": 20},
        # 1000 planetesimals inside Jupiter with star collisions and ejections on, as a
        # formation run has them (ejections checked every 200 yr).
        {"name": "planetesimals", "kind": "planetesimals", "n": 1000, "precision": MIXED, "changeover": RATIONAL,
         "removals": True, "steps": 10},
        # The same in the FP64 form: a convergence check of the mixed form.
        {"name": "planetesimals_fp64", "kind": "planetesimals", "n": 1000, "precision": FP64,
         "changeover": RATIONAL, "removals": False, "steps": 10},
        # A disk whose count is no multiple of any tile, with the quintic changeover.
        {"name": "disk_5003_quintic", "kind": "disk", "n": 5003, "precision": MIXED, "changeover": QUINTIC,
         "steps": 5},
        # The headline workload: 16384 equal bodies, mixed form.
        {"name": "disk_16384", "kind": "disk", "n": 16384, "precision": MIXED, "changeover": RATIONAL, "steps": 5},
        # And its FP64 form.
        {"name": "disk_16384_fp64", "kind": "disk", "n": 16384, "precision": FP64, "changeover": RATIONAL,
         "steps": 1},
        # The production regime: embryos and Jupiter in a swarm of massless planetesimals.
        {"name": "embryos_262144", "kind": "embryos", "n_big": 1024, "n_small": 262144, "precision": MIXED,
         "changeover": RATIONAL, "steps": 5},
        # A smaller, ragged swarm in the FP64 form.
        {"name": "embryos_40001_fp64", "kind": "embryos", "n_big": 301, "n_small": 40001, "precision": FP64,
         "changeover": RATIONAL, "steps": 5},
        # A statistical ensemble: 256 independent systems of 64 to 4096 bodies stepped together.
        {"name": "ensemble_256", "kind": "ensemble", "systems": 256, "lo": 64, "hi": 4096, "precision": MIXED,
         "changeover": RATIONAL, "steps": 5},
        # The encounter-heavy run: 131072 bodies with inflated radii, Jupiter and Saturn.
        {"name": "heavy_131072", "kind": "heavy", "n": 131072, "precision": MIXED, "changeover": RATIONAL,
         "steps": 2},
        # The conserved quantities of the headline system, logged beside its outputs.
        {"name": "energy_16384", "kind": "energy", "n": 16384},
        # The same of device arrays, at the largest count the allocation-free call takes.
        {"name": "energy_device_131072", "kind": "energy_device", "n": 131072},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("tiny", "planetesimals", "disk", "disk", "embryos", "ensemble", "heavy", "energy",
                       "energy_device"))
    if kind == "energy":
        return {"kind": kind, "n": _log_int(rng, 10, 16384)}
    if kind == "energy_device":
        return {"kind": kind, "n": _log_int(rng, 100, 131072)}
    c = {"kind": kind, "precision": rng.choice((MIXED, MIXED, FP64)), "changeover": rng.choice((RATIONAL, QUINTIC))}
    if kind == "tiny":
        return {**c, "n": _log_int(rng, 2, 64), "steps": rng.randint(5, 20)}
    if kind == "planetesimals":
        return {**c, "n": _log_int(rng, 64, 4000), "removals": rng.random() < 0.5, "steps": rng.randint(2, 10)}
    if kind == "disk":
        return {**c, "n": _log_int(rng, 256, 16384), "steps": rng.randint(1, 3)}
    if kind == "embryos":
        return {**c, "n_big": _log_int(rng, 16, 1024), "n_small": _log_int(rng, 500, 262144), "steps": rng.randint(1, 2)}
    if kind == "ensemble":
        lo = _log_int(rng, 8, 256)
        return {**c, "systems": _log_int(rng, 4, 256), "lo": lo, "hi": _log_int(rng, lo + 1, 2048), "steps": 1}
    return {**c, "precision": MIXED, "n": _log_int(rng, 8192, 100000), "steps": 1}


def _seed(seed):
    return int(seed) % (1 << 31)


def _systems(case, seed):
    """The case's systems: a list of `opal_ic.System`, of this seed."""
    kind, s = case["kind"], _seed(seed)
    if kind == "tiny":
        return [ic.tiny(s, case["n"])]
    if kind == "planetesimals":
        return [ic.planetesimals_jupiter(s, case["n"])]
    if kind in ("disk", "energy"):
        return [ic.equal_mass_disk(s, case["n"])]
    if kind == "embryos":
        return [ic.embryos_planetesimals(s, case["n_big"], case["n_small"])]
    if kind == "ensemble":
        # the counts of the repository's ensemble, the bodies of this seed
        sizes = ic.ensemble_sizes(0, case["systems"], case["lo"], case["hi"])
        return [ic.tiny(1000 * s + k, int(n)) for k, n in enumerate(sizes)]
    if kind == "heavy":
        return [ic.encounter_heavy(s, case["n"])]
    return [ic.equal_mass_disk(s, case["n"])]   # energy_device


def prepare(case, seed):
    systems = _systems(case, seed)
    if case["kind"] == "energy_device":
        t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (systems[0].m, systems[0].x, systems[0].v)]
        return {"kind": case["kind"], "n": systems[0].n, "G": systems[0].G, "M0": systems[0].M0, "arrays": t,
                "out": torch.zeros(7, dtype=torch.float64, device="cuda")}
    options = {}
    if case["kind"] != "energy":
        options = {"precision": case["precision"], "changeover": case["changeover"]}
    if case.get("removals"):
        # the Sun's radius; ejections beyond 400 au, checked every 200 yr
        options.update(r_star=0.00465, r_eject=400.0, eject_every=int(round(200.0 * ic.YEAR / systems[0].dt)))
    if case["kind"] == "ensemble":
        sim = opal.Simulation.ensemble(systems, **options)
    else:
        sim = opal.Simulation.from_system(systems[0], **options)
    return {"kind": case["kind"], "sim": sim, "counts": [s.n for s in systems], "steps": case.get("steps", 0)}


def _in_place(st, n):
    """A system's output by body id: bodies merged away or removed have id -1 and zeros."""
    if st["ids"].size == n:
        return st
    out = {"ids": np.full(n, -1, np.int64), "m": np.zeros(n), "x": np.zeros((n, 3)), "v": np.zeros((n, 3)),
           "R": np.zeros(n)}
    for key in out:
        out[key][st["ids"]] = st[key]
    return out


def run(state):
    if state["kind"] == "energy_device":
        m, x, v = state["arrays"]
        opal.energy_momentum_noalloc(state["n"], state["G"], state["M0"], m.data_ptr(), x.data_ptr(), v.data_ptr(),
                                     state["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"E": state["out"][0], "L": state["out"][1:4], "P": state["out"][4:7]}
    sim = state["sim"]
    if state["kind"] == "energy":
        E, L, P, lost = sim.energy()
        return {"E": np.float64(E), "L": L, "P": P, "E_lost": np.float64(lost)}
    sim.step(state["steps"])
    parts = [_in_place(sim.state(k), n) for k, n in enumerate(state["counts"])]
    if len(parts) == 1:
        return parts[0]
    return {key: np.concatenate([p[key] for p in parts]) for key in ("ids", "m", "x", "v", "R")}


def _counts(case):
    """(bodies, directed pairs with a big source) of the case."""
    kind = case["kind"]
    if kind == "planetesimals":
        n = case["n"] + 1
        return n, n * (n - 1)
    if kind == "embryos":
        n, nb = case["n_big"] + case["n_small"], case["n_big"]
        return n, n * nb - nb
    if kind == "heavy":
        n = case["n"] + 2
        return n, n * (n - 1)
    if kind == "ensemble":
        # the mean of a log-uniform count and of its square
        lo, hi, k = case["lo"], case["hi"] + 1, case["systems"]
        w = math.log(hi / lo)
        return int(k * (hi - lo) / w), int(k * (hi * hi - lo * lo) / (2 * w))
    return case["n"], case["n"] * (case["n"] - 1)


def work(case):
    n, pairs = _counts(case)
    if case["kind"] in ("energy", "energy_device"):
        # each unordered pair: 3 differences, the squared distance, 1/r, m m / r and the sum
        return {"bytes": 56.0 * n + 56.0, "flops": 12.0 * (pairs // 2)}
    # a step: 18 flops a directed pair of the kick (the difference, r^2, 1/r, m / r^3 and the
    # sum) and about 600 a body for the drift; bytes: positions and velocities in and out
    # once a step, masses, radii and accelerations, and 80 a body for the output
    steps = case["steps"]
    return {"bytes": steps * 136.0 * n + 80.0 * n, "flops": steps * (18.0 * pairs + 600.0 * n)}


# ------------------------------------------------------------------ exact values

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _exact_energy(s):
    d = _device()
    m, x, v = (torch.from_numpy(np.ascontiguousarray(a)).to(d) for a in (s.m, s.x, s.v))
    V = v - (m[:, None] * v).sum(0) / (s.M0 + m.sum())
    P = (m[:, None] * V).sum(0)
    E = (0.5 * m * (V * V).sum(1)).sum() + (P * P).sum() / (2.0 * s.M0) - (s.G * s.M0 * m / x.norm(dim=1)).sum()
    pot, rows = torch.zeros((), dtype=torch.float64, device=d), max(1, (1 << 25) // s.n)
    for a in range(0, s.n, rows):
        b = min(s.n, a + rows)
        r2 = sum((x[a:b, k, None] - x[None, :, k]) ** 2 for k in range(3))
        r2.diagonal(a).fill_(math.inf)
        pot += m[a:b] @ (r2.rsqrt_() @ m)
    E = E - 0.5 * s.G * pot
    L = (m[:, None] * torch.linalg.cross(x, V)).sum(0)
    return np.float64(E.item()), L.cpu().numpy(), P.cpu().numpy()


def _K(r, rc, form):
    y = ((r - 0.1 * rc) / (0.9 * rc)).clamp(0.0, 1.0)
    if form == RATIONAL:
        return y * y / (2.0 * y * y - 2.0 * y + 1.0)
    return y * y * y * (10.0 - 15.0 * y + 6.0 * y * y)


def _kick(s, m, x, rc, form):
    a, rows = torch.empty_like(x), max(1, (1 << 24) // s.n)
    big = int((m > 0).sum())
    for i in range(0, s.n, rows):
        j = min(s.n, i + rows)
        dx = x[None, :big] - x[i:j, None]
        r = dx.norm(dim=2)
        w = m[:big] * _K(r, torch.maximum(rc[i:j, None], rc[None, :big]), form) / r ** 3
        w[r == 0] = 0.0
        a[i:j] = s.G * torch.einsum("ij,ijk->ik", w, dx)
    return a


def _kepler(mu, dt, x, v):
    """Kepler motion of every row over dt: eccentric anomaly by Newton (bound orbits)."""
    r0, v2, rv = x.norm(dim=1), (v * v).sum(1), (x * v).sum(1)
    a = 1.0 / (2.0 / r0 - v2 / mu)
    n = (mu / a ** 3).sqrt()
    ec, es = 1.0 - r0 / a, rv / (mu * a).sqrt()
    dM = n * dt
    dE = dM.clone()
    for _ in range(30):
        f = dE - ec * dE.sin() + es * (1.0 - dE.cos()) - dM
        dE = dE - f / (1.0 - ec * dE.cos() + es * dE.sin())
    c, sn = dE.cos(), dE.sin()
    r = a * (1.0 - ec * c + es * sn)
    f, g = 1.0 - a / r0 * (1.0 - c), dt - (dE - sn) / n
    fd, gd = -(mu * a).sqrt() / (r * r0) * sn, 1.0 - a / r * (1.0 - c)
    return f[:, None] * x + g[:, None] * v, fd[:, None] * x + gd[:, None] * v


def _near_pairs(s, m, x0, x1, v0, v1, rc):
    """Pairs with a big member that may come within the larger critical radius: both ends
    apart by no more than it plus what the two paths can add between the ends."""
    reach = (x1 - x0).norm(dim=1) + 0.15 * abs(s.dt) * (v0.norm(dim=1) + v1.norm(dim=1))
    # two bodies that travel together: bound the relative path instead, pair by pair
    big, rows, found = int((m > 0).sum()), max(1, (1 << 24) // s.n), []
    for i in range(0, big, rows):
        j = min(big, i + rows)
        d = (x1[i:j, None] - x1[None, :]).norm(dim=2)
        rcm = torch.maximum(rc[i:j, None], rc[None, :])
        p, q = torch.nonzero(d <= rcm + reach[i:j, None] + reach[None, :], as_tuple=True)
        p = p + i
        keep = q > p
        p, q = p[keep], q[keep]
        # the relative cubic at 65 points; the chord between two of them is shorter than the slack
        t = torch.linspace(0.0, 1.0, 65, dtype=torch.float64, device=x0.device)
        best = torch.full((p.numel(),), math.inf, dtype=torch.float64, device=x0.device)
        d0, d1, u0, u1 = x0[p] - x0[q], x1[p] - x1[q], s.dt * (v0[p] - v0[q]), s.dt * (v1[p] - v1[q])
        for tt in t.tolist():
            h = ((1 + 2 * tt) * (1 - tt) ** 2, tt * tt * (3 - 2 * tt), tt * (1 - tt) ** 2, tt * tt * (tt - 1))
            best = torch.minimum(best, (h[0] * d0 + h[1] * d1 + h[2] * u0 + h[3] * u1).norm(dim=1))
        slack = (d1 - d0).norm(dim=1) / 32 + (u0.norm(dim=1) + u1.norm(dim=1)) / 32
        near = best <= torch.maximum(rc[p], rc[q]) + slack
        found.append(torch.stack([p[near], q[near]]))
    return torch.cat(found, 1) if found else torch.zeros((2, 0), dtype=torch.int64, device=x0.device)


def _encounters(s, m, R, x, v, rc, pairs, form):
    """The bodies of `pairs` over dt under the star and the (1 - K) part of their pairs'
    forces: extrapolated midpoint steps, 128 of them, on the host (a few hundred bodies).
    None if two of them touch."""
    where = x.device
    m, R, x, v, rc, pairs = (t.cpu() for t in (m, R, x, v, rc, pairs))
    ids, inv = torch.unique(pairs.reshape(-1), return_inverse=True)
    p, q = inv.reshape(2, -1)
    X, V, M = x[ids], v[ids], m[ids]
    rcm = torch.maximum(rc[ids][p], rc[ids][q])
    touch = R[ids][p] + R[ids][q]
    mp, mq, mu = (s.G * M[p])[:, None], (s.G * M[q])[:, None], s.G * s.M0

    def acc(X):
        d = X[q] - X[p]
        r = d.norm(dim=1)
        w = ((1.0 - _K(r, rcm, form)) / r ** 3)[:, None] * d
        a = -mu * X / X.norm(dim=1, keepdim=True) ** 3
        return a.index_add(0, p, mq * w).index_add(0, q, -mp * w)

    H, least = s.dt / 128, math.inf
    ns = (2, 4, 6, 8, 10, 12)
    for _ in range(128):
        least = min(least, float(((X[q] - X[p]).norm(dim=1) - 4 * touch).min()))
        a0, row = acc(X), []
        for k, n in enumerate(ns):
            h = H / n
            xa, va, xb, vb = X, V, X + h * V, V + h * a0
            for _ in range(n - 1):
                a = acc(xb)
                xa, va, xb, vb = xb, vb, xa + 2 * h * vb, va + 2 * h * a
            new = [(0.5 * (xa + xb + h * vb), 0.5 * (va + vb + h * acc(xb)))]
            for j in range(1, k + 1):
                c = 1.0 / ((n / ns[k - j]) ** 2 - 1.0)
                new.append(tuple(t + c * (t - o) for t, o in zip(new[j - 1], row[j - 1])))
            row = new
        X, V = row[-1]
    return None if least <= 0.0 else (ids.to(where), X.to(where), V.to(where))


def _exact_steps(s, steps, form):
    """`steps` whole steps in 64 bits; None where two bodies come near a collision (its
    moment depends on the integrator's own substeps) or an orbit is not bound."""
    d = _device()
    m, x, v, R = (torch.from_numpy(np.ascontiguousarray(a)).to(d) for a in (s.m, s.x, s.v, s.R))
    mu, n = s.G * s.M0, s.n
    V = v - (m[:, None] * v).sum(0) / (s.M0 + m.sum())
    hill = (m / (3.0 * s.M0)) ** (1.0 / 3.0) * s.rcrit_hill
    A = _kick(s, m, x, hill * x.norm(dim=1), form)
    for _ in range(steps):
        V = V + 0.5 * s.dt * A
        x = x + 0.5 * s.dt / s.M0 * (m[:, None] * V).sum(0)
        x1, V1 = _kepler(mu, s.dt, x, V)
        if not bool(torch.isfinite(x1).all()):
            return None
        rc = hill * x1.norm(dim=1)
        pairs = _near_pairs(s, m, x, x1, V, V1, rc)
        if pairs.shape[1]:
            got = _encounters(s, m, R, x, V, rc, pairs, form)
            if got is None:
                return None
            x1[got[0]], V1[got[0]] = got[1], got[2]
        x, V = x1, V1
        # accelerations at the critical radii of the drift's end
        A = _kick(s, m, x, rc, form)
        x = x + 0.5 * s.dt / s.M0 * (m[:, None] * V).sum(0)
        V = V + 0.5 * s.dt * A
    v = V + (m[:, None] * V).sum(0) / s.M0
    return {"ids": None, "m": s.m, "x": x.cpu().numpy(), "v": v.cpu().numpy(), "R": s.R}


def exact(case, seed):
    s = _systems(case, seed)
    if case["kind"] in ("energy", "energy_device"):
        E, L, P = _exact_energy(s[0])
        out = {"E": E, "L": L, "P": P}
        return {**out, "E_lost": np.float64(0.0)} if case["kind"] == "energy" else out
    # the larger workloads: many thousand pairs near each other at once, or collisions in every step
    if case["kind"] not in ("tiny", "planetesimals", "disk") or s[0].n * case["steps"] > 100000:
        return None
    return _exact_steps(s[0], case["steps"], case["changeover"])
