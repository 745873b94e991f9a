"""Timed cases of the library's public calls, over the sizes and options its users run.

The workloads are those of the repository's own configurations, tests and benchmark:
planetesimal disks (equal masses, dN/da ~ a^-0.5, Rayleigh e and i, optional embryos),
integrated with the paper's critical-radius constants, and compact planetary systems with
GR and tides.  Units: AU, day, solar mass.

A case is a dict of plain values; `kind` names the call that is made:

  kick       System.kick, the accelerations written (the all-pairs changeover kick alone)
  static     genga.kick_static, the kick for callers that cannot allocate
  energy     System.energy (the report of a run's energy and angular momentum)
  step       System.step from a given state: levels, sub-steps, kick arithmetic, test
             particles and collisions as options
  ensemble   Ensemble.step, many small systems with GR and tides
  gradient   autograd.integrate and its backward pass
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2201_10058_gb300 import autograd, genga

G = 0.01720209895 ** 2
EARTH = 1.0 / 332946.0487
AU_CM, DAY_S, MSUN_G = 1.495978707e13, 86400.0, 1.98847e33
R_SUN = 6.957e10 / AU_CM
C_LIGHT = 173.1446326846693
DT = 6.0875
PRECISION = {"fp64": genga.GENGA_FP64, "mixed": genga.GENGA_MIXED}


def listed():
    return [
        # The kick alone, in the default arithmetic, at an odd size in the range of configuration 1.
        {"name": "kick_fp64_20011", "kind": "kick", "n": 20011, "precision": "fp64"},
        # The mixed kick at configuration 1's size: the bulk of a mid-size disk's step.
        {"name": "kick_mixed_16384", "kind": "kick", "n": 16384, "precision": "mixed"},
        # The mixed kick of a large disk, ragged: the size at which the kick is all that counts.
        {"name": "kick_mixed_131071", "kind": "kick", "n": 131071, "precision": "mixed"},
        # The allocation-free kick of a small disk inside another framework's loop: latency counts.
        {"name": "static_mixed_3001", "kind": "static", "n": 3001, "precision": "mixed"},
        # The energy report that a run writes beside its outputs, on the benchmark's disk size.
        {"name": "energy_65540", "kind": "energy", "n": 65540, "precision": "mixed"},
        # One step of configuration 0 with the defaults: the smallest whole step, many short launches.
        {"name": "step_fp64_2048", "kind": "step", "n": 2048, "precision": "fp64", "levels": 1, "substeps": 1,
         "massive": 0, "collide": False},
        # One step of configuration 1: one level, the disk percolates into a giant encounter group.
        {"name": "step_mixed_16384", "kind": "step", "n": 16384, "precision": "mixed", "levels": 1,
         "substeps": 1, "massive": 0, "collide": False},
        # One step of the benchmark's disk: two levels of ten sub-steps.
        {"name": "step_mixed_65540", "kind": "step", "n": 65540, "precision": "mixed", "levels": 2,
         "substeps": 10, "massive": 0, "collide": False},
        # The same disk with most bodies as semi-active test particles.
        {"name": "step_tp_65540", "kind": "step", "n": 65540, "precision": "mixed", "levels": 2,
         "substeps": 10, "massive": 4096, "collide": False},
        # One step of a planetesimal disk with collisions resolved (radii enlarged, as accretion runs do).
        {"name": "step_collide_4096", "kind": "step", "n": 4096, "precision": "fp64", "levels": 2,
         "substeps": 10, "massive": 0, "collide": True},
        # Multi-simulation mode: compact systems of 8 to 64 planets, a few steps in a launch.
        {"name": "ensemble_mixed_2048", "kind": "ensemble", "systems": 2048, "steps": 10, "precision": "mixed"},
        # Gradients of a short integration at configuration 4's size (forward, recording and backward).
        {"name": "gradient_4096", "kind": "gradient", "n": 4096, "steps": 2},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["kick", "kick", "static", "energy", "step", "step", "step", "ensemble", "gradient"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "kick":
        return {"kind": kind, "n": log(2000, 131071 if precision == "mixed" else 65540), "precision": precision}
    if kind == "static":
        return {"kind": kind, "n": log(500, 16384), "precision": precision}
    if kind == "energy":
        return {"kind": kind, "n": log(2000, 65540), "precision": precision}
    if kind == "ensemble":
        return {"kind": kind, "systems": log(200, 2048), "steps": rng.randint(4, 10), "precision": precision}
    if kind == "gradient":
        return {"kind": kind, "n": log(500, 4096), "steps": rng.randint(1, 2)}
    levels = rng.choice([1, 2])
    n = log(2000, 16384 if levels == 1 else 65540 if precision == "mixed" else 32768)
    massive = rng.choice([0, 0, n // rng.randint(4, 16)])
    return {"kind": kind, "n": n, "precision": precision, "levels": levels,
            "substeps": 1 if levels == 1 else rng.randint(5, 10), "massive": massive,
            "collide": massive == 0 and rng.random() < 0.3}


# ------------------------------------------------------------------ inputs

def _cartesian(a, e, inc, Om, om, M, mu):
    """Position and velocity (3, n) from Keplerian elements (elliptic)."""
    E = M + e * np.sin(M)
    for _ in range(12):
        E = E - (E - e * np.sin(E) - M) / (1.0 - e * np.cos(E))
    cE, sE = np.cos(E), np.sin(E)
    b, Ed = a * np.sqrt(1.0 - e * e), np.sqrt(mu / a ** 3) / (1.0 - e * cE)
    X, Y, U, V = a * (cE - e), b * sE, -a * sE * Ed, b * cE * Ed
    cO, sO, co, so, ci, si = np.cos(Om), np.sin(Om), np.cos(om), np.sin(om), np.cos(inc), np.sin(inc)
    P = np.stack([cO * co - sO * so * ci, sO * co + cO * so * ci, so * si])
    Q = np.stack([-cO * so - sO * co * ci, -sO * so + cO * co * ci, co * si])
    return X * P + Y * Q, U * P + V * Q


def _radius(m, rho):
    return (3.0 * m * MSUN_G / rho / (4.0 * np.pi)) ** (1.0 / 3.0) / AU_CM


def _disk(n, seed, massive=0):
    """Planetesimal disk: up to ~20,000 bodies as configurations 0, 1 and 4 (0.5-2 AU, 2 Earth masses),
    above as configuration 2 (0.5-4 AU, 5 Earth masses, 4 embryos of 0.1, placed first)."""
    rng = np.random.default_rng([20110058, n, seed])
    big = n > 24000
    outer, total, embryos = (4.0, 5.0, 4) if big else (2.0, 2.0, 0)
    a = (math.sqrt(0.5) + rng.random(n) * (math.sqrt(outer) - math.sqrt(0.5))) ** 2
    m = np.full(n, total * EARTH / n)
    m[:embryos] = 0.1 * EARTH
    e, inc = np.minimum(rng.rayleigh(0.01, n), 0.9), rng.rayleigh(0.005, n)
    Om, om, M = rng.uniform(0.0, 2.0 * np.pi, (3, n))
    x, v = _cartesian(a, e, inc, Om, om, M, G * (1.0 + m))
    v = v - (m * v).sum(axis=1, keepdims=True) / (1.0 + m.sum())
    if massive:                                # test particles carry little mass
        m[massive:] *= 1e-3
    return x, v, m, _radius(m, 2.0)


def _critical_radius(x, v, m):
    """rc = max(3 R_Hill, 0.4 dt |v|)."""
    hill = np.sqrt((x * x).sum(axis=0)) * np.cbrt(m / 3.0)
    return np.maximum(3.0 * hill, 0.4 * DT * np.sqrt((v * v).sum(axis=0)))


def _compact_systems(S, seed):
    """S systems of 8 to 64 planets (their numbers by S alone), neighbours at least 8 mutual Hill radii apart."""
    rng = np.random.default_rng([20110061, S, seed])
    ms, N = rng.uniform(0.1, 1.0, S), np.random.default_rng([20110063, S]).integers(8, 65, S)
    m = rng.uniform(0.5, 10.0, (S, 64)) * EARTH
    a = np.exp(rng.uniform(math.log(0.01), math.log(0.2), (S, 64)))
    used = np.arange(64) < N[:, None]
    a = np.sort(np.where(used, a, np.inf), axis=1)
    for k in range(63):
        h = ((m[:, k] + m[:, k + 1]) / (3.0 * ms)) ** (1.0 / 3.0)
        low = a[:, k] * (1.0 + 4.0 * h) / (1.0 - 4.0 * h)
        a[:, k + 1] = np.where(used[:, k + 1], np.maximum(a[:, k + 1], low), a[:, k])
    n, own = int(N.sum()), np.repeat(np.arange(S), N)
    m, a, star_m = m[used], a[used], ms[own]
    e, inc = np.minimum(rng.rayleigh(0.02, n), 0.5), rng.rayleigh(0.01, n)
    Om, om, M = rng.uniform(0.0, 2.0 * np.pi, (3, n))
    mu = G * (star_m + m)
    x, v = _cartesian(a, e, inc, Om, om, M, mu)
    offsets = np.concatenate([[0], np.cumsum(N)]).astype(np.int64)
    v = v - (np.add.reduceat(m * v, offsets[:-1], axis=1) / (ms + np.add.reduceat(m, offsets[:-1])))[:, own]
    first = offsets[:-1]
    dt = 2.0 * np.pi * np.sqrt(a[first] ** 3 / mu[first]) / 20.0
    spin = np.zeros((n, 3))
    spin[:, 2] = 1.0
    star = np.zeros((S, 8))
    star[:, 0], star[:, 1], star[:, 2], star[:, 3] = ms ** 0.8 * R_SUN, 0.03, 60.0 / DAY_S, 0.07
    star[:, 6] = 2.0 * np.pi / 10.0
    return SimpleNamespace(offsets=offsets, x=x.T, v=v.T, m=m, R=_radius(m, 5.5), k2=np.full(n, 0.3),
                           tau=np.full(n, 600.0 / DAY_S), rg2=np.full(n, 0.33), spin=spin, m_star=ms, dt=dt,
                           star=star, c_light=C_LIGHT, G=G, n_systems=S)


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    st = SimpleNamespace(case=case)
    if kind == "ensemble":
        st.ens = genga.Ensemble(_compact_systems(case["systems"], seed),
                                genga.default_params(G=G, precision=PRECISION[case["precision"]]))
        st.start = [t.clone() for t in (st.ens.pos, st.ens.vel, st.ens.spin, st.ens.star)]
        return st
    n = case["n"]
    x, v, m, R = _disk(n, seed, case.get("massive", 0))
    st.x, st.v, st.m = _dev(x), _dev(v), _dev(m)
    if kind == "gradient":
        rng = np.random.default_rng([20110062, n, seed])
        st.params = genga.default_params(dt=DT)
        st.leaves = [t.requires_grad_() for t in (st.x, st.v, st.m)]
        st.gx, st.gv = _dev(rng.standard_normal((3, n))), _dev(rng.standard_normal((3, n)) / 0.017)
        return st
    if kind == "static":
        st.rc = _dev(_critical_radius(x, v, m))
        st.acc = torch.empty_like(st.x)
        return st
    st.pos, st.vel, st.mass = st.x.clone(), st.v.clone(), st.m.clone()
    p = genga.default_params(dt=DT, precision=PRECISION[case["precision"]], slevels=case.get("levels", 1),
                             substeps=case.get("substeps", 1))
    if case.get("massive"):
        p.tp_mode, p.n_massive = 2, case["massive"]
    st.sys = genga.System(st.pos, st.vel, st.mass, p)
    if kind == "kick":
        st.acc = torch.empty_like(st.x)
        st.sys.rcrit(DT)
    if case.get("collide"):
        st.R = _dev(5.0 * R)
        st.radius, st.spin = st.R.clone(), torch.zeros_like(st.x)
    return st


def run(st):
    kind = st.case["kind"]
    if kind == "kick":
        st.sys.kick(0.0, acc_out=st.acc)
        return st.acc
    if kind == "static":
        rc = genga.kick_static(st.x, st.m, st.rc, G, 0.0, PRECISION[st.case["precision"]], acc_out=st.acc)
        if rc != 0:
            raise RuntimeError("kick_static: status %d" % rc)
        return st.acc
    if kind == "energy":
        E, L = st.sys.energy()
        return np.array([E]), L
    if kind == "ensemble":
        e = st.ens
        for t, t0 in zip((e.pos, e.vel, e.spin, e.star), st.start):
            t.copy_(t0)
        e.step(st.case["steps"])
        return e.pos, e.vel, e.spin, e.star
    if kind == "gradient":
        x, v = autograd.integrate(*st.leaves, st.params, st.case["steps"])
        return (x, v) + torch.autograd.grad((x, v), st.leaves, (st.gx, st.gv))
    st.pos.copy_(st.x)
    st.vel.copy_(st.v)
    if st.case["collide"]:
        st.mass.copy_(st.m)
        st.radius.copy_(st.R)
        st.spin.zero_()
        st.sys.set_collisions(st.radius, st.spin, 0.01)
        st.sys.step(1)
        return st.pos, st.vel, st.mass, st.radius, st.spin
    st.sys.step(1)
    return st.pos, st.vel


# ------------------------------------------------------------------ floors and 64-bit results

# Operations of one unordered pair: displacement and r^2 (8), r^-3 (4), both masses (2), both sums (12).
PAIR_OPS = 26
# Per body of one step outside the kick: the Kepler drift (~250), the critical radius and the HC sums.
BODY_OPS = 300


def _pairs(n, massive):
    k = massive or n
    return k * (k - 1) / 2 + k * (n - k)


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        n = case["systems"] * 36.0
        # per step: two kicks, the drift and two implicit GR/tide solves (~5 rounds of ~150 operations)
        ops = 2 * PAIR_OPS * case["systems"] * 36 * 35 / 2 + n * (BODY_OPS + 2 * 5 * 150)
        return {"bytes": n * 8 * (9 + 5 + 9), "flops": ops * case["steps"]}
    n = case["n"]
    pairs = _pairs(n, case.get("massive", 0))
    if kind in ("kick", "static"):
        return {"bytes": n * 8 * (3 + 1 + 1 + 3), "flops": PAIR_OPS * pairs}
    if kind == "energy":
        return {"bytes": n * 8 * 7, "flops": 13 * pairs}
    if kind == "gradient":
        # forward, and backward with its replay: two kicks each, and the kick's derivative (~3 kicks' work)
        return {"bytes": n * 8 * (7 + 6 + 6 + 7) * case["steps"],
                "flops": case["steps"] * (PAIR_OPS * pairs * (2 + 2 + 6) + n * BODY_OPS * 4)}
    return {"bytes": n * 8 * (7 + 6), "flops": 2 * PAIR_OPS * pairs + n * BODY_OPS}


def _exact_acceleration(x, m, rc):
    """G sum_j m_j K(r_ij) (x_j - x_i) / r_ij^3 in torch, FP64, blocks of rows."""
    n = m.shape[0]
    out = torch.empty_like(x)
    rows = max(1, (1 << 25) // n)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        d = [x[c][None, :] - x[c][a:b, None] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        r2[torch.arange(b - a), torch.arange(a, b)] = 1.0
        y = ((torch.sqrt(r2) / torch.maximum(rc[a:b, None], rc[None, :]) - 0.1) / 0.9).clamp_(0.0, 1.0)
        w = y * y
        w = w / (2.0 * w - 2.0 * y + 1.0) * m[None, :] / (r2 * torch.sqrt(r2))
        w[torch.arange(b - a), torch.arange(a, b)] = 0.0
        for c in range(3):
            out[c, a:b] = G * (w * d[c]).sum(dim=1)
    return out


def _exact_energy(x, v, m):
    n = m.shape[0]
    pot = torch.zeros((), dtype=torch.float64, device=x.device)
    rows = max(1, (1 << 25) // n)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        r2 = sum((x[c][None, :] - x[c][a:b, None]) ** 2 for c in range(3))
        r2[torch.arange(b - a), torch.arange(a, b)] = math.inf
        pot = pot - 0.5 * G * (m[a:b] * (m[None, :] / torch.sqrt(r2)).sum(dim=1)).sum()
    P = (m * v).sum(dim=1)
    E = (0.5 * m * (v * v).sum(dim=0)).sum() - (G * m / torch.sqrt((x * x).sum(dim=0))).sum() + pot
    E = E + 0.5 * (P * P).sum()
    return np.array([float(E)]), (m * torch.linalg.cross(x, v, dim=0)).sum(dim=1).cpu().numpy()


def exact(case, seed):
    """The kick's accelerations and the energy in plain FP64; the other calls integrate adaptively or
    iterate and have no closed 64-bit value."""
    kind = case["kind"]
    if kind not in ("kick", "static", "energy"):
        return None
    x, v, m, _ = _disk(case["n"], seed)
    rc = _dev(_critical_radius(x, v, m))
    x, v, m = _dev(x), _dev(v), _dev(m)
    return _exact_energy(x, v, m) if kind == "energy" else _exact_acceleration(x, m, rc)
