"""Encounter groups of 17 to 32 members (pairs taken once, or partner by partner
where a group has more than 128 pairs) and of more beside them, forward against the
oracle and backward by the dot-product identity with the oracle's tangent.

Forward bound, as in test_gpu_ensemble_groups.py: 66 times the largest spread that a
one-unit change of all starting positions causes in the oracle (4 draws), at
least 1e-12.  Backward: 1e-9 of the products' sum, as in test_gpu_adjoint.py.
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from workloads import ring

pytestmark = pytest.mark.gpu


def _rings(*members, grow=1.0):
    """Arcs of rings at 1, 1.5, ... whose neighbours are inside each other's critical radius."""
    w = [ring(60 if n <= 32 else n, r=1.0 + 0.5 * k) for k, n in enumerate(members)]
    cut = [np.arange(n) for n in members]
    cat = lambda f: np.concatenate([getattr(a, f)[c] for a, c in zip(w, cut)])
    return dataclasses.replace(w[0], name="rings", n1=grow * w[0].n1, n2=grow * w[0].n2, x=cat("x"), v=cat("v"), m=cat("m"), R=cat("R"))


CASES = {"17": lambda: _rings(17), "24": lambda: _rings(24), "32": lambda: _rings(32),
         "24 and 60": lambda: _rings(24, 60), "32, 60 and 3": lambda: _rings(32, 60, 3),
         "many pairs": lambda: _rings(32, grow=3.0)}


def _run(wl, steps):
    p = O.make_params(wl, nthreads=8)
    x, v, rcs, pairs = wl.x, wl.v, [], []
    for _ in range(steps):
        x, v, rc, pr, st = O.step_record(x, v, wl.m, p)
        assert st == 0
        rcs.append(rc)
        pairs.append(pr)
    return x, v, np.array(rcs), pairs, p


def _system(g, wl):
    import torch
    dev = torch.device("cuda:0")
    pos = torch.tensor(np.ascontiguousarray(wl.x.T), device=dev)
    vel = torch.tensor(np.ascontiguousarray(wl.v.T), device=dev)
    p = g.default_params(G=wl.G, m_star=wl.m_star, dt=wl.dt, n1=wl.n1, n2=wl.n2, f_pc=wl.f_pc)
    return g.System(pos, vel, torch.tensor(wl.m, device=dev), p), pos, vel


def _rel(a, b):
    return np.max(np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1))


@pytest.mark.parametrize("case", CASES)
def test_groups_match_oracle(cuda_lib, case):
    wl = CASES[case]()
    x, v, _, pairs, _ = _run(wl, 3)
    assert len(pairs[0]) > (128 if case == "many pairs" else 10)
    rng = np.random.default_rng(3)
    spread = 0.0
    for _ in range(4):
        w = dataclasses.replace(wl, x=np.nextafter(wl.x, np.where(rng.random(wl.x.shape) < 0.5, -np.inf, np.inf)))
        xw, vw = _run(w, 3)[:2]
        spread = max(spread, _rel(xw, x), _rel(vw, v))
    s, pos, vel = _system(cuda_lib, wl)
    s.step(3)
    assert s.stats()["max_group"] >= min(17, wl.n)
    err = max(_rel(pos.cpu().numpy().T, x), _rel(vel.cpu().numpy().T, v))
    assert err <= max(1e-12, 66.0 * spread), (err, spread)


@pytest.mark.parametrize("case", CASES)
def test_group_adjoints_satisfy_the_dot_product_identity(cuda_lib, case):
    import torch
    wl = CASES[case]()
    _, _, rcs, pairs, p = _run(wl, 2)
    rng = np.random.default_rng(1)
    dx0, dv0 = rng.standard_normal(wl.x.shape), rng.standard_normal(wl.v.shape) * 0.017
    dm0 = rng.standard_normal(wl.m.shape) * wl.m
    x, v, dx, dv = wl.x, wl.v, dx0, dv0
    for rc, pr in zip(rcs, pairs):
        x, v, dx, dv, st = O.step_frozen(x, v, wl.m, p, rc, pr, dx, dv, dm0)
        assert st == 0
    lx, lv = rng.standard_normal(wl.x.shape), rng.standard_normal(wl.v.shape)
    lhs = (lx * dx).sum() + (lv * dv).sum()
    s, _, _ = _system(cuda_lib, wl)
    s.adjoint_load(3, rcs, pairs)
    T = lambda a: torch.tensor(np.ascontiguousarray(a.T), device="cuda:0")
    gx, gv, gm = s.adjoint_backward(T(lx), T(lv))
    parts = [(gx.cpu().numpy().T * dx0).sum(), (gv.cpu().numpy().T * dv0).sum(), (gm.cpu().numpy() * dm0).sum()]
    assert abs(lhs - sum(parts)) <= 1e-9 * sum(abs(q) for q in parts), (lhs, parts)
