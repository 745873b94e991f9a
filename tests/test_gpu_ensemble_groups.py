"""Encounter groups of the ensemble kernel on both Bulirsch-Stoer paths (up to four
members: one warp, all columns of the extrapolation at once; more: the general
path) against the oracle: chains of m planets 4 % apart in one direction, so that
neighbours are inside each other's critical radius.

Such chains amplify rounding (up to 10^8 over the 5 steps), so the bound follows
from the oracle itself: kernel and oracle round differently in every one of the
~100 operations that a component goes through per step, 5 steps, in a random walk:
sqrt(500) ~ 22 units of the last place, 3 sigma 66, against the largest spread that
a one-unit change of all starting positions causes in the oracle (4 draws); at
least 1e-12.  The mixed kick's terms are good to 2^-43, 2^10 units: its bound is
2^10 times that.
"""
import copy

import numpy as np
import pytest

from tests.test_gpu_ensemble import _oracle_run
from workloads.ensemble import ensemble

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.max(np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1))


@pytest.mark.parametrize("kw", [{}, {"gr_split": True}])
@pytest.mark.parametrize("m", [2, 3, 4, 5, 7])
def test_encounter_chain_matches_oracle(cuda_lib, m, kw):
    g = cuda_lib
    wl = ensemble(5, seed=400 + m, nmin=8, nmax=32)
    for s in range(wl.n_systems):
        a = wl.offsets[s]
        for k in range(1, m):
            x = wl.x[a] * (1.0 + 0.04 * k)
            wl.x[a + k] = x
            vc = np.sqrt(wl.G * (wl.m_star[s] + wl.m[a + k]) / np.linalg.norm(x))
            wl.v[a + k] = vc * np.cross([0.0, 0.0, 1.0], x / np.linalg.norm(x))
    rng = np.random.default_rng(m)
    moved = []
    for _ in range(4):
        w = copy.deepcopy(wl)
        w.x = np.nextafter(w.x, np.where(rng.random(w.x.shape) < 0.5, -np.inf, np.inf))
        moved.append(w)
    ref, tol = [], []
    for s in range(wl.n_systems):
        x, v = _oracle_run(wl, s, 5, **kw)[:2]
        spread = max(max(_rel(p[0], x), _rel(p[1], v)) for p in (_oracle_run(w, s, 5, **kw) for w in moved))
        ref.append((x, v))
        tol.append(max(1e-12, 66.0 * spread))
    for precision, threads in ((0, 32), (0, 64), (0, 128), (1, 64)):
        ens = g.Ensemble(wl, g.default_params(G=wl.G, precision=precision), **kw)
        ens.set_tile(threads, 4)
        ens.step(5)
        st = ens.stats()
        assert st["bs_fail"] == 0 and st["n_groups"] > 0 and st["max_group"] >= m
        pos, vel = ens.pos.cpu().numpy().T, ens.vel.cpu().numpy().T
        for s in range(wl.n_systems):
            a, b = wl.offsets[s], wl.offsets[s + 1]
            err = max(_rel(pos[a:b], ref[s][0]), _rel(vel[a:b], ref[s][1]))
            assert err <= tol[s] * (1 if precision == 0 else 1024), (s, err, tol[s])
