"""Encounter groups of two and three members in the ensemble's one-warp path, in metres,
kilograms and seconds, in systems that lie in the y-z plane (x exactly 0): the lanes
without a member must not come near the star.  Against the oracle in the same units; bound as in
test_gpu_ensemble_groups.py."""
import copy

import numpy as np
import pytest

from tests.test_gpu_ensemble import _oracle_run
from tests.test_gpu_ensemble_groups import _rel
from workloads.ensemble import ensemble

pytestmark = pytest.mark.gpu
AU, DAY, MSUN = 1.495978707e11, 86400.0, 1.98847e30


def _si(wl):
    w = copy.deepcopy(wl)
    w.x, w.v, w.m, w.R = wl.x * AU, wl.v * AU / DAY, wl.m * MSUN, wl.R * AU
    w.m_star, w.dt, w.G = wl.m_star * MSUN, wl.dt * DAY, wl.G * AU ** 3 / (MSUN * DAY ** 2)
    return w


@pytest.mark.parametrize("m", [2, 3])
def test_systems_in_the_yz_plane(cuda_lib, m):
    g = cuda_lib
    wl = ensemble(4, seed=420 + m, nmin=8, nmax=16)
    for s in range(wl.n_systems):
        a, b = wl.offsets[s], wl.offsets[s + 1]
        for k in range(a, b):                        # circular orbits, neighbours 20 % apart, the first m 4 %
            i = k - a
            r = 0.02 * (1.0 + 0.04 * i if i < m else 1.2 ** (i - m + 1) * (1.0 + 0.04 * m))
            phi = 0.0 if i < m else 2.4 * i
            vc = np.sqrt(wl.G * (wl.m_star[s] + wl.m[k]) / r)
            wl.x[k] = [0.0, r * np.cos(phi), r * np.sin(phi)]
            wl.v[k] = [0.0, -vc * np.sin(phi), vc * np.cos(phi)]
        wl.dt[s] = 2 * np.pi * np.sqrt(0.02 ** 3 / (wl.G * wl.m_star[s])) / 20
    wl = _si(wl)
    kw = {"gr": False, "tides": False}
    ens = g.Ensemble(wl, g.default_params(G=wl.G), **kw)
    ens.step(1)
    st = ens.stats()
    assert st["bs_fail"] == 0 and st["max_group"] >= m
    pos, vel = ens.pos.cpu().numpy().T, ens.vel.cpu().numpy().T
    rng = np.random.default_rng(m)
    for s in range(wl.n_systems):
        x, v = _oracle_run(wl, s, 1, **kw)[:2]
        spread = 0.0
        for _ in range(4):
            w = copy.deepcopy(wl)
            w.x = np.nextafter(w.x, np.where(rng.random(w.x.shape) < 0.5, -np.inf, np.inf))
            xw, vw = _oracle_run(w, s, 1, **kw)[:2]
            spread = max(spread, _rel(xw, x), _rel(vw, v))
        a, b = wl.offsets[s], wl.offsets[s + 1]
        err = max(_rel(pos[a:b], x), _rel(vel[a:b], v))
        assert err <= max(1e-12, 66.0 * spread), (s, err, spread)
