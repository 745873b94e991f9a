"""The pair potential of the energy report (energy.cu): 1/r of every unordered
pair from float digits, against long double.

Massive disks (the pair potential is 7-25 % of the energy), sizes of one ragged
tile to several, mixed masses, test particles across a tile, a far outlier (the
FP64 path for every pair), close pairs and a pair at one place.  Bound: every
term (kinetic, star, pair, momentum) is formed to a few units of 2^-53 and summed
with compensation, so |dE| <= 2^-49 (T + |star| + |pairs| + P^2 / 2 m_star); the
same for each component of L with its terms' absolute values.
"""
import numpy as np
import pytest

from workloads import G_GAUSS, disk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g(cuda_lib):
    return cuda_lib


def _reference(x, v, m, nm):
    X, V, M = (np.asarray(a, dtype=np.longdouble) for a in (x, v, m))
    n = len(m)
    U = np.longdouble(0)
    with np.errstate(divide="ignore"):
        for i in range(n - 1):
            d = X[i + 1:(n if i < nm else max(nm, i + 1))] - X[i]
            U += M[i] * (M[i + 1:i + 1 + len(d)] / np.sqrt((d * d).sum(axis=1))).sum()
    G = np.longdouble(G_GAUSS)
    P = (M[:, None] * V).sum(axis=0)
    terms = [(M * (V * V).sum(axis=1)).sum() / 2, -(G * M / np.sqrt((X * X).sum(axis=1))).sum(), -G * U,
             (P * P).sum() / 2]
    L = M[:, None] * np.cross(X, V)
    mag = (M[:, None] * (np.abs(X[:, [1, 2, 0]] * V[:, [2, 0, 1]]) + np.abs(X[:, [2, 0, 1]] * V[:, [1, 2, 0]]))).sum(axis=0)
    return float(sum(terms)), float(sum(abs(t) for t in terms)), L.sum(axis=0).astype(float), mag.astype(float)


@pytest.mark.parametrize("n", [1, 2, 5, 128, 129, 700])
@pytest.mark.parametrize("case", ["equal", "mixed", "test particles", "outlier", "close pairs", "one place"])
def test_energy_matches_long_double(g, case, n):
    import torch
    wl = disk(max(n, 2), 0.5, 2.0, 2.0, 500 + n, name="d")
    x, v = wl.x[:n].copy(), wl.v[:n].copy()
    rng = np.random.default_rng(n)
    m = np.full(n, 0.3 / n) * (rng.uniform(0.1, 2.0, n) if case == "mixed" else 1.0)
    nm = max(1, n // 3) if case == "test particles" else n
    if case == "outlier":
        x[n // 2] *= 1e7
    if case == "close pairs" and n > 1:
        k = n // 2
        x[n - k:] = x[:k] + 10.0 ** rng.uniform(-14, -3, (k, 3))
    if case == "one place" and n > 1:
        x[n - 1] = x[0]
    p = g.default_params(G=G_GAUSS)
    if nm < n:
        p.tp_mode, p.n_massive = 2, nm
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda:0")
    s = g.System(T(x.T), T(v.T), T(m), p)
    E, L = s.energy()
    Er, mag, Lr, magL = _reference(x, v, m, nm)
    if np.isinf(Er):
        assert E == Er
    else:
        assert abs(E - Er) <= 2.0 ** -49 * mag, abs(E - Er) / mag
    assert np.all(np.abs(L - Lr) <= 2.0 ** -49 * magL + 1e-300)
    assert s.energy()[0] == E                     # fixed order: the same bits again
