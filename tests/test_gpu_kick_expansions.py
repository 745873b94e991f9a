"""The mixed symmetric kick in float expansions (kick_ff.cu) on the inputs that
select its instances: equal masses per tile, mixed masses, massless and very
light bodies, a far outlier (coordinates of four parts), other units, test
particles across a tile, ragged and single tiles.

Reference: the pair sum in numpy with 64-bit mantissas (long double).  Bound: a
term's relative error is below 2^-43 (r^2 2^-47, r^-3 2^-45, K 2^-43 of it in the
worst case, the product 2^-46), and the float sums of 16 terms add less than
2^-45 of the sum of their absolute values, so |da_i| <= 2^-42 sum_j |a_ij|.
"""
import numpy as np
import pytest

import oracle as O
from workloads import G_GAUSS, disk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g(cuda_lib):
    return cuda_lib


def _reference(x, m, rc, G, nm):
    """Accelerations and sums of the terms' absolute values, in long double."""
    X, M, R = (np.asarray(a, dtype=np.longdouble) for a in (x, m, rc))
    n = len(m)
    acc, mag = np.zeros((n, 3), np.longdouble), np.zeros(n)
    for i in range(n):
        d = X - X[i]
        r2 = (d * d).sum(axis=1)
        r2[i] = 1
        r = np.sqrt(r2)
        rij = np.maximum(R, R[i])
        with np.errstate(divide="ignore"):
            y = np.clip((r / rij - np.longdouble(0.1)) / np.longdouble(0.9), 0, 1)
        w = np.longdouble(G) * M * (y * y / (2 * y * y - 2 * y + 1)) / (r2 * r)
        w[i] = 0
        if i >= nm:
            w[nm:] = 0
        acc[i] = (w[:, None] * d).sum(axis=0)
        mag[i] = float((w * r).sum())
    return acc.astype(np.float64), mag


def _inputs(case, n):
    wl = disk(n, 0.5, 2.0, 2.0, 900 + n, name="d")
    x, v, m = wl.x.copy(), wl.v.copy(), wl.m.copy()
    rng = np.random.default_rng(n)
    nm, scale = n, 1.0
    if case == "mixed masses":
        m *= rng.uniform(0.5, 2.0, n)
    elif case == "one embryo":
        m[n // 2] *= 1000.0
    elif case == "massless":
        m[rng.random(n) < 0.3] = 0.0
    elif case == "very light":
        m[rng.random(n) < 0.3] *= 2.0 ** -45
    elif case == "outlier":
        x[n // 3] *= 3.0e7
    elif case == "far outlier":
        x[0] *= 1.0e12
    elif case == "metres and kilograms":
        scale = 1.495978707e11
        m *= 1.98847e30
    elif case == "test particles":
        nm = n // 3
        m[nm:] *= 1e-4
    elif case == "close pairs":
        k = n // 2
        x[n - k:] = x[:k] + 10.0 ** rng.uniform(-9, -3, (k, 1)) * rng.standard_normal((k, 3))
    rc = O.rcrit(x, v, m, wl.m_star if scale == 1.0 else 1.98847e30, wl.dt, wl.n1, wl.n2)
    if case == "close pairs":
        rc[::2] = 0.0                          # K = 1 between half of the bodies
    return x * scale, v, m, rc * scale, nm


CASES = ["equal masses", "mixed masses", "one embryo", "massless", "very light", "outlier", "far outlier",
         "metres and kilograms", "test particles", "close pairs"]


@pytest.mark.parametrize("n,P", [(5, 1), (128, 1), (129, 1), (700, 2)])
@pytest.mark.parametrize("case", CASES)
def test_expansion_kick_matches_long_double(g, case, n, P):
    import torch
    x, v, m, rc, nm = _inputs(case, n)
    G = G_GAUSS if case != "metres and kilograms" else 6.6743e-11
    dev = torch.device("cuda:0")
    pos = torch.tensor(np.ascontiguousarray(x.T), device=dev)
    vel = torch.tensor(np.ascontiguousarray(v.T), device=dev)
    mass = torch.tensor(m, device=dev)
    p = g.default_params(G=G, precision=g.GENGA_MIXED)
    if nm < n:
        p.tp_mode, p.n_massive = 2, nm
    s = g.System(pos, vel, mass, p)
    s.set_kick_layout(g.GENGA_KICK_SYMMETRIC, P)
    s.set_rcrit(rc)
    acc = torch.zeros((3, n), dtype=torch.float64, device=dev)
    s.kick(0.0, precheck=True, acc_out=acc)
    torch.cuda.synchronize()
    a = acc.cpu().numpy().T
    ref, mag = _reference(x, m, rc, G, nm)
    err = np.linalg.norm(a - ref, axis=1)
    assert np.all(err <= 2.0 ** -42 * mag + 1e-300), (err / np.maximum(mag, 1e-300)).max()
    np.testing.assert_array_equal(s.candidates(), O.precheck(x, rc, p.f_pc, n_massive=nm))
