"""The kick's derivative in the backward pass (adjoint.cu), pair by pair, for adjoint
velocities that are nearly equal: with lv_j - lv_k formed per pair nothing cancels in the
sums over all pairs.

One step of 1e-15 days from rest without encounters: the two half kicks act at the same
positions and the drift adds the star's tide over the step, so that
  grad_x = dt [G sum_j T_kj (m_k lv_j - m_j lv_k) - G m_star (lv_k / r^3 - 3 x (x.lv) / r^5)],
  T = K (I / r^3 - 3 d d^T / r^5) + K' d d^T / r^4,
evaluated in long double.  Bound: every factor of a term is good to a few units of 2^-53
(K' to 2^-48), and up to 300 terms are summed in plain FP64 (worst case 2^-44.7 of the sum
of their absolute values): 2^-44 sum_j (4 |K| + |K'| r) |m_k lv_j - m_j lv_k| / r^3, where
m_k lv_j - m_j lv_k is m_k (lv_j - lv_k) + (m_k - m_j) lv_k.
"""
import numpy as np
import pytest

from workloads import G_GAUSS, disk

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _reference(x, m, rc, lv, dt, m_star):
    X, M, L, R = (np.asarray(a, dtype=LD) for a in (x, m, lv, rc))
    n = len(m)
    g, mag = np.zeros((n, 3), LD), np.zeros(n)
    for k in range(n):
        d = X - X[k]
        r2 = (d * d).sum(axis=1)
        r2[k] = 1
        r = np.sqrt(r2)
        rij = np.maximum(R, R[k])
        y = (r / rij - LD(0.1)) / LD(0.9)
        inside = (y > 0) & (y < 1)
        y = np.clip(y, 0, 1)
        D = 2 * y * y - 2 * y + 1
        K = y * y / D
        dK = np.where(inside, 2 * y * (1 - y) / (D * D) / (LD(0.9) * rij), 0)
        e = M[k] * (L - L[k]) + (M[k] - M)[:, None] * L[k]
        K[k] = dK[k] = 0
        de = (d * e).sum(axis=1)
        g[k] = ((K / (r2 * r))[:, None] * e + ((dK / r - 3 * K / r2) / (r2 * r) * de)[:, None] * d).sum(axis=0)
        mag[k] = float(((4 * K + dK * r) / (r2 * r) * np.sqrt((e * e).sum(axis=1))).sum())
    r = np.sqrt((X * X).sum(axis=1))[:, None]
    star = -LD(m_star) * (L / r ** 3 - 3 * X * (X * L).sum(axis=1)[:, None] / r ** 5)
    G = LD(G_GAUSS) * LD(dt)
    return G * (g + star), float(G) * mag, np.sqrt((star * star).sum(axis=1)).astype(float) * float(G)


@pytest.mark.parametrize("masses", ["equal", "mixed"])
@pytest.mark.parametrize("spread", [0.0, 1e-9, 1e-6, 1.0])
@pytest.mark.parametrize("n,band", [(2, False), (129, False), (300, False), (300, True)])
def test_kick_derivative_of_nearly_equal_adjoints(cuda_lib, n, band, spread, masses):
    import torch
    g = cuda_lib
    wl = disk(n, 0.8, 1.2, 2.0, 70 + n, name="d")
    rng = np.random.default_rng(n)
    m = np.full(n, 1e9) * (rng.uniform(0.5, 2.0, n) if masses == "mixed" else 1.0)
    lv = np.array([1.0, -2.0, 0.5]) + spread * rng.standard_normal((n, 3))
    rc = np.full(n, 0.2 if band else 1e-9)
    dt = 1e-15
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    s = g.System(T(wl.x.T), T(np.zeros((3, n))), T(m), g.default_params(G=G_GAUSS, dt=dt))
    s.adjoint_load(1, rc[None], [np.zeros((0, 2), np.uint32)])
    gx = s.adjoint_backward(T(np.zeros((3, n))), T(lv.T))[0].cpu().numpy().T
    ref, mag, star = _reference(wl.x, m, rc, lv, dt, 1.0)
    err = np.linalg.norm((gx - ref).astype(float), axis=1)
    assert np.all(err <= 2.0 ** -44 * mag + 2.0 ** -45 * star), (err / (mag + star)).max()
