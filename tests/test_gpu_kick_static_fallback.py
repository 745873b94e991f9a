"""The allocation-free kick beyond the size whose packed bodies and one partial sum per
body fit its 16 MiB of scratch: kick_kernel on thresholds and partial sums, both
precisions, against long double on sampled rows.  Bounds as in test_gpu_kick_tiled.py:
2^-47 (FP64) and 2^-42 (mixed) of sum_j |a_ij|."""
import numpy as np
import pytest

import oracle as O
from workloads import disk

pytestmark = pytest.mark.gpu
LD = np.longdouble
PACKED_BYTES = 64          # a body's seven pairs of floats and 1/rc (56 + 8), at least
PARTIAL_BYTES = 24         # one partial sum
ROWS = 24


@pytest.fixture(scope="module")
def case():
    out = {}
    for n in (200001, 279616):                   # the second: the largest accepted
        assert (PACKED_BYTES + PARTIAL_BYTES) * n > 16 << 20
        wl = disk(n, 0.5, 2.0, 2.0, 7, name="d")
        rc = O.rcrit(wl.x, wl.v, wl.m, wl.m_star, wl.dt, wl.n1, wl.n2)
        X, M, R = (np.asarray(a, dtype=LD) for a in (wl.x, wl.m, rc))
        rows = np.unique(np.concatenate([[0, 127, 128, n - 1], np.linspace(0, n - 1, ROWS).astype(int)]))
        ref, mag = np.zeros((len(rows), 3), LD), np.zeros(len(rows))
        for k, i in enumerate(rows):
            d = X - X[i]
            r2 = (d * d).sum(axis=1)
            r2[i] = 1
            r = np.sqrt(r2)
            y = np.clip((r / np.maximum(R, R[i]) - LD("0.1")) / LD("0.9"), 0, 1)
            w = LD(wl.G) * M * (y * y / (2 * y * y - 2 * y + 1)) / (r2 * r)
            w[i] = 0
            ref[k], mag[k] = (w[:, None] * d).sum(axis=0), float((w * r).sum())
        out[n] = wl, rc, rows, ref, mag
    return out


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [200001, 279616])
def test_fallback_matches_long_double(cuda_lib, case, n, precision):
    import torch
    g = cuda_lib
    wl, rc, rows, ref, mag = case[n]
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    acc, vel = torch.zeros((3, n), dtype=torch.float64, device=dev), T(wl.v.T)
    assert g.kick_static(T(wl.x.T), T(wl.m), T(rc), wl.G, 0.25, precision, vel, acc) == 0
    a = acc.cpu().numpy().T
    err = np.linalg.norm((a[rows] - ref).astype(float), axis=1)
    assert np.all(err <= (2.0 ** -47, 2.0 ** -42)[precision] * mag), (err / mag).max()
    np.testing.assert_allclose(vel.cpu().numpy().T, wl.v + 0.25 * a, rtol=1e-15, atol=0)
