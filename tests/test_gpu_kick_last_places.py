"""The FP64 tiled kick's accelerations of a single term, to 2^-50: the displacement is
exact, r^-3 within 2^-52, mass, product, G and the fold 2^-53 each.

* a mass with all 53 bits set at random, in the instances of unequal masses (its own tile
  and others): its third float counts;
* a full tile of equal masses of which one body is near and comes last, the others a
  thousand times farther (10^-4 of the acceleration together): the instance of equal
  masses, on bodies of other tiles.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _check(g, x, m, rows):
    import torch
    n = len(m)
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    pos, mass, acc = T(x.T), T(m), torch.zeros((3, n), dtype=torch.float64, device=dev)
    s = g.System(pos, torch.zeros_like(pos), mass, g.default_params(G=1.0, precision=0))
    s.set_kick_layout(g.GENGA_KICK_TILED)
    s.set_rcrit(np.full(n, 1e-9))
    s.kick(0.0, acc_out=acc)
    acc2 = torch.zeros_like(acc)
    assert g.kick_static(pos, mass, T(np.full(n, 1e-9)), 1.0, 0.0, 0, None, acc2) == 0
    X, M = x.astype(LD), m.astype(LD)
    src = np.flatnonzero(m)
    for a in (acc, acc2):
        a = a.cpu().numpy().T
        worst = 0.0
        for i in rows:
            d = X[src] - X[i]
            r2 = (d * d).sum(axis=1)
            ref = ((M[src] / (r2 * np.sqrt(r2)))[:, None] * d).sum(axis=0)
            worst = max(worst, float(np.sqrt(((a[i] - ref) ** 2).sum() / (ref * ref).sum())))
        assert worst <= 2.0 ** -50, worst * 2.0 ** 50


@pytest.mark.parametrize("seed", range(4))
def test_mass_of_53_bits(cuda_lib, seed):
    rng = np.random.default_rng(seed)
    n = 1500
    m = np.zeros(n)
    k = int(rng.integers(0, n))
    m[k] = 3e-6 * (1.0 + rng.random())
    _check(cuda_lib, rng.uniform(-2.0, 2.0, (n, 3)), m, [i for i in range(n) if i != k])


@pytest.mark.parametrize("seed", range(4))
def test_equal_masses_on_distant_tiles(cuda_lib, seed):
    rng = np.random.default_rng(seed)
    n = 128 * 6
    m = np.zeros(n)
    m[:128] = 3e-6 * (1.0 + rng.random())
    u = rng.standard_normal((127, 3))
    x = rng.uniform(0.1, 1.0, (n, 3))
    x[:127] = 1e3 * u / np.linalg.norm(u, axis=1)[:, None]
    x[:127][np.abs(x[:127]) < 1.0] = 1.0
    _check(cuda_lib, x, m, range(128, n))
