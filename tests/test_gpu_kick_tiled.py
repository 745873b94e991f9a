"""The tiled kick on packed bodies (kick_tile.cu), FP64 and mixed, on the inputs that
select its instances and its FP64 buffer of near pairs, at sizes around a group
of 64, a tile of 128 and several chunks; and the allocation-free kick on both of
its paths.

Reference: the pair sum in long double.  Bounds, relative to sum_j |a_ij|:
  * mixed: a term's error is below 2^-43 and the float sums of 32 terms add less
    than 2^-45 each: 2^-42;
  * FP64: the displacement is within 2^-53 of |d| (2^-51 of the term), r^-3 within
    2^-52, and the sum of up to 256 terms in plain FP64 is a random walk of
    roundings of at most 2^-53 of the sum so far, 6 sigma below 2^-47: 2^-47 in all.
"""
import numpy as np
import pytest

import oracle as O
from tests.test_gpu_kick_expansions import CASES, _inputs, _reference
from workloads import G_GAUSS, disk

pytestmark = pytest.mark.gpu
BOUND = {0: 2.0 ** -47, 1: 2.0 ** -42}


@pytest.fixture(scope="module")
def g(cuda_lib):
    return cuda_lib


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case,n", [("equal masses", 1)] + [(c, n) for c in CASES for n in (5, 64, 65, 129, 700)])
def test_tiled_kick_matches_long_double(g, case, n, precision):
    import torch
    x, v, m, rc, nm = _inputs(case, max(n, 2))
    x, v, m, rc, nm = x[:n], v[:n], m[:n], rc[:n], min(nm, n)
    G = G_GAUSS if case != "metres and kilograms" else 6.6743e-11
    dev = torch.device("cuda:0")
    pos = torch.tensor(np.ascontiguousarray(x.T), device=dev)
    vel = torch.tensor(np.ascontiguousarray(v.T), device=dev)
    mass = torch.tensor(m, device=dev)
    p = g.default_params(G=G, precision=precision)
    if nm < n:
        p.tp_mode, p.n_massive = 2, nm
    s = g.System(pos, vel, mass, p)
    s.set_kick_layout(g.GENGA_KICK_TILED)
    s.set_rcrit(rc)
    acc = torch.zeros((3, n), dtype=torch.float64, device=dev)
    s.kick(0.0, precheck=True, acc_out=acc)
    torch.cuda.synchronize()
    a = acc.cpu().numpy().T
    ref, mag = _reference(x, m, rc, G, nm)
    err = np.linalg.norm(a - ref, axis=1)
    assert np.all(err <= BOUND[precision] * mag + 1e-300), (err / np.maximum(mag, 1e-300)).max()
    if n > 1:
        np.testing.assert_array_equal(s.candidates(), O.precheck(x, rc, p.f_pc, n_massive=nm))
    if nm == n:                                # the same kernels, on the entry point's own memory
        acc2 = torch.zeros_like(acc)
        assert g.kick_static(pos, mass, torch.tensor(rc, device=dev), G, 0.0, precision, None, acc2) == 0
        assert np.all(np.linalg.norm(acc2.cpu().numpy().T - ref, axis=1) <= BOUND[precision] * mag + 1e-300)


@pytest.mark.parametrize("precision", [0, 1])
def test_static_kick_where_the_packed_bodies_do_not_fit(g, precision):
    """150,001 bodies: the scratch holds only the thresholds and one partial sum per
    body, the path of kick_kernel; against the system's kick to the mixed bound."""
    import torch
    n = 150001
    wl = disk(n, 0.5, 2.0, 2.0, 3, name="d")
    rc = O.rcrit(wl.x, wl.v, wl.m, wl.m_star, wl.dt, wl.n1, wl.n2)
    dev = torch.device("cuda:0")
    pos = torch.tensor(np.ascontiguousarray(wl.x.T), device=dev)
    vel = torch.tensor(np.ascontiguousarray(wl.v.T), device=dev)
    mass = torch.tensor(wl.m, device=dev)
    acc, acc2 = (torch.zeros((3, n), dtype=torch.float64, device=dev) for _ in range(2))
    assert g.kick_static(pos, mass, torch.tensor(rc, device=dev), wl.G, 0.0, precision, None, acc) == 0
    s = g.System(pos, vel, mass, g.default_params(G=wl.G, precision=0))
    s.set_rcrit(rc)
    s.kick(0.0, precheck=False, acc_out=acc2)
    torch.cuda.synchronize()
    rows = np.arange(0, n, 5003)
    mag = np.array([_mag(wl.x, wl.m, wl.G, i) for i in rows])
    err = (acc - acc2).norm(dim=0).cpu().numpy()[rows]
    assert np.all(err <= BOUND[1] * mag), (err / mag).max()


def _mag(x, m, G, i):
    r2 = ((x - x[i]) ** 2).sum(axis=1)
    r2[i] = np.inf
    return G * (m / r2).sum()


def test_r3_next_to_powers_of_two(g):
    """The FP64 kick forms m r^-3 as a float plus a whole number of last places of a
    double, which changes scale at powers of two.  One body of mass 2^-20 and 20,000
    massless ones at distances whose r^-3 lies within 40 float places (2^-24 relative)
    on either side of one: each acceleration has a single term, good to 2^-50 (displacement 2^-51, r^-3
    2^-52, product, G and the fold 2^-53 each)."""
    import torch
    n = 20001
    rng = np.random.default_rng(9)
    k = rng.integers(-6, 7, n)
    r = (2.0 ** k * (1.0 + rng.uniform(-40, 40, n) * 2.0 ** -24)) ** (-1.0 / 3.0)
    u = rng.standard_normal((n, 3))
    x = np.array([1.0, 0.5, 0.25]) + r[:, None] * u / np.linalg.norm(u, axis=1)[:, None]
    x[0] = [1.0, 0.5, 0.25]
    m = np.zeros(n)
    m[0] = 2.0 ** -20
    dev = torch.device("cuda:0")
    pos = torch.tensor(np.ascontiguousarray(x.T), device=dev)
    s = g.System(pos, torch.zeros_like(pos), torch.tensor(m, device=dev), g.default_params(G=1.0, precision=0))
    s.set_kick_layout(g.GENGA_KICK_TILED)
    s.set_rcrit(np.full(n, 1e-9))
    acc = torch.zeros_like(pos)
    s.kick(0.0, precheck=False, acc_out=acc)
    X = x.astype(np.longdouble)
    d = X[0] - X[1:]
    d2 = (d * d).sum(axis=1)
    ref = np.longdouble(m[0]) * d / (d2 * np.sqrt(d2))[:, None]
    err = np.sqrt(((acc.cpu().numpy().T[1:] - ref) ** 2).sum(axis=1) / (ref * ref).sum(axis=1)).astype(float)
    assert err.max() <= 2.0 ** -50, (err.max(), int((err > 2.0 ** -50).sum()))
