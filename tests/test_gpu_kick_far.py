"""The kick with bodies far outside the others (ejected ones): the packed coordinates'
grid (kick_ff.cu) leaves a few of them out, whose pairs take FP64 one by one, and where a
system is spread too wide every pair takes FP64 displacements.

Reference (some 150 rows and the far bodies') and bounds as in
test_gpu_kick_components.py.  The mixed kick forms r^-2 in floats, down to 2^-126: its
distances end at 1e12.  At 2,500 bodies (10 blocks of the bounds) one far body is left
out, three are not.
"""
import numpy as np
import pytest

import oracle as O
from tests.test_gpu_kick_components import BOUND, LD
from workloads import G_GAUSS, disk

pytestmark = pytest.mark.gpu


def _inputs(case, n):
    wl = disk(n, 0.5, 2.0, 2.0, 40 + n, name="d")
    x, v, m = wl.x.copy(), wl.v.copy(), wl.m.copy()
    rc = O.rcrit(x, v, m, 1.0, wl.dt, wl.n1, wl.n2)
    kind, d = case
    which = {"one": [n // 3], "three": [1, n // 2, n - 1], "half": list(range(0, n, 2)), "embryo": [n // 3]}[kind]
    for i in which:
        x[i] *= d / np.linalg.norm(x[i])
    if kind == "embryo":
        m[n // 3] *= 1e4
    return x, v, m, rc, sorted({*which[:3], *range(0, n, max(1, n // 150))})


def _reference(x, m, rc, rows, nm):
    X, M, R = (np.asarray(a, dtype=LD) for a in (x, m, rc))
    acc, mag = np.zeros((len(rows), 3), LD), np.zeros((len(rows), 3), LD)
    for k, i in enumerate(rows):
        d = X - X[i]
        r2 = (d * d).sum(axis=1)
        r2[i] = 1
        r = np.sqrt(r2)
        y = np.clip((r / np.maximum(R, R[i]) - LD("0.1")) / LD("0.9"), 0, 1)
        w = LD(G_GAUSS) * M * (y * y / (2 * y * y - 2 * y + 1)) / (r2 * r)
        w[i] = 0
        if i >= nm:
            w[nm:] = 0
        t = w[:, None] * d
        acc[k], mag[k] = t.sum(axis=0), abs(t).sum(axis=0)
    return acc, mag


CASES = [("one", 1e2), ("one", 1e3), ("one", 1e5), ("one", 1e7), ("one", 1e12), ("embryo", 1e4), ("three", 1e5),
         ("three", 1e9), ("half", 1e5), ("one", 1e30), ("one", 1e60), ("one", 1e160)]


@pytest.mark.parametrize("n", [129, 700, 2500])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "%s %g" % c)
def test_far_bodies_match_long_double(cuda_lib, case, n):
    import torch
    g = cuda_lib
    x, v, m, rc, rows = _inputs(case, n)
    ref, mag = _reference(x, m, rc, rows, n)
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    pos, mass, acc = T(x.T), T(m), torch.zeros((3, n), dtype=torch.float64, device=dev)

    def check(precision, what):
        err = np.abs(acc.cpu().numpy().T[rows] - ref)
        assert np.all(err <= BOUND[precision] * mag + 1e-300), (what, (err / np.maximum(mag, 1e-300)).max(axis=0))

    cand = O.precheck(x, rc, 1.5)
    for precision, layout in ((0, g.GENGA_KICK_TILED), (1, g.GENGA_KICK_TILED), (1, g.GENGA_KICK_SYMMETRIC)):
        if precision and case[1] > 1e12:
            continue
        s = g.System(pos, T(v.T), mass, g.default_params(G=G_GAUSS, precision=precision, f_pc=1.5))
        s.set_kick_layout(layout)
        s.set_rcrit(rc)
        s.kick(0.0, precheck=True, acc_out=acc)
        check(precision, (precision, layout))
        np.testing.assert_array_equal(s.candidates(), cand)
        s.kick(0.0, acc_out=acc)
        check(precision, (precision, layout))
        assert g.kick_static(pos, mass, T(rc), G_GAUSS, 0.0, precision, None, acc) == 0
        check(precision, "static")


@pytest.mark.parametrize("kind", ["test particles", "massless", "very light"])
@pytest.mark.parametrize("case", [("one", 1e5), ("half", 1e5), ("three", 1e9)], ids=lambda c: "%s %g" % c)
@pytest.mark.parametrize("n", [700, 2500])
def test_far_bodies_with_masked_pairs_and_light_masses(cuda_lib, n, case, kind):
    import torch
    g = cuda_lib
    x, v, m, rc, rows = _inputs(case, n)
    nm = n
    if kind == "test particles":
        nm = n // 3
        m[nm:] *= 1e-4
    else:
        m[1::3] *= 0.0 if kind == "massless" else 2.0 ** -45
    ref, mag = _reference(x, m, rc, rows, nm)
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    out = torch.zeros((3, n), dtype=torch.float64, device=dev)
    for precision, layout in ((0, g.GENGA_KICK_TILED), (1, g.GENGA_KICK_TILED), (1, g.GENGA_KICK_SYMMETRIC)):
        p = g.default_params(G=G_GAUSS, precision=precision, f_pc=1.5)
        if nm < n:
            p.tp_mode, p.n_massive = 2, nm
        s = g.System(T(x.T), T(v.T), T(m), p)
        s.set_kick_layout(layout)
        s.set_rcrit(rc)
        s.kick(0.0, precheck=True, acc_out=out)
        err = np.abs(out.cpu().numpy().T[rows] - ref)
        assert np.all(err <= BOUND[precision] * mag + 1e-300), (precision, layout, (err / np.maximum(mag, 1e-300)).max(axis=0))
        np.testing.assert_array_equal(s.candidates(), O.precheck(x, rc, 1.5, n_massive=nm))
