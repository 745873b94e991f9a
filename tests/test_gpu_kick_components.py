"""Every component of the kick's accelerations, relative to the sum of that component's
terms: nearly coplanar systems, where one component of the positions is 10^6 to 10^17
times smaller than the others, with and without inclined bodies, and single bodies next
to an axis.  The packed coordinates (kick_ff.cu) hold these on their axis' own scale, or
the pairs take FP64 displacements.

Reference: long double.  Bounds as in test_gpu_kick_tiled.py, which hold for each
component: FP64 2^-47, mixed 2^-42 of sum_j |a_ij,c|.
"""
import numpy as np
import pytest

import oracle as O
from workloads import G_GAUSS, disk

pytestmark = pytest.mark.gpu
LD = np.longdouble
BOUND = {0: 2.0 ** -47, 1: 2.0 ** -42}


def _inputs(case, n):
    wl = disk(max(n, 2), 0.5, 2.0, 2.0, 60 + n, name="d")
    x, m = wl.x[:n].copy(), wl.m[:n].copy()
    rng = np.random.default_rng(n)
    z = x[:, 2] / np.abs(x[:, 2]).max()
    k = n // 3
    if case.startswith("plane"):
        x[:, 2] = float(case.split()[1].strip(",")) * z
    if case.endswith("inclined"):
        x[k, 2] = 0.05
    if case.endswith("half"):
        x[::2, 2] = 0.03 * z[::2]
    if case == "one in the plane":
        x[k, 2] = 1.3e-13
    if case == "one on an axis":
        x[k, 0] = -2.1e-9
    if case == "single precision":
        x = x.astype(np.float32).astype(np.float64) * np.array([1.0, 1.0, 1e-9])
    if case == "in the plane":
        x[:, 2] = 0.0
    if case == "tilted":                          # a plane through rounding: components of 1e-17
        c, s = np.cos(1.0), np.sin(1.0)
        y = x[:, 1].copy()
        x[:, 1], x[:, 2] = c * y, s * y
        x[:, 1], x[:, 2] = c * x[:, 1] + s * x[:, 2], c * x[:, 2] - s * x[:, 1]
    if case == "mixed masses, inclined":
        m *= rng.uniform(0.1, 10.0, n)
    return x, wl.v[:n], m, O.rcrit(x, wl.v[:n], m, 1.0, wl.dt, wl.n1, wl.n2)


def _reference(x, m, rc):
    X, M, R = (np.asarray(a, dtype=LD) for a in (x, m, rc))
    n = len(m)
    acc, mag = np.zeros((n, 3), LD), np.zeros((n, 3), LD)
    for i in range(n):
        d = X - X[i]
        r2 = (d * d).sum(axis=1)
        r2[i] = 1
        r = np.sqrt(r2)
        y = np.clip((r / np.maximum(R, R[i]) - LD("0.1")) / LD("0.9"), 0, 1)
        w = LD(G_GAUSS) * M * (y * y / (2 * y * y - 2 * y + 1)) / (r2 * r)
        w[i] = 0
        t = w[:, None] * d
        acc[i], mag[i] = t.sum(axis=0), abs(t).sum(axis=0)
    return acc, mag


CASES = ["plane 1e-6", "plane 1e-8", "plane 1e-12", "plane 1e-17", "plane 1e-7, inclined", "plane 1e-12, inclined",
         "plane 1e-9, half", "one in the plane", "one on an axis", "single precision", "in the plane", "tilted",
         "mixed masses, inclined"]


@pytest.mark.parametrize("n", [2, 65, 129, 700])
@pytest.mark.parametrize("case", CASES)
def test_components_match_long_double(cuda_lib, case, n):
    import torch
    g = cuda_lib
    x, v, m, rc = _inputs(case, n)
    ref, mag = _reference(x, m, rc)
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    pos, mass, acc = T(x.T), T(m), torch.zeros((3, n), dtype=torch.float64, device=dev)

    def check(precision, what):
        err = np.abs(acc.cpu().numpy().T - ref)
        assert np.all(err <= BOUND[precision] * mag + 1e-300), (what, (err / np.maximum(mag, 1e-300)).max(axis=0))

    cand = O.precheck(x, rc, 1.5)
    for precision, layout in ((0, g.GENGA_KICK_TILED), (0, g.GENGA_KICK_SYMMETRIC), (1, g.GENGA_KICK_TILED),
                              (1, g.GENGA_KICK_SYMMETRIC)):
        s = g.System(pos, T(v.T), mass, g.default_params(G=G_GAUSS, precision=precision, f_pc=1.5))
        s.set_kick_layout(layout)
        s.set_rcrit(rc)
        s.kick(0.0, precheck=True, acc_out=acc)
        check(precision, (precision, layout))
        np.testing.assert_array_equal(s.candidates(), cand)
        s.kick(0.0, acc_out=acc)                  # without the pre-check
        check(precision, (precision, layout))
    for precision in (0, 1):
        assert g.kick_static(pos, mass, T(rc), G_GAUSS, 0.0, precision, None, acc) == 0
        check(precision, "static")
