"""Mergers inside a giant close-encounter group (a 300-body ring, the persistent
Bulirsch-Stoer kernel) in the course of the integration: the overlap search over
all members, with and without a collision precision, against the oracle.  Bounds
as in test_gpu_collisions.py.  Three pairs are set to meet after 0.3, 0.5 and 0.8
of the step; no radius reaches a neighbour otherwise."""
import numpy as np
import pytest

import oracle as O
from tests.test_gpu_collisions import _host, _same_log, _system
from workloads import ring

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coll_tol", [0.0, 1e-3])
def test_mid_step_mergers_match_oracle(cuda_lib, coll_tol):
    g = cuda_lib
    wl = ring(300)
    R = np.full(wl.n, 0.15 * wl.extra["spacing"])
    for a, when in ((0, 0.5), (100, 0.3), (201, 0.8)):
        d = wl.x[a] - wl.x[a + 1]
        wl.v[a + 1] += 0.7 * d / (when * wl.dt)          # 0.7 of the spacing closed by then
    s = _system(g, wl, R, precision=coll_tol)
    s.step(1)
    assert s.stats()["max_group"] == 300
    glog, gdU = s.mergers()
    x, v, m, R1, S1, alive, U, olog, status, st = O.step_coll(wl.x, wl.v, wl.m, R, np.zeros((wl.n, 3)),
                                                             O.make_params(wl, nthreads=8), 1, coll_tol=coll_tol)
    assert status == 0 and len(olog) == 3
    _same_log(glog, olog)
    np.testing.assert_array_equal(s.alive(), alive)
    np.testing.assert_array_equal(s.mass.cpu().numpy(), m)
    err = np.linalg.norm(_host(s.pos) - x, axis=1) / np.linalg.norm(x, axis=1)
    assert err.max() <= 1e-12, err.max()
