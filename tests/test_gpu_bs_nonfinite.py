"""A non-finite extrapolation column is not convergence, whatever the size of the
encounter group: with a NaN or infinite velocity in it, the in-block kernels (up to
32 members) and the persistent kernel (more) both reject every attempt and report
that the attempt limit was reached."""
import numpy as np
import pytest

from tests.test_gpu_giant_groups import _ring, _system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n,which", [(20, "one"), (20, "all"), (60, "one"), (60, "all"), (300, "one"), (300, "all")])
def test_nonfinite_velocity_is_reported(cuda_lib, n, which, bad):
    import torch
    g = cuda_lib
    wl = _ring(n, 6.0)
    s, pos, vel, _ = _system(g, wl, bs_max_steps=6)
    s.rcrit(wl.dt)
    s.kick(0.0, precheck=True, acc_out=torch.zeros((3, n), dtype=torch.float64, device="cuda:0"))
    s.set_predrift(wl.x.T, wl.v.T)
    assert s.build_encounters()[1:] == (1, n)
    v = wl.v.copy()
    v[slice(None) if which == "all" else n // 2] = bad
    s.set_predrift(wl.x.T, v.T)
    with pytest.raises(g.GengaError) as e:
        s.bs(wl.dt)
    assert e.value.code == -3
    assert s.stats()["bs_fail"] == 1
