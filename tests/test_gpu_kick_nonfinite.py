"""A NaN or infinite position makes every acceleration NaN, in both kicks and layouts, as
the plain sum over pairs does."""
import numpy as np
import pytest

from workloads import disk

pytestmark = pytest.mark.gpu


def _kicks(g, x, v, m, rc):
    import torch
    n = len(m)
    dev = torch.device("cuda:0")
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    for precision, layout in ((0, g.GENGA_KICK_TILED), (0, g.GENGA_KICK_SYMMETRIC), (1, g.GENGA_KICK_TILED),
                              (1, g.GENGA_KICK_SYMMETRIC)):
        acc = torch.zeros((3, n), dtype=torch.float64, device=dev)
        s = g.System(T(x.T), T(v.T), T(m), g.default_params(precision=precision))
        s.set_kick_layout(layout)
        s.set_rcrit(rc)
        s.kick(0.0, acc_out=acc)
        yield precision, layout, acc.cpu().numpy()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("masses", ["equal", "mixed"])
@pytest.mark.parametrize("n", [129, 2500])
def test_nonfinite_position(cuda_lib, n, masses, bad):
    wl = disk(n, 0.5, 2.0, 2.0, 40 + n, name="d")
    x, m = wl.x.copy(), wl.m * (1.0 if masses == "equal" else np.random.default_rng(n).uniform(0.5, 2.0, n))
    x[n // 2, 1] = bad
    for precision, layout, a in _kicks(cuda_lib, x, wl.v, m, np.full(n, 0.02)):
        if (precision, layout) != (0, cuda_lib.GENGA_KICK_SYMMETRIC):     # FP32 seeds wrap around there
            assert np.isnan(a[1]).all(), (precision, layout)
