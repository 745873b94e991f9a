"""Two planets of an ensemble's system far closer than any radius: the first, coarse steps
of their encounter overflow the seed's range.  They are rejected, not taken for converged:
the group ends at the attempt limit, reported, with finite positions -- in the one-warp
path (groups of two) as in the general one (five).  Below 1e-19 the kick before the
encounter overflows already (its seed is FP32), which is reported as a non-finite state."""
import numpy as np
import pytest

from workloads.ensemble import ensemble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gap", [1e-12, 1e-15, 1e-16, 1e-18, 1e-19, 1e-21, 1e-25])
@pytest.mark.parametrize("members", [2, 5])
def test_close_members_are_reported_and_stay_finite(cuda_lib, members, gap):
    g = cuda_lib
    wl = ensemble(3, seed=77, nmin=8, nmax=8)
    for s in range(wl.n_systems):
        a = wl.offsets[s]
        wl.x[a, 2] = 0.0
        wl.x[a + 1], wl.v[a + 1] = wl.x[a], wl.v[a]
        wl.x[a + 1, 2] = gap
        for k in range(2, members):                  # a chain of neighbours 4 % apart
            x = wl.x[a] * (1.0 + 0.04 * (k - 1))
            wl.x[a + k] = x
            vc = np.sqrt(wl.G * (wl.m_star[s] + wl.m[a + k]) / np.linalg.norm(x))
            wl.v[a + k] = vc * np.cross([0.0, 0.0, 1.0], x / np.linalg.norm(x))
    ens = g.Ensemble(wl, g.default_params(G=wl.G, bs_max_steps=200), gr=False, tides=False)
    with pytest.raises(g.GengaError) as e:
        ens.step(1)
    if gap < 1e-19:
        assert e.value.code == -5
        return
    assert e.value.code == -3
    st = ens.stats()
    assert st["bs_fail"] == wl.n_systems and st["max_group"] >= members
    assert np.isfinite(ens.pos.cpu().numpy()).all()
