"""The time-out message of the persistent Bulirsch-Stoer kernel names the limit that ran
out: the first wait's is longer by the in-block limit where smaller groups are integrated
beside it.  A block that does not exist makes the first wait run out, after 51 ms at most."""
import pytest

from tests.test_gpu_bs_groups import _rings, _system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members,limit", [((60,), "0.001 s"), ((24, 60), "0.051 s")])
def test_message_names_the_limit(cuda_lib, members, limit):
    g = cuda_lib
    s, _, _ = _system(g, _rings(*members))
    s.set_wait_limits(bs_group_seconds=0.05, barrier_seconds=1e-3, barrier_absent_blocks=1)
    with pytest.raises(g.GengaError) as e:
        s.step(1)
    assert e.value.code == -4 and limit in str(e.value), str(e.value)
    s.set_wait_limits()
    s.step(1)
