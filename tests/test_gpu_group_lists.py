"""Partner lists, groups and group lists at the edges of the one-block scans (passes of
16,384 entries, up to 32,768 or 131,072 bodies) and past it, on clusters of known members:
bodies of one cluster are inside each other's critical radius, clusters far apart."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 16383, 16384, 16385, 32768, 32769, 131072, 131073])
def test_clusters_become_groups(cuda_lib, n):
    import torch
    g = cuda_lib
    rng = np.random.default_rng(n)
    sizes = []
    while sum(sizes) < n:
        sizes.append(min(int(rng.integers(1, 6)), n - sum(sizes)))
    cluster = rng.permutation(np.repeat(np.arange(len(sizes)), sizes))       # of each body
    side = int(np.ceil(len(sizes) ** (1 / 3)))
    centre = 1.0 + np.stack(np.unravel_index(np.arange(len(sizes)), (side,) * 3), axis=1)
    x = centre[cluster] + 1e-4 * rng.random((n, 3))
    dev = torch.device("cuda:0")
    pos = torch.tensor(np.ascontiguousarray(x.T), device=dev)
    s = g.System(pos, torch.zeros_like(pos), torch.full((n,), 1e-12, dtype=torch.float64, device=dev),
                 g.default_params(precision=g.GENGA_MIXED))
    s.set_rcrit(np.full(n, 1e-3))
    s.kick(0.0, precheck=True, acc_out=torch.zeros((3, n), dtype=torch.float64, device=dev))
    s.set_predrift(x.T, np.zeros((3, n)))
    npairs, ngroups, maxg = s.build_encounters()
    order = np.argsort(cluster, kind="stable")
    ends = np.cumsum(sizes)
    pairs, label = [], np.full(n, -1)
    for e, k in zip(ends, sizes):
        mem = np.sort(order[e - k:e])
        if k > 1:
            label[mem] = mem[0]
            a, b = np.triu_indices(k, 1)
            pairs.append(np.stack([mem[a], mem[b]], axis=1))
    pairs = np.concatenate(pairs) if pairs else np.zeros((0, 2), int)
    pairs = pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))]
    assert npairs == len(pairs)
    np.testing.assert_array_equal(s.pairs(0), pairs)
    np.testing.assert_array_equal(s.groups(), label)
    assert ngroups == sum(k > 1 for k in sizes) and maxg == (max(sizes) if max(sizes) > 1 else 0)
