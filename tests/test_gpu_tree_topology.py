"""The octree built in one pass over the sorted keys, at the sizes where its
rules meet their ends: fewer particles than a window of leaf_max + 1, exactly
one window, runs of identical keys (nodes of every level down to the deepest),
leaf_max 1 and 64, and nodes on both sides of the size kernels' limits (32 and
1024 particles).  Every array of the tree equals the oracle's."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("leaf_max", [1, 3, 8, 64])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 33, 64, 65, 1500, 5000])
def test_tree_equals_oracle(orc, n, leaf_max):
    rng = np.random.default_rng(n)
    p = rng.random((n, 3))
    if n >= 1500:   # duplicates, near duplicates, clusters
        p[:70] = p[0]
        p[70:80] = p[71] + 1e-7 * rng.random((10, 3))
        p[100:1200] = 0.3 + 1e-4 * rng.random((1100, 3))
    box = np.array([0.0, 1.0, 0.0, 1.0, 0.0, 1.0])
    m = 0.5 + rng.random(n)
    to = orc.build_tree(p[:, 0], p[:, 1], p[:, 2], m, box, leaf_max)
    tg = api.build_tree(api.Context(0), *(dev(p[:, k]) for k in range(3)), dev(m), box, leaf_max)
    g = {k: v.cpu().numpy() for k, v in tg.get().items()}
    assert tg.info() == (n, to.nnode, int(to.level.max()))
    assert np.array_equal(g["label"].astype(np.uint64), to.label)
    for k in ("perm", "level", "parent", "first", "count", "nchild", "mass", "com", "size"):
        assert np.array_equal(g[k], getattr(to, k)), k
    assert np.array_equal(g["first_child"], np.where(to.nchild > 0, to.first_child, -1))
