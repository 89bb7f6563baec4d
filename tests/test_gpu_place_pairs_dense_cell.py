"""find_pairs where one cell holds more hits than a warp orders in shared memory
(2,048) and the others hold few: the radix sort orders the whole list; a range
of cells without the dense one is placed per cell, one with it is sorted; all
give the same list."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("ndense", [2047, 2048, 2049, 3000])
def test_one_dense_cell(orc, ndense):
    w = inputs.uniform_cube(1500, 200, seed=31, gen_seed=32)
    rng = np.random.default_rng(33)
    g = np.array([w.gx[77], w.gy[77], w.gz[77]])
    cells = orc.voronoi(w.gx, w.gy, w.gz, w.box)
    base = orc.find_pairs(w.x, w.y, w.z, w.h, cells)
    here = int((base.pair_j == 77).sum())
    p = np.concatenate([np.stack([w.x, w.y, w.z], 1), g + 1e-4 * rng.random((ndense - here, 3))])
    h = np.concatenate([w.h, np.full(ndense - here, 1e-4)])
    perm = rng.permutation(len(h))
    p, h = p[perm], h[perm]
    o = orc.find_pairs(*p.T, h, cells)
    assert np.bincount(o.pair_j, minlength=200).max() == ndense
    ctx = api.Context(0)
    vor = api.build_voronoi(ctx, dev(w.gx), dev(w.gy), dev(w.gz), w.box)
    X = [dev(p[:, k]) for k in range(3)] + [dev(h)]
    for c0, c1 in ((0, 200), (0, 77), (70, 80), (78, 200)):
        pr = api.find_pairs_cells(ctx, *X, vor, c0, c1, 0)
        q = {k: v.cpu().numpy() for k, v in pr.get().items()}
        m = (o.pair_j >= c0) & (o.pair_j < c1)
        assert np.array_equal(q["pair_i"], o.pair_i[m]) and np.array_equal(q["pair_j"], o.pair_j[m])
        assert np.array_equal(q["cell_pair_off"], np.searchsorted(o.pair_j[m], np.arange(201)))
