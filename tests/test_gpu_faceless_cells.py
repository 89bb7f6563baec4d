"""Cells without faces, as a range build leaves those outside its range: pair
finding over the whole grid lists the particles within 2h of their generators,
and every mapping gives these pairs weight 0 and the built cells' pairs the
weights that the whole grid's have."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("c0,c1", [(0, 1), (40, 90), (150, 150)])
@pytest.mark.parametrize("precision,tol", [(0, 1e-5), (1, 1e-5), (1, 0.0)])   # tol 0: nearly every pair in FP64
def test_weights_of_a_range_built_grid(c0, c1, precision, tol):
    w = inputs.uniform_cube(400, 150, seed=3, gen_seed=4)
    ctx = api.Context(0)
    X, m = [dev(a) for a in (w.x, w.y, w.z, w.h)], dev(w.m)
    par = api.Params(precision=precision, fp64_threshold=tol)
    got = []
    for vor in (api.build_voronoi(ctx, dev(w.gx), dev(w.gy), dev(w.gz), w.box),
                api.build_voronoi_cells(ctx, dev(w.gx), dev(w.gy), dev(w.gz), w.box, c0, c1)):
        pr = api.find_pairs(ctx, *X, vor)
        wt, rho = api.map_exact(ctx, pr, *X, m, vor, par)[:2]
        q = pr.get()
        got.append([t.cpu().numpy() for t in (q["pair_i"], q["pair_j"], wt, rho)])
    (ai, aj, aw, ar), (bi, bj, bw, br) = got
    sa, sb = (aj >= c0) & (aj < c1), (bj >= c0) & (bj < c1)
    assert np.array_equal(ai[sa], bi[sb]) and np.array_equal(aj[sa], bj[sb])
    assert np.array_equal(aw[sa], bw[sb]) and np.array_equal(ar[c0:c1], br[c0:c1])
    d = np.sqrt((w.x[bi] - w.gx[bj]) ** 2 + (w.y[bi] - w.gy[bj]) ** 2 + (w.z[bi] - w.gz[bj]) ** 2)
    assert np.all(d[~sb] < 2.0001 * w.h[bi[~sb]]) and (~sb).sum() > 100
    assert np.all(bw[~sb] == 0.0)
