"""The one-pass sums of the inverse mapping and of short pair lists, by eight
lanes per particle (rows of eight pairs or more on average) and by a thread per
particle, against the same sums in order on the host, bit for bit: rows of 0, 1
and around multiples of 8 and 32, a last warp that is not full, and infinities
among the weights and cell values."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [
    [0, 1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 0, 300, 24, 40, 127, 2],   # lanes
    [100],                                                            # lanes, one row
    [0, 1, 7, 8, 9, 0, 3, 2, 1, 33, 0, 0, 5],                          # a thread per row
])
@pytest.mark.parametrize("special", [False, True])
def test_rows_equal_sums_in_order(rows, special):
    rng = np.random.default_rng(3)
    nc, n, ctx = 400, len(rows), api.Context(0)
    g = inputs.uniform_cube(10, nc, seed=1, gen_seed=2)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    vor = api.build_voronoi(ctx, dev(g.gx), dev(g.gy), dev(g.gz), g.box)
    pairs = np.array(sorted((j, i) for i, m in enumerate(rows) for j in rng.choice(nc, m, replace=False)), dtype=np.int32)
    pi, pj = pairs[:, 1], pairs[:, 0]
    w = rng.random(len(pi)) * 10.0 ** rng.uniform(-12, 0, len(pi))
    f = rng.random(nc)
    if special:
        w[::37], f[::41] = np.inf, -np.inf
    num, den = np.zeros(n), np.zeros(n)
    with np.errstate(invalid="ignore"):
        for k in range(len(pi)):   # ascending cell: the order of the sums
            num[pi[k]] += w[k] * f[pj[k]]
            den[pi[k]] += w[k]
        want = [num / den, num, den]
    pr = api.pairs_from_list(ctx, dev(pi), dev(pj), n, vor)
    z = lambda: torch.zeros(n, dtype=torch.float64, device="cuda")  # noqa: E731
    got = [api.map_back(ctx, pr, dev(w), dev(f))[0], *api.map_back_sums(ctx, pr, dev(w), dev(f), z(), z())]
    for x, y in zip(got, want):
        x = x.cpu().numpy()
        assert np.array_equal(np.isnan(x), np.isnan(y))
        assert np.array_equal(x[~np.isnan(y)].view(np.int64), y[~np.isnan(y)].view(np.int64))
