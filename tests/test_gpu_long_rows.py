"""The sums of the inverse mapping and of the weights per particle at the limits
of their split by row length: rows of one thread's length and just beyond, around
a tile of a long row, of just under and over the length from which a block takes
few, none or whole groups of each kind, many rows per class, in one launch (below
2^20 pairs) and in two; against the sums in order on the host, bit for bit, with
infinities and NaN among the weights and cell values."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu

NC = 6000
EDGE = [0, 1, 2, 3, 4, 5, 95, 96, 97, 98, 107, 108, 109, 119, 120, 121, 131, 132, 133, 1085, 1086, 1087, 1088, 1152, 1153,
        2999, 3000, 6000, 0]
ROWS = {
    "edges": EDGE,
    "one": [97],
    "no long": [96] * 70 + [0, 5],
    "32 long": [200] * 32 + [1] * 100,
    "33 long, shuffled": list(np.random.default_rng(1).permutation([130] * 33 + [96] * 200 + [7] * 31)),
    "8 very long": [1500] * 8 + [100] * 31,
    "9 very long": [40] * 40 + [1500] * 9 + [100] * 33,
    "a thread per row": [1] * 3000 + [0, 97, 2000, 2, 3, 1500],
    "every length": list(np.random.default_rng(2).permutation(np.arange(0, 700))),
    "two launches": EDGE * 20 + list(np.random.default_rng(3).integers(0, 1500, 1200)),
    "two launches, short": [6] * 200000,
}


@pytest.mark.parametrize("kind", ROWS)
@pytest.mark.parametrize("special", [False, True])
def test_sums_in_order(kind, special):
    rng = np.random.default_rng(7)
    rows = np.array(ROWS[kind], dtype=np.int64)
    ctx, n = api.Context(0), len(rows)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    g = inputs.uniform_cube(10, NC, seed=1, gen_seed=2)
    vor = api.build_voronoi(ctx, dev(g.gx), dev(g.gy), dev(g.gz), g.box)
    # a row's cells: a stride through the cells from a random start, distinct
    i = np.repeat(np.arange(n), rows)
    t = np.arange(len(i)) - np.repeat(np.cumsum(rows) - rows, rows)
    j = (rng.integers(0, NC, n)[i] + 7 * t) % NC
    order = np.lexsort((j, i))   # the rows in ascending cell, row by row
    i, j = i[order], j[order]
    w = rng.random(len(i)) * 10.0 ** rng.uniform(-12, 0, len(i))
    f = rng.random(NC)
    if special:
        w[::50021], w[7::80021], f[5], f[9] = np.nan, np.inf, np.inf, np.nan
    num, den = np.zeros(n), np.zeros(n)
    at = np.concatenate([[0], np.cumsum(rows)])
    with np.errstate(invalid="ignore"):
        for r in np.nonzero(rows)[0]:   # cumsum adds in order
            s = slice(at[r], at[r + 1])
            num[r], den[r] = np.cumsum(w[s] * f[j[s]])[-1], np.cumsum(w[s])[-1]
        want = [num / den, num, den, 1.0 + num, 2.0 + den]
    ji = np.lexsort((i, j))
    pr = api.pairs_from_list(ctx, dev(i[ji].astype(np.int32)), dev(j[ji].astype(np.int32)), n, vor)
    W, F = dev(w[ji]), dev(f)
    z = lambda v: torch.full((n,), v, dtype=torch.float64, device="cuda")  # noqa: E731
    got = [api.map_back(ctx, pr, W, F)[0], *api.map_back_sums(ctx, pr, W, F, z(0.0), z(0.0)),
           *api.map_back_sums(ctx, pr, W, F, z(1.0), z(2.0))]
    for x, y in zip(got, want):
        x = x.cpu().numpy()
        assert np.array_equal(np.isnan(x), np.isnan(y))
        assert np.array_equal(x[~np.isnan(y)].view(np.int64), y[~np.isnan(y)].view(np.int64))
