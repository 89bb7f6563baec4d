"""The two-pass sums of the inverse mapping and of the weights per particle
(from 2^20 pairs on) against the one-pass kernel, bit for bit: rows of 0, 1, 15,
16, 17 and 16 k + r pairs up to thousands in one warp, a last warp that is not
full, and NaN and infinities among the weights and cell values."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def sums(ctx, pr, w, f, np_):
    z = lambda: torch.zeros(np_, dtype=torch.float64, device="cuda")  # noqa: E731
    return [api.map_back(ctx, pr, w, f)[0], *api.map_back_sums(ctx, pr, w, f, z(), z())]


@pytest.mark.parametrize("special", [False, True])
def test_rows_equal_one_pass(special):
    rng = np.random.default_rng(5)
    nc, ctx = 6000, api.Context(0)
    g = inputs.uniform_cube(10, nc, seed=1, gen_seed=2)
    vor = api.build_voronoi(ctx, *(torch.as_tensor(a, device="cuda") for a in (g.gx, g.gy, g.gz)), g.box)
    rows = [0, 1, 15, 16, 17, 31, 32, 33, 6000, 47, 48, 5999] + list(rng.integers(0, 700, 2999)) + [6000] * 35
    pairs = [(j, i) for i, n in enumerate(rows) for j in rng.choice(nc, n, replace=False)]
    order = np.array(sorted(pairs), dtype=np.int32)
    i, j = (torch.as_tensor(np.ascontiguousarray(order[:, k]), device="cuda") for k in (1, 0))
    assert len(pairs) > 1 << 20
    w = torch.as_tensor(rng.random(len(pairs)) * 10.0 ** rng.uniform(-12, 0, len(pairs)), device="cuda")
    f = torch.as_tensor(rng.random(nc), device="cuda")
    if special:
        w[::100003], w[7::200003], f[5], f[9] = float("nan"), float("inf"), float("inf"), float("nan")
    got = sums(ctx, api.pairs_from_list(ctx, i, j, len(rows), vor), w, f, len(rows))
    # the same rows in lists short enough for the one-pass kernel
    for a in range(0, len(rows), 1500):
        m = (i >= a) & (i < a + 1500)
        assert int(m.sum()) < 1 << 20
        part = api.pairs_from_list(ctx, i[m].contiguous(), j[m].contiguous(), len(rows), vor)
        for x, y in zip(got, sums(ctx, part, w[m].contiguous(), f, len(rows))):
            assert np.array_equal(x[a:a + 1500].cpu().numpy().view(np.int64), y[a:a + 1500].cpu().numpy().view(np.int64))
