"""find_pairs' ordering of each cell's hits at its limits: cells with no pair,
with a few, with more than a warp's buffer (several segments), with exactly and
just over what one warp orders in shared memory (the radix sort takes over), a
first call that outgrows its buffer, and a range of cells.  The list equals the
one a sort by (cell, particle) of all pairs within reach gives, from the
oracle's test where that is affordable and otherwise from cells whose hits are
every particle."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [3, 224, 225, 256, 257, 2047, 2048, 2049, 5000])
def test_cells_holding_every_particle(n):
    """Particles whose support holds the box: every cell lists all of them."""
    rng = np.random.default_rng(n)
    p, nc = rng.random((n, 3)), 7
    g = inputs.uniform_cube(10, nc, seed=1, gen_seed=2)
    ctx = api.Context(0)
    vor = api.build_voronoi(ctx, dev(g.gx), dev(g.gy), dev(g.gz), g.box)
    pr = api.find_pairs(ctx, *(dev(p[:, k]) for k in range(3)), dev(np.full(n, 2.0)), vor)
    q = {k: v.cpu().numpy() for k, v in pr.get().items()}
    assert np.array_equal(q["pair_i"], np.tile(np.arange(n), nc))
    assert np.array_equal(q["pair_j"], np.repeat(np.arange(nc), n))
    assert np.array_equal(q["cell_pair_off"], np.arange(nc + 1) * n) and not q["near"].any()


@pytest.mark.parametrize("hscale", [0.3, 1.0, 4.0])
def test_mixed_counts_against_oracle(orc, hscale):
    w = inputs.uniform_cube(1200, 300, seed=8, gen_seed=9)
    h = w.h * hscale
    h[::50] = 0.9                 # a few supports over most of the box
    cells = orc.voronoi(w.gx, w.gy, w.gz, w.box)
    o = orc.find_pairs(w.x, w.y, w.z, h, cells)
    ctx = api.Context(0)
    vor = api.build_voronoi(ctx, dev(w.gx), dev(w.gy), dev(w.gz), w.box)
    X = [dev(a) for a in (w.x, w.y, w.z, h)]
    for pr in (api.find_pairs(ctx, *X, vor), api.find_pairs(ctx, *X, vor)):
        q = {k: v.cpu().numpy() for k, v in pr.get().items()}
        assert np.array_equal(q["pair_i"], o.pair_i) and np.array_equal(q["pair_j"], o.pair_j)
    part = api.find_pairs_cells(ctx, *X, vor, 40, 111, 16)   # a hint far too small
    q = {k: v.cpu().numpy() for k, v in part.get().items()}
    m = (o.pair_j >= 40) & (o.pair_j < 111)
    assert np.array_equal(q["pair_i"], o.pair_i[m]) and np.array_equal(q["pair_j"], o.pair_j[m])
    assert np.array_equal(q["cell_pair_off"], np.searchsorted(o.pair_j[m], np.arange(301)))
