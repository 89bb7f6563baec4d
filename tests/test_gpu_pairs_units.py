"""find_pairs does not depend on the unit of length: a grid, its particles and
their h scaled by a power of two, which scales every FP64 step of the predicate
exactly, give the same list, also where the squares of FP32 lengths are
subnormal, zero or infinite.  (The sizes are 2^-3 to 2^1 before scaling; FP32
holds the lengths themselves for the scales here.)"""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def dev(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.fixture(scope="module")
def grid(orc):
    w = inputs.uniform_cube(900, 250, seed=21, gen_seed=22)
    h = w.h * np.where(np.arange(len(w.h)) % 3, 1.0, 0.2)
    cells = orc.voronoi(w.gx, w.gy, w.gz, w.box)
    return w, h, cells, orc.find_pairs(w.x, w.y, w.z, h, cells)


@pytest.mark.parametrize("e", [-130, -100, -80, -76, -74, -72, -68, -64, -56, -48, 0, 48, 60, 62, 63, 64, 66, 80, 110])
def test_scaled_by_a_power_of_two(grid, e):
    w, h, c, o = grid
    s = 2.0 ** e
    ctx = api.Context(0)
    gen = np.stack([w.gx, w.gy, w.gz], 1)
    vor = api.voronoi_from_cells(ctx, dev(gen.reshape(-1) * s), dev(c.cell_face_off, torch.int64),
                                 dev(c.face_vert_off, torch.int64), dev(c.verts.reshape(-1) * s),
                                 dev(c.normals.reshape(-1)), None, dev(c.volume * s ** 3))
    pr = api.find_pairs(ctx, *(dev(a * s) for a in (w.x, w.y, w.z, h)), vor)
    q = {k: v.cpu().numpy() for k, v in pr.get().items()}
    assert np.array_equal(q["pair_i"], o.pair_i) and np.array_equal(q["pair_j"], o.pair_j)
    assert not q["near"].any()
