"""The FP32 pass where its quadrature's rules change: particles whose foot on
a face plane lies next to an edge line (a long segment in units of the
distance A to the line, cut into sub-pieces), next to a vertex, or across the
foot, at kernel sizes from a cell that holds the whole support to many cells
inside it.  Against the oracle within the mixed mode's tolerance, 1e-5 |w| +
1e-14, with most pairs decided in FP32."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def dev(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-7, 1e-11])
@pytest.mark.parametrize("scale", [0.3, 1.0, 3.0])
def test_feet_next_to_edges_and_vertices(orc, eps, scale):
    rng = np.random.default_rng(11)
    g = inputs.uniform_cube(40, 60, seed=21, gen_seed=22)
    cells = orc.voronoi(g.gx, g.gy, g.gz, g.box)
    fvo, n = cells.face_vert_off, cells.normals.reshape(-1, 3)
    v = cells.verts.reshape(-1, 3)
    pts = []
    for f in rng.choice(len(fvo) - 1, 40, replace=False):
        a, b = v[fvo[f]], v[fvo[f] + 1]
        u = (b - a) / np.linalg.norm(b - a)
        m = np.cross(u, n[f])
        side = rng.choice([-1.0, 1.0], 3)
        d = 0.02 + 0.1 * rng.random()
        pts.append(a + 0.4 * (b - a) + eps * side[0] * m + d * side[1] * n[f])   # foot next to an edge
        pts.append(a + eps * (m + side[2] * u) + d * side[1] * n[f])             # next to a vertex
    p = np.clip(np.array(pts), 0.01, 0.99)
    h = scale * 0.25 * (0.5 + rng.random(len(p)))
    pairs = orc.find_pairs(p[:, 0], p[:, 1], p[:, 2], h, cells)
    wo = orc.map_exact(pairs, p[:, 0], p[:, 1], p[:, 2], h, cells)
    ctx = api.Context(0)
    vor = api.voronoi_from_cells(ctx, dev(cells.gen.reshape(-1)), dev(cells.cell_face_off, torch.int64),
                                 dev(fvo, torch.int64), dev(cells.verts.reshape(-1)), dev(cells.normals.reshape(-1)),
                                 dev(cells.nbr, torch.int64), dev(cells.volume))
    pr = api.pairs_from_list(ctx, dev(pairs.pair_i, torch.int32), dev(pairs.pair_j, torch.int32), len(p), vor)
    w, _, _, nf = api.map_exact(ctx, pr, *(dev(p[:, k]) for k in range(3)), dev(h), dev(np.ones(len(p))), vor,
                                api.Params(precision=1, fp64_threshold=1e-5))
    err = np.abs(w.cpu().numpy() - wo)
    assert pairs.n > 200 and nf < pairs.n / 2
    assert np.all(err <= 1e-5 * np.abs(wo) + 1e-14), float(np.max(err / (1e-5 * np.abs(wo) + 1e-14)))
