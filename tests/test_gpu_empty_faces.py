"""Imported cells with faces of no vertices: such a face bounds nothing and is
read nowhere, so a cell with some of them maps as the cell without them, and
cells of nothing else import, hold the particles within 2h of their generator
and weigh 0."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import _native as N, api

pytestmark = pytest.mark.gpu


def dev(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.mark.parametrize("where", [(0,), (6,), (0, 0, 3, 6, 6)])
@pytest.mark.parametrize("precision", [0, 1])
def test_extra_empty_faces(orc, where, precision):
    rng = np.random.default_rng(5)
    cells = orc.cells_from_faces([orc.box_cell((0, 0, 0), (1, 0.8, 0.6))], gen=[[0.5, 0.4, 0.3]], volume=[0.48])
    fvo = np.insert(cells.face_vert_off, list(where), cells.face_vert_off[list(where)])
    normals = np.insert(cells.normals, list(where), [0.0, 0.0, 1.0], axis=0)
    p, h = rng.random((50, 3)) * 1.6 - 0.3, 0.2 + 0.5 * rng.random(50)
    X, m = [dev(p[:, k]) for k in range(3)] + [dev(h)], dev(np.ones(50))
    ctx = api.Context(0)
    out = []
    for f, n in ((cells.face_vert_off, cells.normals), (fvo, normals)):
        vor = api.voronoi_from_cells(ctx, dev(cells.gen), dev([0, len(n)], torch.int64), dev(f, torch.int64),
                                     dev(cells.verts.reshape(-1)), dev(n.reshape(-1)), None, dev(cells.volume))
        pr = api.find_pairs(ctx, *X, vor)
        w = api.map_exact(ctx, pr, *X, m, vor, api.Params(precision=precision))[0]
        c = api.voronoi_centroids(ctx, vor)
        out.append([t.cpu().numpy() for t in (pr.get()["pair_i"], w, *c)])
    a, b = out
    assert np.array_equal(a[0], b[0]) and len(a[0]) > 10
    # the mixed mode recomputes the second cell's pairs in FP64 (a face of distance 0): its own bound apart
    assert np.allclose(a[1], b[1], rtol=1e-5 if precision else 0, atol=1e-14 if precision else 0)
    assert np.allclose(a[2:], b[2:], rtol=1e-14, atol=1e-15)   # summed over the faces in another grouping


@pytest.mark.parametrize("precision", [0, 1])
def test_no_vertices_at_all(precision):
    ctx, L = api.Context(0), N.lib()
    gen = dev([[0.0, 0.0, 0.0], [4.0, 0.0, 0.0]])
    cfo, fvo = dev([0, 2, 3], torch.int64), dev([0, 0, 0, 0], torch.int64)
    verts, normals, vol = dev(np.zeros(3)), dev(np.ones(9)), dev(np.ones(2))
    h = C.c_void_p()
    ptr = [C.c_void_p(t.data_ptr()) for t in (gen, cfo, fvo, verts, normals)]
    assert L.voronoi_from_cells(ctx.handle, 2, 3, 0, *ptr, None, C.c_void_p(vol.data_ptr()), C.byref(h)) == N.EM_OK
    vor = api.Voronoi(ctx, h)
    assert vor.info() == (2, 3, 0)
    X = [dev([0.1, 0.3, 4.1, 2.0]), dev(np.zeros(4)), dev(np.zeros(4)), dev(np.full(4, 0.1))]
    pr = api.find_pairs(ctx, *X, vor)
    q = pr.get()
    assert q["pair_i"].tolist() == [0, 2] and q["pair_j"].tolist() == [0, 1]   # radius 0
    w = api.map_exact(ctx, pr, *X, dev(np.ones(4)), vor, api.Params(precision=precision))[0]
    assert w.tolist() == [0.0, 0.0]
