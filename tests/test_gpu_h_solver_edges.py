"""The node h-solver where its FP32 approach hands over: populations too small
for a root (h_0), nodes without neighbours inside 2 h_0 (bisection), more
neighbours inside 2 h_0 than a warp's list holds, a core of leaves inside the
2h of every node around it (solved by teams of warps), and coordinates far from
the origin.  Status and h as the oracle's, whose evaluations are all FP64; at a
tolerance just above and just below the one from which the FP32 approach is
used, the same statuses."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def cloud(kind):
    rng = np.random.default_rng(17)
    if kind == "few":                     # fewer than pi h_fact^3 = 5.4 entries: no root
        return rng.random((5, 3)) * np.array([1.0, 0.1, 0.1])
    if kind == "clusters":                # nodes far apart: Newton leaves the bracket at once
        return np.concatenate([c + 1e-3 * rng.random((40, 3)) for c in rng.random((60, 3))])
    if kind == "pairs":                   # tight pairs: h_0 far below the spacing
        c = rng.random((300, 3))
        return np.concatenate([c, c + 1e-6 * rng.random((300, 3))])
    if kind == "dense":                   # large nodes over a dense core: long lists
        v = rng.normal(size=(6000, 3))
        return v / np.linalg.norm(v, axis=1, keepdims=True) * (rng.random(6000) ** 2)[:, None]
    if kind == "core":                    # 60,000 particles' leaves within 2h of 400 outer nodes
        v = rng.normal(size=(60400, 3))
        r = np.concatenate([0.04 * rng.random(60000) ** (1 / 3), 0.3 + 0.7 * rng.random(400)])
        return v / np.linalg.norm(v, axis=1, keepdims=True) * r[:, None]
    return 1000.0 + rng.random((3000, 3))   # "far"


@pytest.mark.parametrize("kind", ["few", "clusters", "pairs", "dense", "core", "far"])
@pytest.mark.parametrize("theta", [0.3, 1.5])
@pytest.mark.parametrize("tol", [1e-13, 9.9e-10, 1.1e-9])
def test_status_and_h(orc, kind, theta, tol):
    p = cloud(kind)
    lo, hi = p.min(0), p.max(0)
    box = np.stack([lo - 0.01, hi + 0.01], 1).reshape(-1)
    m, h = np.full(len(p), 1.0 / len(p)), np.full(len(p), 0.05)
    src = lo[None] - 0.3 if kind != "core" else np.zeros((1, 3))
    o, _, _ = orc.make_pseudo_particles(p[:, 0], p[:, 1], p[:, 2], m, h, box, src, 0.05, 0.1, theta, h_fact=1.2,
                                        tol=tol)
    ctx = api.Context(0)
    tree = api.build_tree(ctx, *(dev(p[:, k]) for k in range(3)), dev(m), box, 8)
    ps = api.make_pseudo_particles(ctx, tree, dev(h), src, api.Params(theta=theta, h_tol=tol))
    g = {k: v.cpu().numpy() for k, v in ps.get().items()}
    assert np.array_equal(g["origin"], o.origin)
    assert np.array_equal(g["status"], o.status)
    # Newton ends converged; a bisection's midpoint is the same unless a sign
    # next to the root differs, which moves it by at most its last interval
    rel = np.abs(g["h"] / o.h - 1)
    assert np.all(rel[o.status == 0] < max(1e-12, 3 * tol))
    assert np.all(np.abs(g["h"] - o.h)[o.status == 1] <= 1e-12 * o.h[o.status == 1] + tol * 1.0)
    assert np.array_equal(g["h"][o.status >= 2], o.h[o.status >= 2])
