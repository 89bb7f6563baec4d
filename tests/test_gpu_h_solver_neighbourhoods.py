"""The node h-solver on neighbourhoods that are hard on Newton's iteration:
shells of entries at 0.006 to 160 h_0 around a node, so that f' of Eq. 9 comes
near 0, iterates cross the whole bracket [1e-2 h_0, 1e2 h_0] and roots lie
anywhere in it.  Every particle is a leaf and a node of its own (leaf_max 1,
nothing closed), with its own h as h_0.  The status is the oracle's.  h after
Newton is the root to the rounding of FP64 sums, 1e-13, whatever the tolerance;
the midpoint of a bisection is the same unless a midpoint lies within that of
the root, which moves it by at most its last interval, tol h_0."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def neighbourhood(seed, k):
    rng = np.random.default_rng([seed, k])
    r = []
    for _ in range(rng.integers(1, 5)):
        rad = 10 ** (-2.2 + 4.4 * rng.random())
        m = 1 + int(10 ** (rng.random() * 2.0))
        width = 10 ** (-4 + 4 * rng.random())
        r.append(rad * (1 + width * (rng.random(m) - 0.5)))
    r = np.concatenate(r)
    v = rng.normal(size=(len(r), 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    h = 10 ** (rng.random(len(r) + 1) - 0.5)
    h[0] = 1.0
    return np.concatenate([np.zeros((1, 3)), v * r[:, None]]), h


@pytest.mark.parametrize("seed,ks,tol,max_newton", [
    (1, [8442, *range(20)], 1e-13, 50),
    (2, range(60), 1e-9, 50),
    (3, range(60), 1e-12, 8)])
def test_status_and_h(orc, seed, ks, tol, max_newton):
    ctx = api.Context(0)
    par = api.Params(theta=0.0, h_tol=tol, max_newton=max_newton)
    seen = np.zeros(3, int)
    for k in ks:
        p, h0 = neighbourhood(seed, k)
        lo, hi = p.min(0), p.max(0)
        w = (hi - lo).max() * 1e-6 + 1e-9
        tree = api.build_tree(ctx, *(dev(p[:, c]) for c in range(3)), dev(np.ones(len(p))),
                              np.stack([lo - w, hi + w], 1).reshape(-1), 1)
        ps = api.make_pseudo_particles(ctx, tree, dev(h0), lo[None] - 1e7, par)
        assert ps.info()[0] == len(p)
        i = tree.get()["perm"].long()[ps.get()["first"].long()].cpu().numpy()
        h, st = np.empty(len(p)), np.empty(len(p), np.int32)
        h[i], st[i] = ps.get()["h"].cpu().numpy(), ps.get()["status"].cpu().numpy()
        ho, so, _ = orc.h_solve(p, p, h0, 1.2, tol, max_newton)
        assert np.array_equal(st, so)
        seen += np.bincount(so, minlength=3)
        assert np.all(np.abs(h / ho - 1)[so == 0] < 1e-13)
        assert np.all(np.abs(h - ho)[so == 1] <= (tol * h0 + 1e-13 * ho)[so == 1])
        assert np.array_equal(h[so == 2], ho[so == 2])
    assert seen.min() > 0
