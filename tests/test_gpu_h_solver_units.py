"""make_pseudo_particles does not depend on the unit of length: a cloud, its h,
its source and the two radii scaled by a power of two, which scales every FP64
step exactly, give the oracle's statuses and h, also where FP32 squares of the
lengths are subnormal, zero or infinite and outside the range of h_0 in which
the FP32 approach is used (2^-49 to 2^49)."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import api

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def cloud():
    rng = np.random.default_rng(23)
    c = rng.random((30, 3))
    return np.concatenate([rng.random((900, 3)), *(a + 3e-3 * rng.random((30, 3)) for a in c)])


@pytest.fixture(scope="module")
def ref(orc):
    p = cloud()
    m, h, box = np.full(len(p), 1.0 / len(p)), np.full(len(p), 0.05), np.array([-0.01, 1.01] * 3)
    src = np.array([[0.5, 0.5, 0.5]])
    return p, m, h, box, src, orc.make_pseudo_particles(*p.T, m, h, box, src, 0.05, 0.1, 0.4, h_fact=1.2, tol=1e-13)[0]


@pytest.mark.parametrize("e", [-100, -78, -74, -70, -66, -62, -56, -48, 0, 44, 52, 58, 62, 63, 64, 66, 70, 100])
def test_scaled_by_a_power_of_two(ref, e):
    p, m, h, box, src, o = ref
    s = 2.0 ** e
    ctx = api.Context(0)
    tree = api.build_tree(ctx, *(dev(p[:, k] * s) for k in range(3)), dev(m), box * s, 8)
    ps = api.make_pseudo_particles(ctx, tree, dev(h * s), src * s,
                                   api.Params(theta=0.4, h_tol=1e-13, r_part=0.05 * s, r_leaf=0.1 * s))
    g = {k: v.cpu().numpy() for k, v in ps.get().items()}
    assert np.array_equal(g["origin"], o.origin) and np.array_equal(g["status"], o.status)
    assert set(o.status) >= {0, 1}
    # the root to the rounding of FP64 sums; a bisection's midpoint by at most
    # its last interval (tol h_0, h_0 <= 100 h) besides
    assert np.all(np.abs(g["h"] / s / o.h - 1) <= np.where(o.status == 1, 1e-11, 1e-13))
