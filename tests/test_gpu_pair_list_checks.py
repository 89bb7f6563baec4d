"""pairs_from_list refuses lists with indices out of range or out of order,
wherever they stand, and writes nothing outside the offsets while it looks:
a list made before is as it was."""
import numpy as np
import pytest
import torch

from paper_2410_15227_gb300 import _native as N, api, inputs

pytestmark = pytest.mark.gpu


def dev(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.mark.parametrize("pi,pj", [
    ([0, 1], [-5, 3]), ([0, 1, 2], [-70000, -70000, 0]), ([0, 1], [0, -1]), ([0, 1], [0, 40]), ([0, 1], [2, 1]),
    ([-2, 1], [0, 1]), ([-70000, 3], [0, 1]), ([0, 30], [0, 1]), ([3, 3], [1, 1]), ([2 ** 31 - 1, 0], [0, 1])])
def test_refused(pi, pj):
    w = inputs.uniform_cube(30, 40, seed=3, gen_seed=4)
    ctx = api.Context(0)
    vor = api.build_voronoi(ctx, dev(w.gx), dev(w.gy), dev(w.gz), w.box)
    good = api.pairs_from_list(ctx, dev([5, 7, 5], torch.int32), dev([0, 0, 39], torch.int32), 30, vor)
    before = {k: v.cpu().numpy() for k, v in good.get().items()}
    with pytest.raises(N.NativeError) as e:
        api.pairs_from_list(ctx, dev(pi, torch.int32), dev(pj, torch.int32), 30, vor)
    assert e.value.status == N.EM_EINVAL
    assert before["cell_pair_off"].tolist() == [0] + [2] * 39 + [3]
    assert all(np.array_equal(before[k], v.cpu().numpy()) for k, v in good.get().items())
