"""Heralded states whose first axis is so long that one matrix per root would not fit the plan's memory: every point then
sweeps all groups itself. The same state with its groups in another order, the long axis last, has the same tables."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

LONG = 60000                                             # x (94 x 96 + 3) x 16 bytes of depth 1: above 8 GiB


@pytest.mark.parametrize("sizes,cutoff,disp", [([1, 46], [LONG - 1, 0], False), ([1, 40, 6], [LONG - 1, 0, 1], True)])
def test_long_first_axis(cuda_lib, sizes, cutoff, disp):
    M, L = sum(sizes) + 1, len(sizes)
    prob = synth.random_problem(np.random.default_rng(L), M, 1, 1, [1], displaced=disp, r_range=(0.2, 0.8))
    roles = np.concatenate([np.repeat(np.arange(L), sizes), [-2]])
    with cuda_lib.HeraldPlan(prob, roles, cutoff, 0) as h:
        rho, pr = (x.cpu().numpy() for x in h.states())
        d = h.diagnostics()
    order = list(range(1, L)) + [0]                      # new group i is old group order[i]
    back = np.argsort(order)
    with cuda_lib.HeraldPlan(prob, np.where(roles < 0, roles, back[roles]), [cutoff[o] for o in order], 0) as h:
        rho2, pr2 = (x.cpu().numpy() for x in h.states())
        d2 = h.diagnostics()
    assert d["status"] == 0 and d2["status"] == 0 and d["n_bad_points"] == 0
    assert d["launches"] == 1 + L                        # the points and a transform per axis, no first level's launch
    axes = [order.index(l) for l in range(L)]
    # entries below 1 from eliminations of 96 rows: some hundreds of eps
    assert np.abs(rho - rho2.transpose(*axes, L, L + 1)).max() < 1e-13
    assert np.abs(pr - pr2.transpose(axes)).max() < 1e-13
    assert pr.sum() > 0.1
