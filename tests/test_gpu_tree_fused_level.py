"""The small tree's first level within the second's launch or apart, by the number of children that would repeat it,
against the oracle point by point."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disp", [False, True])
@pytest.mark.parametrize("sizes,cut,precision,together", [
    ([4, 4, 4], [8, 8, 2], 0, True),                     # 81 children, one turn of the SMs
    ([4, 4, 4], [39, 39, 1], 0, False),                  # 1600
    ([4, 4, 4], [39, 39, 1], 1, False),
    ([4, 4, 4], [15, 15, 2], 1, True),                   # 256
    ([2, 2, 2], [26, 26, 2], 1, True),                   # 729: both levels by one elimination
    ([6, 6, 6], [2, 2, 2], 0, False),                    # 12 rows: their sums outweigh a launch
    ([4, 4, 4, 4], [2, 2, 2, 2], 1, True),               # second and third level in one launch
    ([4, 4, 4, 4], [20, 21, 2, 1], 1, False),
])
def test_first_level_within_the_second(cuda_lib, sizes, cut, precision, together, disp):
    gb = cuda_lib
    M, L = sum(sizes), len(sizes)
    prob = synth.random_problem(np.random.default_rng(50 + M), M, 1, L, cut, displaced=disp, r_range=(0.2, 1.0))
    prob.bin_of_mode = np.repeat(np.arange(L), sizes).astype(np.int32)
    with gb.Plan(prob, precision=precision) as p:
        P = p.table().cpu().numpy()
        st, d = p.diagnostics()
        lq, mp = gb.gbsbin_read_points(p.handle, d["n_evaluated"])
    assert st == 0 and mp.min() > 0
    # the levels after the first (merged where few), leaves, transform
    levels = 2 if tuple(cut) == (20, 21, 2, 1) else 1
    assert d["launches"] == levels + 2 + (0 if together else 1)
    ref = oracle.binned(prob)
    flat = np.ravel_multi_index(tuple(gb.evaluated_point_digits(prob.cutoff).T), prob.radix)
    # log q is a sum of n logarithms of factors within [1e-2, 2]: n eps of FP64, n 2^-46 of pairs, some tens over
    assert np.abs(lq - ref["logq"].reshape(-1)[flat]).max() < (1e-12 if precision == 0 else 1e-10)
    assert np.abs(P - ref["P"]).max() < (1e-13 if precision == 0 else 1e-11)
