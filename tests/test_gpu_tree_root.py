"""The small tree's first level from the spectral form of the first group's block, apart and within the second
level's launch, at the block sizes where its teams and butterflies change, against the oracle point by point."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("disp", [False, True])
@pytest.mark.parametrize("bins,cut", [
    ([0, 1], [1, 1]),                                    # n = 4: one-row pairs, the smallest tree
    ([0] * 24 + [1] * 8, [5, 2]),                        # n = 64, a first block of 48 rows: two rounds of the path record
    ([0] * 17 + [1] * 2 + [2] * 3, [3, 4, 2]),           # 34 rows, then 4 and 6
    ([0] + [1] * 9 + [2] * 2 + [3] * 2, [2, 1, 3, 2]),   # a first block of 2 rows before 18
    ([2, 0, 1, 0, 2, 1, 0, 2], [4, 0, 3]),               # interleaved groups, a one-point axis
])
def test_first_level(cuda_lib, bins, cut, disp, precision):
    gb = cuda_lib
    M, L = len(bins), len(cut)
    prob = synth.random_problem(np.random.default_rng(1000 + M + L), M, 1, L, cut, displaced=disp, r_range=(0.2, 1.0))
    prob.bin_of_mode = np.array(bins, dtype=np.int32)
    with gb.Plan(prob, precision=precision) as p:
        P = p.table().cpu().numpy()
        st, d = p.diagnostics()
        lq, mp = gb.gbsbin_read_points(p.handle, d["n_evaluated"])
    assert st == 0 and d["kernel_name"] == ("tree_df32" if precision else "tree_fp64") and mp.min() > 0
    ref = oracle.binned(prob)
    dig = gb.evaluated_point_digits(prob.cutoff)
    flat = np.ravel_multi_index(tuple(dig.T), prob.radix)
    # log q is a sum of n logarithms of factors within [1e-2, 2]: n eps of FP64, n 2^-46 of pairs, some tens over
    assert np.abs(lq - ref["logq"].reshape(-1)[flat]).max() < (1e-12 if precision == 0 else 1e-10)
    assert np.abs(P - ref["P"]).max() < (1e-13 if precision == 0 else 1e-11)
