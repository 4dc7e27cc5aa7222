"""The large-matrix tree's Householder reduction by a cluster per node (few nodes) at last groups around its
divisions: columns dealt over 2 to 4 CTAs with remainders, the row counts where one CTA's shared memory ends,
against the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("last,cut,disp", [
    (16, [5, 3], True),          # 32 rows, 4 CTAs
    (17, [30, 2], False),        # 34 rows
    (25, [60, 1], True),         # 31 first-axis roots, 50 rows
    (29, [110, 1], False),       # 56 roots: two CTAs of 58 rows
    (58, [3, 3], True),          # 116 rows
    (59, [6, 2], False),         # 118 rows: beyond one CTA's shared memory
    (96, [2, 2], True),          # 192 rows, the largest
])
def test_cluster_reduction(cuda_lib, last, cut, disp, precision):
    gb = cuda_lib
    M = last + 3
    prob = synth.random_problem(np.random.default_rng(last), M, 1, 2, cut, displaced=disp, r_range=(0.2, 0.8))
    prob.bin_of_mode = np.array([0] * 3 + [1] * last, dtype=np.int32)
    with gb.Plan(prob, precision=precision, tile_override=13 if precision else 14) as p:
        P = p.table().cpu().numpy()
        st, d = p.diagnostics()
        lq, mp = gb.gbsbin_read_points(p.handle, d["n_evaluated"])
    assert st == 0 and mp.min() > 0
    ref = oracle.binned(prob)
    flat = np.ravel_multi_index(tuple(gb.evaluated_point_digits(prob.cutoff).T), prob.radix)
    # n = 198 at most: n eps of FP64 and n 2^-46 of pairs times a few
    assert np.abs(lq - ref["logq"].reshape(-1)[flat]).max() < (1e-11 if precision == 0 else 1e-10)
    assert np.abs(P - ref["P"]).max() < (1e-12 if precision == 0 else 1e-11)
