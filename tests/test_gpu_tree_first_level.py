"""The small tree's first level by elimination and from the spectral form, as the plan's sizes decide: a state's upload
holds the spectral form only where a table gains what the decomposition costs the host, and both forms agree with the
oracle, at the plan's first state and after set_state."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _problem(seed, bins, cut, disp):
    prob = synth.random_problem(np.random.default_rng(seed), len(bins), 1, len(cut), cut, displaced=disp, r_range=(0.2, 1.0))
    prob.bin_of_mode = np.array(bins, dtype=np.int32)
    return prob


@pytest.mark.parametrize("disp", [False, True])
@pytest.mark.parametrize("bins,cut,precision,spectral", [
    ([0] * 24 + [1] * 8, [5, 2], 0, False),              # 48 of 64 rows: 0.19 ms of host for 0.11 of the table
    ([0] * 24 + [1] * 8, [5, 2], 1, False),
    ([0] * 24 + [1] * 8, [199, 1], 0, True),             # two turns of the SMs, eigenvalues in two rounds of the path record
    ([0] * 24 + [1] * 8, [799, 1], 1, True),
    ([0] * 12 + [1] * 4, [4, 4], 0, False),              # 24 of 32 rows: 28 us for 20
    ([0] * 8 + [1] * 8, [4, 4], 1, False),               # 16 of 32 rows in pairs: 14 us for 6
    ([0] * 8 + [1] * 8, [4, 4], 0, True),                # in FP64 15
    ([0] * 7 + [1] * 7 + [2] * 7, [3, 2, 2], 0, True),
    ([0] * 7 + [1] * 7 + [2] * 7, [3, 2, 2], 1, False),
    ([0] * 4 + [1] * 4 + [2] * 4 + [3] * 4, [2, 2, 1, 2], 1, True),
    ([0] * 8 + [1] * 8 + [2] * 8, [19, 17, 1], 1, True),   # 360 children: three turns of the SMs
])
def test_first_level_form(cuda_lib, bins, cut, precision, spectral, disp):
    gb = cuda_lib
    a, b = _problem(31, bins, cut, disp), _problem(32, bins, cut, disp)
    n = 2 * len(bins)
    with gb.Plan(a, precision=precision) as p:
        for prob in (a, b):
            gb.gbsbin_plan_set_state(p.handle, prob)
            P = p.table().cpu().numpy()
            st, d = p.diagnostics()
            lq, mp = gb.gbsbin_read_points(p.handle, d["n_evaluated"])
            assert st == 0 and d["kernel_name"] == ("tree_df32" if precision else "tree_fp64") and mp.min() > 0
            # 16 bytes a slot: the permuted state alone is n^2 + 2 n + 3 of them (rounded up to 256 bytes)
            assert (d["state_upload_bytes"] > 16 * (n * n + 2 * n + 3) + 256) == spectral
            ref = oracle.binned(prob)
            flat = np.ravel_multi_index(tuple(gb.evaluated_point_digits(prob.cutoff).T), prob.radix)
            # log q is a sum of n logarithms of factors within [1e-2, 2]: n eps of FP64, n 2^-46 of pairs, some tens over
            assert np.abs(lq - ref["logq"].reshape(-1)[flat]).max() < (1e-12 if precision == 0 else 1e-10)
            assert np.abs(P - ref["P"]).max() < (1e-13 if precision == 0 else 1e-11)
