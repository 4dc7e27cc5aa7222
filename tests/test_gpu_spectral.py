"""The one-group kernel (spectral form of XA, O(n) per grid point) where its lanes-per-point rule changes
and at the smallest matrix, against the oracle's eigenvalue-free LU at sampled points and numpy's FFT."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disp", [False, True])
@pytest.mark.parametrize("M,points", [(1, 2), (1, 3), (17, 2431), (17, 2433), (17, 19455), (17, 19457), (65, 31)])
def test_lanes_per_point(cuda_lib, M, points, disp):
    # 1216 and 9728 evaluated points are the last of 32 and of 8 lanes per point on 152 SMs; n = 2, 34 and
    # 130 leave lanes without a factor, or with one more than others.  log q: ~n roundings of a sum whose
    # terms are below 10, under 1e-12; the table: eps times |log q| of an entry below 1
    gb = cuda_lib
    prob = synth.random_problem(np.random.default_rng(points + M), M, 1, 1, points - 1, displaced=disp,
                                r_range=(0.2, 0.9))
    with gb.Plan(prob) as p:
        P = p.table().cpu().numpy()
        st, d = p.diagnostics()
        lq, mp = gb.gbsbin_read_points(p.handle, d["n_evaluated"])
    assert st == 0 and d["n_bad_points"] == 0 and d["min_pivot_re"] > 0 and np.all(mp > 0)
    assert d["min_pivot_re"] == mp.min()
    XA, gamma, labels = oracle.plan(prob)
    dig = gb.evaluated_point_digits(prob.cutoff)
    pick = np.unique(np.concatenate([[0, len(dig) - 1], np.random.default_rng(1).integers(0, len(dig), 12)]))
    ref, _, _ = oracle.logq_points(XA, gamma, labels, prob.radix, dig[pick])
    assert np.abs(lq[pick] - ref).max() < 1e-12
    assert abs(d["log_q1_re"] - lq[0].real) < 1e-12
    G = np.exp(lq - lq[0])
    assert np.abs(P - np.fft.hfft(G, n=points) / points).max() < 1e-13
