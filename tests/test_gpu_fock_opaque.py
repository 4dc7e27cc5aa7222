"""Fock inputs through a nearly opaque circuit: most states' entries lie far below their columns' largest, so that their
products come from low digits alone."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,states", [(12, 3, 924), (14, 2, 3432), (16, 2, 12870), (18, 2, 48620)])
def test_pairs_against_fp64(cuda_lib, N, L, states):
    fp = synth.random_fock_problem(np.random.default_rng(N), N + 4, [1] * N + [0] * 4, L, N, eta_range=(0.02, 0.05))
    tables = []
    for precision in (0, 1):
        with cuda_lib.FockPlan(fp, precision=precision) as p:
            tables.append(p.table().cpu().numpy())
            assert p.diagnostics()["launches"] > 2, "the rule did not take the convolution"
    # a dropped lo x lo is below 2^-58 of its columns' largest entries, these below 1: two in a component, one for each
    # state, and a result takes two pairs of columns at most at this size
    assert np.abs(tables[1] - tables[0]).max() < states * 2.0 ** -56
