"""Heralded states along the tree of block eliminations at the sizes its branches turn on: one group (spectral form
alone), more groups than one level launch of the tables takes, no traced modes, coefficients beyond shared memory,
grids whose first two axes do not fit it, even radices; against the oracle."""
import numpy as np
import pytest

import synth
from oracle import herald

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,roles,cutoff,cut,over,disp", [
    ("one_group_traced", [0, -1, 0, -2, -1], [3], 3, 2, True),
    ("one_group_only_kept_left", [0, -2], [4], 4, 1, False),
    ("six_groups", [0, 1, 2, -2, 3, 4, 5, -1], [1, 0, 1, 1, 2, 1], 2, 1, True),
    ("coefficients_in_global", [0, -2, -2], [2], 9, 1, True),
    ("wide_axes", [0, 1, -2], [79, 77], 1, 1, True),
    ("even_radices_three", [0, 0, 1, 2, -2, -1], [3, 1, 5], 2, 1, False),
    ("four_kept", [0, -2, -2, -2, -2], [1], 1, 1, True),
])
def test_herald_branches(cuda_lib, name, roles, cutoff, cut, over, disp):
    prob = synth.random_problem(np.random.default_rng(len(name)), len(roles), 1, 1, [1], displaced=disp,
                                r_range=(0.2, 0.8))
    ref, pr_ref = herald.table(prob, roles, cutoff, cut, oversample=over)
    with cuda_lib.HeraldPlan(prob, roles, cutoff, cut, oversample=over) as h:
        rho, pr = (x.cpu().numpy() for x in h.states())
        d = h.diagnostics()
    assert d["status"] == 0 and d["n_bad_points"] == 0
    # entries below 1, eliminations of at most 16 rows: some tens of eps
    assert np.abs(rho - ref).max() < 1e-13 and np.abs(pr - pr_ref).max() < 1e-13
