"""The reverse pass along the large-matrix tree with its leaves inverted in the Hessenberg basis of
each parent's Schur complement (last axes of many roots), against the per-point reverse pass (one
n x n Gauss-Jordan inverse per evaluated point) on the same state.

Tolerance: both passes invert matrices with |inv(M)| <= 1 / (1 - |XA|) (under 30 for these
squeezings) in arithmetic of unit 2^-46 (pairs) or 2^-53, with sums of up to n = 232 terms: relative
to the largest entry n * 30 * 2^-46 = 1e-10 at most, for either arithmetic's gradient."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _grads(gb, prob, pbar, precision, tile):
    import torch
    with gb.Plan(prob, precision=precision, want_backward=True, tile_override=tile) as p:
        p.table()
        g = p.backward(torch.from_numpy(pbar).cuda(), want=("r", "T", "alpha", "V", "sigma1", "zbar"))
        st, d = p.diagnostics()
        assert st == 0
    return g, d


CASES = [
    # rows of the last group, and what they reach: 100 (a block column of 4), 34 (one of 2, two slots of the
    # row), 64 (whole blocks, eight lanes a row), 116 (the largest; one CTA per SM); leaves of one parent over
    # several CTAs and several parents in one CTA, more parents than SMs, no displacement
    ("l2_100", 100, 2, [44, 60], [50, 50], True),
    ("l2_100_plain", 100, 2, [200, 24], [50, 50], False),
    ("l3_34", 61, 3, [10, 12, 24], [22, 22, 17], True),
    ("l2_64", 70, 2, [50, 49], [38, 32], True),
    ("l2_116", 116, 2, [40, 60], [58, 58], True),
]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32pairs"])
@pytest.mark.parametrize("name,M,L,cutoff,sizes,displaced", CASES, ids=[c[0] for c in CASES])
def test_hessenberg_leaves_match_per_point(cuda_lib, name, M, L, cutoff, sizes, displaced, precision):
    gb = cuda_lib
    rng = np.random.default_rng(4100 + M + L)
    prob = synth.random_problem(rng, M, 1, L, cutoff, displaced=displaced)
    prob.bin_of_mode = np.repeat(np.arange(L), sizes).astype(np.int32)
    pbar = rng.standard_normal(tuple(int(c) + 1 for c in prob.cutoff))
    gt, dt = _grads(gb, prob, pbar, precision, 0)
    gp, dp = _grads(gb, prob, pbar, precision, 6 if precision else 3)
    assert dt["backward_path"] == 2 and dp["backward_path"] == 1
    for k in gt:
        if gt[k] is None:
            continue
        scale = max(1.0, float(np.abs(gp[k]).max()))
        assert np.abs(gt[k] - gp[k]).max() < 1e-10 * scale, (name, k, np.abs(gt[k] - gp[k]).max(), scale)
