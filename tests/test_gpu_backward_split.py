"""The tree's reverse pass with few parents: their products and assembly split by columns over several
CTAs and small blocks updated entry by entry, against the per-point reverse pass.  Column counts that
the splits do not divide and blocks with partly filled panels.

Tolerance: n * 30 * 2^-46 = 3e-11 relative to the largest entry (n = 66, |inv(M)| < 30 for these
squeezings, pairs of FP32 the coarser arithmetic), taken as 1e-10 as for the larger shapes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32pairs"])
@pytest.mark.parametrize("sizes,cutoff", [([20, 13], [4, 6]), ([26, 9], [2, 9]), ([11, 12, 11], [2, 3, 5])],
                         ids=["40+26", "52+18", "22+24+22"])
def test_split_reverse_pass_matches_per_point(cuda_lib, sizes, cutoff, precision):
    import torch
    gb = cuda_lib
    rng = np.random.default_rng(5200 + sizes[0])
    prob = synth.random_problem(rng, sum(sizes), 1, len(sizes), cutoff, displaced=True)
    prob.bin_of_mode = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    pbar = rng.standard_normal(tuple(int(c) + 1 for c in prob.cutoff))
    out = []
    for tile, path in ((0, 2), (6 if precision else 3, 1)):
        with gb.Plan(prob, precision=precision, want_backward=True, tile_override=tile) as p:
            p.table()
            g = p.backward(torch.from_numpy(pbar).cuda(), want=("r", "T", "alpha", "sigma1", "zbar"))
            st, d = p.diagnostics()
            assert st == 0 and d["backward_path"] == path
        out.append(g)
    for k in ("r", "T", "alpha", "sigma1", "zbar"):
        scale = max(1.0, float(np.abs(out[1][k]).max()))
        assert np.abs(out[0][k] - out[1][k]).max() < 1e-10 * scale, k
