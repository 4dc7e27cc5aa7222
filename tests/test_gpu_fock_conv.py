"""Fock inputs by the convolution over sub-multisets against the node walk (kernel 9 asked for by name), over
the forms the rule sends there: odd and even photon numbers, repeated photons, one to four groups, folded and
oversampled grids, shuffled groups, a lossless and a nearly opaque circuit, a permutation (most states zero)."""
import numpy as np
import pytest

import synth
from oracle import fock

pytestmark = pytest.mark.gpu


def _cases():
    rng = np.random.default_rng(4242)
    c = {
        "even_l3": (synth.random_fock_problem(rng, 16, [1] * 12 + [0] * 4, 3, 12), 1),
        "odd_l2": (synth.random_fock_problem(rng, 15, [1] * 15, 2, 15, shuffle_bins=True), 1),
        "repeated_l2": (synth.random_fock_problem(rng, 9, [3, 0, 2, 2, 1, 3, 2, 3, 1], 2, 17), 1),
        "folded_l3": (synth.random_fock_problem(rng, 14, [1] * 13 + [0], 3, [5, 13, 7]), 1),
        "oversampled_l2": (synth.random_fock_problem(rng, 13, [1] * 13, 2, 8), 2),
        "l4": (synth.random_fock_problem(rng, 11, [1] * 9 + [2, 0], 4, [6, 5, 7, 6], shuffle_bins=True), 1),
        "l1": (synth.random_fock_problem(rng, 18, [1] * 18, 1, 18), 1),
    }
    fp = synth.random_fock_problem(rng, 12, [1] * 12, 3, 12)
    fp.T = synth.haar_unitary(12, rng)
    c["lossless"] = (fp, 1)
    fp = synth.random_fock_problem(rng, 12, [1] * 12, 3, 12)
    fp.T = 1e-3 * fp.T
    c["opaque"] = (fp, 1)
    fp = synth.random_fock_problem(rng, 12, [1] * 12, 3, 12)
    fp.T = np.eye(12, dtype=complex)[rng.permutation(12)]
    c["permutation"] = (fp, 1)
    return c


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("name", list(_cases()))
def test_convolution_against_node_walk(cuda_lib, name, precision):
    # both sides carry ~2^-50 of values below 1 summed over at most ~1e4 entries: 1e-13 absolute
    fp, over = _cases()[name]
    with cuda_lib.FockPlan(fp, precision=0, oversample=over, tile_override=9) as p:
        ref = p.table().cpu().numpy()
    with cuda_lib.FockPlan(fp, precision=precision, oversample=over) as p:
        P = p.table().cpu().numpy()
        again = p.table().cpu().numpy()
        d = p.diagnostics()
    # (ten grid points for one group leave the walk in pairs of FP32 cheaper)
    assert d["launches"] > 2 or name == "l1", "the rule did not take the convolution"
    assert np.abs(P - ref).max() < 1e-13
    assert np.array_equal(P, again)
    assert d["status"] == 0 and abs(d["sum_P"] - P.sum()) < 1e-13 and d["max_imag"] < 1e-13
    if name == "permutation":
        b = np.zeros(3, int)
        for i, l in enumerate(fp.bin_of_mode):
            b[l] += 1
        assert abs(P[tuple(b)] - 1.0) < 1e-13


def test_convolution_set_transfer(cuda_lib):
    rng = np.random.default_rng(77)
    a = synth.random_fock_problem(rng, 12, [1] * 12, 2, 12)
    b = synth.random_fock_problem(rng, 12, [1] * 12, 2, 12, eta_range=(0.01, 0.02))
    with cuda_lib.FockPlan(a) as p:
        p.set_transfer(b.T)
        P = p.table().cpu().numpy()
        assert p.diagnostics()["launches"] > 2
    assert np.abs(P - fock.table(b)["P"]).max() < 1e-13
