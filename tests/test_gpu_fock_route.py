"""Which Fock plans take the convolution: few-node walks stay, against the oracle on both sides of the line."""
import numpy as np
import pytest

import synth
from oracle import fock

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("photons,L,conv", [
    ([4], 1, False), ([5], 2, False), ([2, 2], 1, False), ([2, 2], 4, False), ([3, 1], 3, False), ([5, 5], 2, False),
    ([2, 1, 1], 1, False), ([2, 2, 1], 1, False), ([2, 1, 1], 2, True), ([3, 2, 1], 1, True), ([1, 1, 1, 1], 1, True),
])
def test_route(cuda_lib, photons, L, conv, precision):
    M = max(len(photons), L) + 2
    fp = synth.random_fock_problem(np.random.default_rng(11), M, photons + [0] * (M - len(photons)), L, sum(photons))
    with cuda_lib.FockPlan(fp, precision=precision) as p:
        P = p.table().cpu().numpy()
        d = p.diagnostics()
    assert (d["launches"] > 2) == conv
    # as the other Fock tests: ~2^-46 of values below 1 over at most a hundred nodes
    assert np.abs(P - fock.table(fp)["P"]).max() < (1e-13 if precision == 0 else 1e-11)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("N,L", [(13, 1), (14, 1), (16, 1), (12, 2)])
def test_walk_of_many_parts(cuda_lib, N, L, precision):
    # a short output axis after up to 1024 partial sums, against the convolution's table
    fp = synth.random_fock_problem(np.random.default_rng(N), N + 1, [1] * N + [0], L, N)
    with cuda_lib.FockPlan(fp, precision=0) as p:
        ref = p.table().cpu().numpy()
    with cuda_lib.FockPlan(fp, precision=precision, tile_override=9 + precision) as p:
        P = p.table().cpu().numpy()
        assert p.diagnostics()["launches"] == 2
    assert abs(P.sum() - 1.0) < 1e-11
    assert np.abs(P - ref).max() < (1e-13 if precision == 0 else 1e-11)
