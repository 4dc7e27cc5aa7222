"""A caller's own CUDA graph of an execute, replayed after the plan took another state or circuit: what belongs to the state
is read from device memory, so the replay gives the new state's table."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _captured(gb, execute, handle, P):
    import torch
    execute(handle, P)                                       # (first use outside the capture)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        execute(handle, P, torch.cuda.current_stream().cuda_stream)
    return g


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("M,cut,disp", [(20, 12, False), (5, 6, True), (80, 30, True)])
def test_one_group_table_of_a_later_state(cuda_lib, M, cut, disp, precision):
    import torch
    gb = cuda_lib
    # squeezing apart by a factor, so that q(1) of one state is far from the other's
    a = synth.random_problem(np.random.default_rng(1), M, 1, 1, [cut], displaced=disp, r_range=(0.1, 0.3))
    b = synth.random_problem(np.random.default_rng(2), M, 1, 1, [cut], displaced=disp, r_range=(0.9, 1.2))
    with gb.Plan(b, precision=precision) as q:
        ref = q.table().cpu().numpy()
        ref_piv = q.diagnostics()[1]["min_pivot_re"]
    with gb.Plan(a, precision=precision) as p:
        P = p.table()
        g = _captured(gb, gb.gbsbin_execute, p.handle, P)
        gb.gbsbin_plan_set_state(p.handle, b)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(P.cpu().numpy(), ref)          # the same launches on the same state
        assert p.diagnostics()[1]["min_pivot_re"] == ref_piv


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
def test_fock_table_of_a_later_circuit(cuda_lib, precision):
    import torch
    gb = cuda_lib
    rng = np.random.default_rng(3)
    a = synth.random_fock_problem(rng, 14, [1] * 12 + [0] * 2, 2, 12)
    b = synth.random_fock_problem(rng, 14, [1] * 12 + [0] * 2, 2, 12, eta_range=(0.01, 0.02))
    b.T = b.T * np.linspace(0.02, 1.0, 14)[:, None]          # rows of other magnitudes: other powers of two
    with gb.FockPlan(b, precision=precision) as q:
        ref = q.table().cpu().numpy()
    with gb.FockPlan(a, precision=precision) as p:
        P = p.table()
        assert p.diagnostics()["launches"] > 2, "the rule did not take the convolution"
        g = _captured(gb, gb.gbsbin_fock_execute, p.handle, P)
        p.set_transfer(b.T)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(P.cpu().numpy(), ref)
