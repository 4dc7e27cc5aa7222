"""min_pivot_re of heralded states in FP64: the smallest real part over the points of the traced rows' pivots, the first
group's factors 1 - w lambda, the other groups' and the kept rows' pivots."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _pivots(B):
    """Pivots of the unpivoted elimination of B's leading block, and what it leaves of the rest."""
    B = B.copy()
    out = []
    for k in range(len(B)):
        out.append(B[k, k])
        B[k + 1:, k + 1:] -= np.outer(B[k + 1:, k] / B[k, k], B[k, k + 1:])
    return np.array(out)


def _expected(prob, roles, radix):
    A = oracle.state.adjacency(*oracle.state.sigma1_zbar(prob))[0]   # XA
    nm = len(roles)
    rows = {r: [m + h * nm for h in (0, 1) for m in range(nm) if roles[m] == r] for r in set(roles)}
    order = rows.get(-1, []) + sum((rows[l] for l in range(len(radix))), []) + rows[-2]
    A = A[np.ix_(order, order)]
    nt, n0 = len(rows.get(-1, [])), len(rows[0])
    least = np.inf
    if nt:                                               # traced rows at w = 1
        T = np.eye(nt) - A[:nt, :nt]
        least = _pivots(T).real.min()
        A = A[nt:, nt:] + A[nt:, :nt] @ np.linalg.solve(T, A[:nt, nt:])
    lam, Q = np.linalg.eigh(A[:n0, :n0])
    for k in np.ndindex(*radix):
        w = np.exp(2j * np.pi * np.array(k) / radix)
        least = min(least, (1 - w[0].real * lam).min())
        B = A[n0:, n0:] + A[n0:, :n0] @ (Q * (w[0] / (1 - w[0] * lam))) @ (Q.conj().T @ A[:n0, n0:])
        D = np.concatenate([np.full(len(rows[l]), w[l]) for l in range(1, len(radix))] + [np.ones(len(rows[-2]))])
        least = min(least, _pivots(np.eye(len(B)) - D[:, None] * B).real.min())
    return least


@pytest.mark.parametrize("roles,cutoff,r", [
    ([0, 0, -2], [3], (0.8, 1.2)), ([0, -1, 0, -2, -1], [2], (0.2, 0.8)), ([0, 1, 0, 1, -2, -1], [2, 3], (0.3, 1.0)),
    ([0] * 17 + [1] * 3 + [2] * 2 + [-2, -2], [1, 2, 1], (0.2, 1.4)),
])
def test_min_pivot_is_fp64(cuda_lib, roles, cutoff, r):
    prob = synth.random_problem(np.random.default_rng(len(roles)), len(roles), 1, 1, [1], displaced=True, r_range=r)
    with cuda_lib.HeraldPlan(prob, roles, cutoff, 1) as h:
        h.states()
        got = h.diagnostics()["min_pivot_re"]
    want = _expected(prob, roles, np.array(cutoff) + 1)
    assert abs(got - want) < 1e-12 * abs(want)           # FP32 keeps 6e-8
