"""The host's spectral decomposition at entries far below 1, whose squares and reciprocals leave FP64's range, compiled
from the library's sources on the CPU, and tables of states that hold such entries (GPU)."""
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_17742_gb300", "csrc")

MAIN = '''
#include <cstdio>
#include "gbsbin_host_state.h"
int main() {                          // n m, A (n x n), X (n x m) -> 1, the eigenvalues, Q^H X
  int n, m;
  if (std::scanf("%d %d", &n, &m) != 2) return 1;
  auto num = [] { double v = 0; return std::scanf("%la", &v) == 1 ? v : 0.0; };
  std::vector<std::complex<double>> A((size_t)n * n);
  for (auto& a : A) { const double re = num(); a = {re, num()}; }
  std::vector<double> xr((size_t)n * m), xi((size_t)n * m), lam;
  for (size_t q = 0; q < xr.size(); ++q) { xr[q] = num(); xi[q] = num(); }
  std::printf("%d\\n", gbsbin::hermitian_spectrum(A, n, lam, xr.data(), xi.data(), m) ? 1 : 0);
  for (double v : lam) std::printf("%a ", v);
  for (size_t q = 0; q < xr.size(); ++q) std::printf("%a %a ", xr[q], xi[q]);
}
'''


@pytest.fixture(scope="module")
def spectrum(tmp_path_factory):
    d = tmp_path_factory.mktemp("spectrum")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "spectrum")
    subprocess.run(["g++", "-O2", "-std=c++17", str(d / "main.cpp"), os.path.join(CSRC, "gbsbin_host_eigen.cpp"),
                    os.path.join(CSRC, "gbsbin_host_pool.cpp"), "-I", CSRC, "-lpthread", "-o", exe], check=True)

    def run(A, X):
        n, m = X.shape
        vals = np.concatenate([np.asarray(A, complex).ravel(), np.asarray(X, complex).ravel()])
        text = f"{n} {m}\n" + "\n".join(f"{float(v.real).hex()} {float(v.imag).hex()}" for v in vals)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
        f = np.array([float.fromhex(v) if "nan" not in v and "inf" not in v else np.nan for v in out[1:]])
        return out[0] == "1", f[:n], (f[n::2] + 1j * f[n + 1::2]).reshape(n, m)

    return run


@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e-80, 1e-100, 1e-150, 1e-200, 1e-290])
@pytest.mark.parametrize("kind", ["all", "coupling", "last"])
@pytest.mark.parametrize("n", [2, 3, 8, 21])
def test_small_entries(spectrum, n, kind, scale):
    rng = np.random.default_rng(n)
    Z = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    H = 0.2 * (Z + Z.conj().T)
    if kind == "all":                                   # every entry scaled
        A, unit = H * scale, scale
    elif kind == "coupling":                            # the off-diagonal ones
        A, unit = np.diag(np.diag(H)) + (H - np.diag(np.diag(H))) * scale, 1.0
    else:                                               # the last row's and column's
        A, unit = H.copy(), 1.0
        A[-1, :-1] *= scale
        A[:-1, -1] *= scale
    X = rng.standard_normal((n, 3)) + 1j * rng.standard_normal((n, 3))
    ok, lam, Y = spectrum(A, X)
    assert ok and np.isfinite(lam).all() and np.isfinite(Y).all()
    # n steps of unitary transformations: some n eps of the matrix' size
    tol = 40 * n * 2.0 ** -53
    assert np.abs(np.sort(lam) - np.linalg.eigvalsh(A / unit) * unit).max() <= tol * unit * 2 * np.sqrt(n)
    assert np.abs(np.linalg.norm(Y, axis=0) - np.linalg.norm(X, axis=0)).max() <= tol * np.linalg.norm(X)
    quad = np.einsum("ij,ik,kj->j", X.conj(), A / unit, X).real
    assert np.abs((lam / unit) @ np.abs(Y) ** 2 - quad).max() <= tol * 2 * np.sqrt(n) * np.linalg.norm(X) ** 2


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("cut", [[5], [3, 4], [2, 2, 3]])
@pytest.mark.parametrize("kind", ["weak_squeezing", "weak_coupling"])
def test_tables_of_weak_states(cuda_lib, kind, cut, precision):
    gb = cuda_lib
    M, L = 9, len(cut)
    prob = synth.random_problem(np.random.default_rng(17), M, 1, L, cut, r_range=(0.3, 0.8))
    if kind == "weak_squeezing":
        prob.r = np.where(np.arange(M)[:, None] % 3 == 0, prob.r, 1e-100)
    else:                                               # coupling of neighbours exp(-200): overlaps of distant modes
        x = np.arange(M)
        prob.T = 0.9 * np.exp(-200.0 * np.minimum((x[:, None] - x[None, :]) ** 2, 3)).astype(complex)
    with gb.Plan(prob, precision=precision) as p:
        P = p.table().cpu().numpy()
        st, d = p.diagnostics()
    # the small tables' bounds: n eps of FP64, n 2^-46 of pairs, some tens over
    assert st == 0 and d["n_bad_points"] == 0
    assert np.abs(P - oracle.binned(prob)["P"]).max() < (1e-13 if precision == 0 else 1e-11)
