"""Coefficients of the Fock convolution whose real and imaginary parts both lie just below their row's power of two:
the sum of their high digits has to fit an int (compiled from the library's header on the CPU), and the tables of
circuits made of them have to agree with the node walk (GPU)."""
import os
import subprocess
from types import SimpleNamespace

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _by_groups(M, T, photons, L):
    p = np.zeros(M, dtype=np.int32)
    p[list(photons)] = 1
    return SimpleNamespace(M=M, T=T, photons=p, bin_of_mode=np.arange(M, dtype=np.int32) % L,
                           cutoff=np.full(L, len(photons), dtype=np.int32))


def _blocks(loss=0.0):
    """Four lossless 4 x 4 blocks: a column of equal amplitudes, then two of a phase e^{i pi/4}."""
    c, f = (1 / np.sqrt(2)) ** 2, np.exp(0.25j * np.pi) / np.sqrt(2)
    B = np.zeros((4, 4), dtype=complex)
    B[:, 0] = c
    B[:2, 1] = f * np.array([1, -1])
    B[2:, 2] = f * np.array([1, -1])
    B[:, 3] = c * np.array([1, 1, -1, -1])
    T = np.kron(np.eye(4), B) * np.sqrt(1.0 - loss)
    return _by_groups(16, T, [4 * b + i for b in range(4) for i in range(3)], 4)


def _pair():
    """An entry 0.25 (1 - 2^-40) (1 + i) beside a diagonal of 0.2 in every group."""
    a, x = np.sqrt(0.2), 0.25 * (1 - 2.0 ** -40)
    B = np.zeros((4, 2), dtype=complex)
    B[:, 0] = a
    B[0, 1] = x * (1 + 1j) / a
    B[1, 1] = -0.1 * (1 + 1j) / a
    T = np.zeros((16, 16), dtype=complex)
    for b in range(4):
        T[4 * b:4 * b + 4, 4 * b:4 * b + 2] = B
    for j in range(16):
        if j % 4 >= 2:
            T[j, j] = 0.1
    return _by_groups(16, T, [j for j in range(16) if j % 4 < 3], 4)


CASES = {"blocks": lambda: _blocks(), "blocks_lossy": lambda: _blocks(1e-11), "pair": _pair}


def _coefficients(fp):
    """The matrices I - T^dag T and T_l^dag T_l over the occupied inputs, [m][j][k]."""
    T = fp.T[:, fp.photons > 0]
    rows = [np.eye(T.shape[1]) - T.conj().T @ T]
    return np.array(rows + [T[fp.bin_of_mode == l].conj().T @ T[fp.bin_of_mode == l] for l in range(len(fp.cutoff))])


def test_digit_sums_fit(tmp_path):
    src = tmp_path / "digits.cpp"
    src.write_text('''
#include <cstdio>
#include "gbsbin_fock_conv.h"
using namespace gbsbin;
int main() {                       // rows "n big all", then n pairs (re, im): the largest |hi re + hi im| of all
  int n;
  double big, all;
  long long worst = 0;
  while (std::scanf("%d %la %la", &n, &big, &all) == 3) {
    const int e = conv_row_exponent(big, all);
    for (int i = 0; i < n; ++i) {
      double re, im;
      if (std::scanf("%la %la", &re, &im) != 2) return 1;
      int h[2], l[2];
      digits<kConvDigit>(conv_fixed(re, e), h[0], l[0]);
      digits<kConvDigit>(conv_fixed(im, e), h[1], l[1]);
      worst = std::max(worst, std::llabs((long long)h[0] + h[1]));
    }
  }
  std::printf("%lld\\n", worst);
}
''')
    exe = str(tmp_path / "digits")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", str(src), "-o", exe, "-I", os.path.join(cuda, "include"),
                    "-I", os.path.join(ROOT, "paper_2412_17742_gb300", "csrc")], check=True)
    rows = [np.array([complex(1 - 2.0 ** -53, 1 - 2.0 ** -53)])]       # the largest that a row's power of two allows
    for make in CASES.values():
        B = _coefficients(make())
        rows += [B[:, j, :].ravel() for j in range(B.shape[1])]
    text = ""
    for r in rows:
        parts = np.concatenate([np.abs(r.real), np.abs(r.imag)])
        text += f"{len(r)} {float(parts.max()).hex()} {float(parts.sum()).hex()}\n"
        text += "\n".join(f"{float(v.real).hex()} {float(v.imag).hex()}" for v in r) + "\n"
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    assert 0 < int(out) < 2 ** 31


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "df32"])
@pytest.mark.parametrize("name", list(CASES))
def test_tables_at_the_digit_bound(cuda_lib, name, precision):
    # both sides carry ~2^-50 of values below 1 summed over at most ~1e4 entries: 1e-13 absolute
    fp = CASES[name]()
    with cuda_lib.FockPlan(fp, precision=0, tile_override=9) as p:
        ref = p.table().cpu().numpy()
    with cuda_lib.FockPlan(fp, precision=precision) as p:
        P = p.table().cpu().numpy()
        assert p.diagnostics()["launches"] > 2, "the rule did not take the convolution"
    assert abs(ref.sum() - 1.0) < 1e-12
    assert np.abs(P - ref).max() < 1e-13
