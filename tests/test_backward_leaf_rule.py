"""Which leaves the reverse pass along the large-matrix tree takes: Hessenberg leaves nowhere that Gauss-Jordan leaves were
measured faster, in either arithmetic, and still where they gain most."""
import ctypes
import re
import subprocess

import pytest

SMS = 152
# reverse-pass kernels, time with Hessenberg leaves over time with Gauss-Jordan leaves, by (pairs, rows of the last
# group, parents): leaves per SM -> ratio
MEASURED = {
    (False, 32, 30): {8: 1.51, 16: 1.28, 24: 1.10}, (False, 32, 61): {8: 1.48, 16: 1.22, 24: 1.10},
    (False, 32, 140): {8: 1.85, 16: 1.57, 24: 1.36}, (False, 40, 30): {8: 1.21, 11: 1.12, 24: 0.83},
    (False, 40, 61): {8: 1.20, 11: 1.11, 24: 0.83}, (False, 40, 140): {8: 1.52, 16: 1.23, 24: 1.04},
    (False, 48, 30): {8: 1.19, 11: 1.10, 24: 0.81}, (False, 48, 61): {8: 1.18, 11: 1.09, 24: 0.81},
    (False, 48, 140): {8: 1.48, 16: 1.20}, (False, 60, 30): {6: 1.23, 11: 0.86, 24: 0.63},
    (False, 60, 140): {8: 1.18, 11: 1.09, 24: 0.78}, (False, 80, 30): {4: 1.20, 8: 0.71, 16: 0.56},
    (False, 80, 61): {4: 1.23, 11: 0.81, 16: 0.65}, (False, 80, 140): {6: 1.21, 8: 1.06, 16: 0.81},
    (False, 100, 61): {4: 1.05, 8: 0.71, 16: 0.49}, (False, 100, 140): {6: 1.11, 11: 0.76, 16: 0.64},
    (True, 32, 30): {8: 1.17, 11: 1.10, 24: 0.89}, (True, 32, 61): {8: 1.14, 11: 1.09, 24: 0.88},
    (True, 32, 140): {8: 1.15, 11: 1.11}, (True, 40, 30): {6: 1.27, 8: 1.06, 16: 0.91},
    (True, 40, 61): {6: 1.12, 8: 1.04, 16: 0.87}, (True, 40, 140): {6: 1.14, 8: 1.08, 24: 0.82},
    (True, 48, 61): {4: 1.10, 8: 0.91, 16: 0.74}, (True, 60, 30): {4: 1.31, 8: 0.89, 16: 0.75},
    (True, 60, 140): {4: 1.30, 11: 0.89, 24: 0.71}, (True, 100, 61): {8: 0.55, 24: 0.34},
    (True, 116, 140): {8: 0.63, 24: 0.39},
}


@pytest.fixture(scope="module")
def suits():
    from paper_2412_17742_gb300 import build
    path = build.build()
    names = subprocess.run(["nm", "-D", path], capture_output=True, text=True, check=True).stdout
    f = getattr(ctypes.CDLL(path), re.search(r"\S*backward_hess_suits\S*", names).group(0))
    f.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_bool]
    f.restype = ctypes.c_bool
    return f


@pytest.mark.parametrize("df,rows,parents", list(MEASURED))
def test_rule_follows_the_measured_crossing(suits, df, rows, parents):
    for leaves, ratio in MEASURED[df, rows, parents].items():
        taken = suits(rows, parents, max(2, round(leaves * SMS / parents)), SMS, df)
        if ratio > 1.02:
            assert not taken, (leaves, ratio)
        if ratio < 0.92:
            assert taken, (leaves, ratio)


def test_limits(suits):
    assert not suits(30, 61, 4000, SMS, True) and not suits(38, 61, 4000, SMS, False)
    assert not suits(118, 61, 4000, SMS, True) and suits(116, 61, 4000, SMS, False)
