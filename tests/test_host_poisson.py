"""Host-callable parts of the direct Poisson solve (csrc/poisson_direct.h; no GPU)."""
import ctypes
import os
import subprocess
from decimal import Decimal, getcontext

import pytest

from paper_1003_4570_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_4570_gb300", "csrc")


def test_pivots_are_exact_to_rounding(tmp_path):
    """The closed form against the recurrence in 60 digits, from eigenvalues far below the z spacing's
    to far above: about 16 roundings, 32 allowed."""
    (tmp_path / "w.cu").write_text('#include "%s/poisson_direct.h"\nextern "C" double pivot(double s, int j) { return pivot_at(s, j); }\n' % CSRC)
    subprocess.run([build._nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", str(tmp_path / "w.so"), str(tmp_path / "w.cu")],
                   check=True, capture_output=True)
    f = ctypes.CDLL(str(tmp_path / "w.so")).pivot
    f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double, ctypes.c_int]
    getcontext().prec = 60
    for e in range(-14, 13):
        for m in (1.0, 3.7):
            s = m * 10.0 ** e
            c = Decimal(0)
            for j in range(1, 300):
                c = 1 / (2 + 4 * Decimal(s) - c)
                if j < 5 or j % 37 == 0:
                    assert abs(Decimal(f(s, j)) / c - 1) <= 32 * Decimal(2) ** -53, (s, j)
    assert f(0.0, 7) == 7 / 8
