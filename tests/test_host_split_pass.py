"""The passes of a restart's combination (csrc/split_pass.h; host code, no GPU)."""
import ctypes
import os
import subprocess

from paper_1003_4570_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_4570_gb300", "csrc")
WRAP = """
#include "%s/split_pass.h"
extern "C" int passes(int na, int total, long* work) {
  int n = 0;
  for (int c0 = 0; c0 < total; ++n) {
    const SplitPass p = split_pass(na, total, total - c0);
    if (p.cols < 1 || p.cols > p.kernel || p.cols > total - c0) return -1;
    if (p.kernel != 8 && p.kernel != 16 && p.kernel != 25) return -2;
    if ((size_t)na * p.kernel * 8 > 227 * 1024) return -3;   // FP32 pairs in shared memory
    c0 += p.cols;
    *work += p.kernel;
  }
  return n;
}
"""


def test_every_basis_has_its_passes(tmp_path):
    """Every number of columns from every basis that a solve accepts is covered by passes whose
    coefficients fit shared memory, with no more passes than 16 columns each take where those fit,
    and fewer idle columns than a pass of 8 holds beyond that."""
    (tmp_path / "w.cu").write_text(WRAP % CSRC)
    subprocess.run([build._nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", str(tmp_path / "w.so"), str(tmp_path / "w.cu")],
                   check=True, capture_output=True)
    f = ctypes.CDLL(str(tmp_path / "w.so")).passes
    for na in [2, 48, 64, 97, 655, 1162, 1163, 1816, 1817, 2047, 2048]:
        for total in list(range(1, 130)) + [400, 1024, 2048]:
            if total > na:
                break
            work = ctypes.c_long(0)
            n = f(na, total, ctypes.byref(work))
            assert n > 0, (na, total, n)
            if na <= 1816:
                assert n <= -(-total // 16) and work.value - total < 9, (na, total, n, work.value)
