"""The FP32 pair an FP64 number is split into by integer operations (csrc/df.cuh; host code, no GPU).

hi is the number rounded to 24 bits, lo the rest rounded to 24: |v - hi - lo| <= 2^-49 |v|, the bound
of rounding twice.  Numbers whose leading bits carry into the exponent, ties, both signs and ranges.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1003_4570_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_4570_gb300", "csrc")
WRAP = """
#include "%s/df.cuh"
extern "C" void split(const unsigned long long* v, long n, int shift, unsigned* hi, unsigned* scale, int* rest) {
  for (long i = 0; i < n; ++i) {
    const SplitBits s = shift ? split_rounded_bits<32>(v[i]) : split_rounded_bits<0>(v[i]);
    hi[i] = s.hi, scale[i] = s.scale, rest[i] = s.rest;
  }
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "w.cu").write_text(WRAP % CSRC)
    subprocess.run([build._nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", str(d / "w.so"), str(d / "w.cu")], check=True,
                   capture_output=True)
    f = ctypes.CDLL(str(d / "w.so")).split

    def call(v, shift):
        v = np.ascontiguousarray(v, dtype=np.float64)
        hi, scale, rest = np.zeros(v.size, np.uint32), np.zeros(v.size, np.uint32), np.zeros(v.size, np.int32)
        f(*(ctypes.c_void_p(v.ctypes.data), ctypes.c_long(v.size), ctypes.c_int(shift)),
          *(ctypes.c_void_p(a.ctypes.data) for a in (hi, scale, rest)))
        return hi.view(np.float32), rest.astype(np.float32) * scale.view(np.float32)
    return call


@pytest.mark.parametrize("shift", [0, 32])
def test_pair_is_within_two_roundings(split, shift):
    rng = np.random.default_rng(3)
    m = np.concatenate([rng.uniform(1, 2, 200000), 2 - 2.0 ** -52 * np.arange(1, 200), 1 + 2.0 ** -24 * (1 + 2 * np.arange(200)),
                        1 + 2.0 ** -24 + 2.0 ** -52 * np.arange(-100, 100)])
    v = m * rng.choice([-1.0, 1.0], m.size) * 2.0 ** (rng.integers(-70, 120, m.size) - shift)
    hi, lo = split(v, shift)
    back = (hi.astype(np.float64) + lo.astype(np.float64)) * 2.0 ** -shift
    assert np.abs((hi.astype(np.float64) * 2.0 ** -shift - v) / v).max() <= 2.0 ** -24
    assert np.abs((back - v) / v).max() <= 2.0 ** -49


@pytest.mark.parametrize("shift", [0, 32])
def test_out_of_range(split, shift):
    hi, lo = split(np.array([0.0, -0.0, 1e-300, -1e-60, 2.0 ** -159]) * 2.0 ** (32 - shift), shift)
    assert (hi == 0).all() and (lo == 0).all()
    hi, _ = split([np.inf, -np.inf, np.nan, 1e300, -2.0 ** (128 - shift)], shift)
    assert np.isnan(hi).all()
