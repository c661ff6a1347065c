"""The reduced Slater–Koster blocks the product applies, against the oracle's rotated blocks.

csrc/sk_device.cuh writes the block of a bond along (1,1,1) as 25 numbers (10 for sp3s*); expanded
here by their definition (sums, multiples of the identity, the e pair's zero-sum triple) and
signed for each direction, they must give the oracle's block of every direction, for both ends of
the bond (host code of the library, no GPU).  Tolerance: a few roundings of numbers of size 3 eV.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth
from oracle import lattice, sk
from paper_1003_4570_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_4570_gb300", "csrc")
WRAP = """
#include "%s/sk_device.cuh"
extern "C" void block(const double* v12, const double* v21, int norb, int transposed, double* c) {
  reduced_block(v12, v21, norb, transposed != 0, c);
}
"""


@pytest.fixture(scope="module")
def block(tmp_path_factory):
    d = tmp_path_factory.mktemp("reduced")
    (d / "w.cu").write_text(WRAP % CSRC)
    subprocess.run([build._nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", str(d / "w.so"), str(d / "w.cu")], check=True,
                   capture_output=True)
    f = ctypes.CDLL(str(d / "w.so")).block

    def call(v12, v21, norb, transposed):
        c = np.zeros(28)
        a, b = (np.ascontiguousarray(v, dtype=np.float64) for v in (v12, v21))
        f(a.ctypes.data_as(ctypes.c_void_p), b.ctypes.data_as(ctypes.c_void_p), norb, int(transposed), c.ctypes.data_as(ctypes.c_void_p))
        return c
    return call


def expand(c, norb):
    """The full block along (1,1,1) from its reduced numbers."""
    one, eye = np.ones((3, 3)), np.eye(3)
    B = np.zeros((norb, norb))
    if norb == 5:
        B[0, [0, 1, 2, 3, 4]] = [c[0], c[1], c[1], c[1], c[2]]
        B[4, [0, 1, 2, 3, 4]] = [c[3], c[4], c[4], c[4], c[5]]
        B[1:4, 0], B[1:4, 4], B[1:4, 1:4] = c[6], c[7], c[8] * one + c[9] * eye
        return B
    r = np.sqrt(3.0) / 2
    q = np.array([[r, -0.5], [-r, -0.5], [0.0, 1.0]])         # zero-sum triple of (x2-y2, 3z2-r2)
    for row, at in ((0, 0), (9, 4)):
        B[row, 0], B[row, 1:4], B[row, 4:7], B[row, 9] = c[at:at + 4]
    for rows, at in ((slice(1, 4), 8), (slice(4, 7), 15)):
        B[rows, 0], B[rows, 9] = c[at], c[at + 1]
        B[rows, 1:4], B[rows, 4:7] = c[at + 2] * one + c[at + 4] * eye, c[at + 3] * one + c[at + 5] * eye
        B[rows, 7:9] = c[at + 6] * q
    B[8, 1:4], B[8, 4:7] = c[22] * q[:, 1], c[23] * q[:, 1]
    B[7, 1:4], B[7, 4:7] = c[25] * np.array([1, -1, 0]), c[26] * np.array([1, -1, 0])
    B[7:9, 7:9] = c[24] * np.eye(2)
    return B


@pytest.mark.parametrize("norb", [5, 10])
def test_reduced_blocks_give_the_rotated_blocks(block, norb):
    p = synth.draw_tb_params(17, norb, 3)
    g = np.random.default_rng(1)
    V = p.V + (p.V != 0) * g.uniform(-1, 1, p.V.shape)        # every ordered pair its own integrals
    for i in range(3):
        for j in range(3):
            for k, u in enumerate(lattice.BOND_DIRS):
                want = sk.sk_block(u / np.sqrt(3.0), V[i, j], V[j, i], norb)
                s = np.ones(norb)
                s[1:4] = u
                if norb == 10:
                    s[4:7] = u
                for transposed in (False, True):
                    got = s[:, None] * expand(block(V[i, j], V[j, i], norb, transposed), norb) * s[None, :]
                    np.testing.assert_allclose(got, want.T if transposed else want, atol=2e-14, rtol=0)
