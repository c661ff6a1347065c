"""Single-vector Lanczos on enough rows for the wide form of its step kernels.

Below 152 x 256 rows the step kernels share a row among several threads and take narrow CTAs; the
other eigenvalue tests stay there (or run real FP64 at full size).  39,200 rows, real and complex,
FP64 and FP32 refined in FP64, against scipy's ARPACK on the oracle's matrix: 1e-9 eV (FP64) and 1e-8
eV (refined), as for the smaller problems.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import hamiltonian  # noqa: E402


@pytest.mark.parametrize("bloch", [False, True])
@pytest.mark.parametrize("refined", [False, True])
def test_lowest_levels_of_a_wide_problem(bloch, refined):
    from paper_1003_4570_gb300 import omen
    ctx = omen.omen_create(0, torch.cuda.current_stream().cuda_stream)
    spec = synth.lattice_spec(7, 7, 20, (2, 2, 0) if bloch else (0, 0, 0), seed=91, alloy_fraction=0.3, strain_amp=0.02)
    p = synth.draw_tb_params(91, 5, 2)
    k = (0.3, 0.2, 0.0) if bloch else None
    prec = omen.OMEN_F32_REFINE64 if refined else omen.OMEN_F64
    ham = omen.omen_assemble_H(ctx, omen.omen_build_lattice(ctx, spec), p, precision=prec, k=k)
    tol = 1e-8 if refined else 1e-9
    ev, info, _ = omen.omen_eigs(ctx, ham, 3, tol=tol, block=1, basis=48, max_iter=20000)
    assert info["converged"] == 1, info
    ref = np.sort(spla.eigsh(hamiltonian.assemble(spec, p, kvec=k), k=5, which="SA", tol=1e-12, ncv=60)[0])[:3]
    np.testing.assert_allclose(ev, ref, atol=tol, rtol=0)
