"""Both thread layouts of the H·X product against the oracle.

Small products take one lane per bond, larger ones (more cells, or more vectors at once) one lane
per row.  The same vectors go through both: alone, and as part of a block large enough for the
other layout.  Extents around the warp's 32 cells and the 8 (complex: 4) cells of the lane-per-bond
form; every boundary kind, both bases, spin-orbit.  Tolerances as for the product everywhere else:
FP64 1e-12, FP32 2e-6 of max |y|.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import hamiltonian  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    from paper_1003_4570_gb300 import omen
    return omen.omen_create(0, torch.cuda.current_stream().cuda_stream)


CASES = [
    # (cells, boundaries, basis, spin-orbit, k, precision)
    ((1, 1, 1), (1, 1, 1), 10, False, None, 0),
    ((3, 1, 3), (0, 1, 0), 10, False, None, 0),
    ((11, 3, 1), (1, 0, 1), 5, False, None, 0),
    ((31, 1, 1), (0, 0, 0), 10, False, None, 1),
    ((1, 1, 5), (2, 2, 0), 10, False, (0.9, -0.4, 0.0), 0),
    ((2, 3, 11), (2, 1, 2), 10, False, (0.5, 0.0, -0.3), 1),
    ((5, 1, 7), (2, 2, 0), 5, False, (0.2, 1.3, 0.0), 0),
    ((4, 3, 3), (0, 1, 0), 10, True, None, 0),
    ((1, 2, 17), (2, 2, 0), 10, True, (0.7, -0.2, 0.0), 1),
    ((3, 2, 2), (1, 1, 2), 5, True, (0.0, 0.0, 0.6), 0),
]


@pytest.mark.parametrize("case", CASES, ids=[f"p{i}" for i in range(len(CASES))])
def test_both_layouts_match_oracle(ctx, case):
    from paper_1003_4570_gb300 import omen
    cells, per, basis, so, k, prec = case
    spec = synth.lattice_spec(*cells, per, seed=81, alloy_fraction=0.4, strain_amp=0.02)
    p = synth.draw_tb_params(81, basis, 3)
    spec.species[::5] = 2
    U = np.random.default_rng(8).uniform(-0.2, 0.2, spec.natoms)
    H = hamiltonian.assemble(spec, p, U_atom=U, kvec=k, spin_orbit=so)
    lat = omen.omen_build_lattice(ctx, spec)
    ham = omen.omen_assemble_H(ctx, lat, p, spin_orbit=so, precision=prec, k=k, U_atom_dev=torch.from_numpy(U).cuda())
    tiles = (spec.ncells + 31) // 32 * 8
    nvec = 900 // tiles + 1                        # past every line between the layouts
    x = synth.random_vectors(6, H.shape[0], nvec, dtype=complex if ham.is_complex else float)
    xd = torch.from_numpy(x.astype(ham.numpy_dtype)).cuda()
    tol = 1e-12 if prec == 0 else 2e-6
    y = torch.empty_like(xd)
    omen.omen_hx(ctx, ham, xd, y, nvec=nvec, sigma=0.3)
    y1 = torch.empty_like(xd[:1])
    for v in (0, nvec - 1):
        omen.omen_hx(ctx, ham, xd[v:v + 1].contiguous(), y1, nvec=1, sigma=0.3)
        torch.cuda.synchronize()
        xv = x[v].astype(ham.numpy_dtype).astype(complex if ham.is_complex else float)
        ref = H @ xv - 0.3 * xv
        for got in (y[v], y1[0]):
            np.testing.assert_allclose(got.cpu().numpy(), ref, atol=tol * np.abs(ref).max(), rtol=0)


LAYOUTS = [
    # (cells, boundaries, basis, spin-orbit, k, precision, vectors that take the middle layout)
    ((4, 4, 9), (0, 1, 0), 10, False, None, 0, 4),
    ((5, 4, 9), (0, 0, 1), 10, False, None, 1, 8),
    ((3, 3, 7), (2, 2, 0), 10, False, (0.5, -0.3, 0.0), 0, 5),
    ((2, 3, 11), (2, 1, 2), 10, False, (0.5, 0.0, -0.3), 1, 4),
    ((3, 3, 5), (0, 1, 0), 10, True, None, 0, 3),
    ((4, 4, 9), (1, 0, 0), 5, False, None, 0, 4),
    ((3, 3, 7), (2, 2, 0), 5, False, (0.2, 1.3, 0.0), 0, 5),
]


@pytest.mark.parametrize("case", LAYOUTS, ids=[f"p{i}" for i in range(len(LAYOUTS))])
def test_three_layouts_match_oracle(ctx, case):
    """A warp per kind of row (few vectors), a lane per bond (some) and a lane per row (many)."""
    from paper_1003_4570_gb300 import omen
    cells, per, basis, so, k, prec, mid = case
    spec = synth.lattice_spec(*cells, per, seed=83, alloy_fraction=0.4, strain_amp=0.02)
    p = synth.draw_tb_params(83, basis, 3)
    spec.species[::5] = 2
    U = np.random.default_rng(9).uniform(-0.2, 0.2, spec.natoms)
    H = hamiltonian.assemble(spec, p, U_atom=U, kvec=k, spin_orbit=so)
    lat = omen.omen_build_lattice(ctx, spec)
    ham = omen.omen_assemble_H(ctx, lat, p, spin_orbit=so, precision=prec, k=k, U_atom_dev=torch.from_numpy(U).cuda())
    many = 900 // ((spec.ncells + 31) // 32 * 8) + 1
    x = synth.random_vectors(6, H.shape[0], many, dtype=complex if ham.is_complex else float)
    xd = torch.from_numpy(x.astype(ham.numpy_dtype)).cuda()
    tol = 1e-12 if prec == 0 else 2e-6
    for nvec in (1, mid, many):
        y = torch.empty_like(xd[:nvec])
        omen.omen_hx(ctx, ham, xd[:nvec].contiguous(), y, nvec=nvec, sigma=0.3)
        torch.cuda.synchronize()
        for v in (0, nvec - 1):
            xv = x[v].astype(ham.numpy_dtype).astype(complex if ham.is_complex else float)
            ref = H @ xv - 0.3 * xv
            np.testing.assert_allclose(y[v].cpu().numpy(), ref, atol=tol * np.abs(ref).max(), rtol=0)
