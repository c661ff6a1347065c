"""Deposit and gather over grids of every relation to the structure, and the forms of calls whose
small inputs travel with the launch.

Deposit and gather look the atoms' cloud-in-cell positions up per axis: grids finer and coarser
than the atomic planes, a box shorter than the structure (its atoms wrap in x and y and are
grounded in z) or longer, one- and two-point axes; 1e-12 of the largest value against the oracle.
Electrons per atom from more than 64 states against 64 of them, and k batches of more than 128 wave
vectors against the same call in parts (bit for bit) and against the oracle (1e-12).
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import charge, hamiltonian, lattice, poisson  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    from paper_1003_4570_gb300 import omen
    return omen.omen_create(0, torch.cuda.current_stream().cuda_stream)


GRIDS = [
    # (cells, grid points, box relative to the structure)
    ((2, 3, 4), (5, 7, 21), (1.0, 1.0, 1.0)), ((3, 2, 2), (40, 3, 33), (1.0, 1.0, 1.0)),
    ((1, 1, 3), (1, 2, 9), (1.0, 1.0, 1.0)), ((4, 3, 2), (6, 9, 5), (0.4, 0.3, 1.0)),
    ((2, 2, 5), (8, 8, 6), (1.0, 1.0, 0.6)), ((2, 1, 2), (37, 33, 12), (1.9, 1.0, 1.5)),
]


@pytest.mark.parametrize("case", GRIDS, ids=[f"g{i}" for i in range(len(GRIDS))])
def test_deposit_and_gather_match_oracle(ctx, case):
    from paper_1003_4570_gb300 import omen
    cells, n, rel = case
    spec = synth.lattice_spec(*cells, (1, 1, 0), seed=4)
    g = poisson.Grid(*n, *[c * spec.a_nm * r for c, r in zip(cells, rel)])
    pos = lattice.positions(*cells) * (spec.a_nm / 4)
    lat = omen.omen_build_lattice(ctx, spec)
    rng = np.random.default_rng(7)
    q, phi = rng.normal(size=spec.natoms) * 1e-19, rng.normal(size=g.shape)
    rho = torch.full(g.shape, 7.0, dtype=torch.float64, device="cuda")
    omen.omen_deposit(ctx, lat, g, torch.from_numpy(q).cuda(), rho)
    at = torch.empty(spec.natoms, dtype=torch.float64, device="cuda")
    omen.omen_gather(ctx, lat, g, torch.from_numpy(phi).cuda(), at)
    want = charge.deposit(g, pos, q)
    np.testing.assert_allclose(rho.cpu().numpy(), want, atol=1e-12 * max(np.abs(want).max(), 1e-30), rtol=0)
    want = charge.gather(g, phi, pos)
    np.testing.assert_allclose(at.cpu().numpy(), want, atol=1e-12 * np.abs(phi).max(), rtol=0)


def test_density_of_more_states_than_a_launch_carries(ctx):
    """64 states travel with the launch; a 65th, empty one sends the same sum the other way."""
    from paper_1003_4570_gb300 import omen
    spec = synth.lattice_spec(3, 2, 2, (1, 1, 0), seed=5)
    ham = omen.omen_assemble_H(ctx, omen.omen_build_lattice(ctx, spec), synth.draw_tb_params(5, 10, 1))
    psi = torch.from_numpy(np.random.default_rng(2).normal(size=(65, ham.nrows))).cuda()
    occ = np.append(np.linspace(1.0, 0.1, 64), 0.0)
    n = torch.zeros((2, spec.natoms), dtype=torch.float64, device="cuda")
    omen.omen_density_accum(ctx, ham, psi, 64, occ[:64], 2.0, n[0])
    omen.omen_density_accum(ctx, ham, psi, 65, occ, 2.0, n[1])
    assert torch.equal(n[0], n[1]) and bool((n[0] > 0).all())


def test_kbatch_of_more_wave_vectors_than_a_launch_carries(ctx):
    from paper_1003_4570_gb300 import omen
    spec = synth.lattice_spec(2, 1, 3, (2, 2, 0), seed=9, alloy_fraction=0.3, strain_amp=0.02)
    p = synth.draw_tb_params(9, 10, 2)
    ham = omen.omen_assemble_H(ctx, omen.omen_build_lattice(ctx, spec), p, k=(0.0, 0.0, 0.0))
    nk = 131
    ks = np.random.default_rng(3).uniform(-2, 2, size=(nk, 3)) * [1, 1, 0]
    x = synth.random_vectors(3, ham.nrows, nk, dtype=complex)
    xd = torch.from_numpy(x).cuda()
    y = torch.empty_like(xd)
    omen.omen_hx_kbatch(ctx, ham, ks, xd, y, sigma=0.2)
    parts = torch.empty_like(xd)
    for a, b in ((0, 128), (128, nk)):
        omen.omen_hx_kbatch(ctx, ham, ks[a:b], xd[a:b], parts[a:b], sigma=0.2)
    assert torch.equal(y, parts)
    for q in (0, 127, 128, nk - 1):
        ref = hamiltonian.assemble(spec, p, kvec=ks[q]) @ x[q] - 0.2 * x[q]
        np.testing.assert_allclose(y[q].cpu().numpy(), ref, atol=1e-12 * np.abs(ref).max(), rtol=0)
