"""The direct corrections of omen_poisson against the oracle's sparse direct solve.

Grids through every part of it: line lengths with factors 4, 2, 3, 5 and larger primes, one- and
two-point axes, planes transformed at once and line by line (more than 3,072 points a plane), one
plane, an odd last plane, tridiagonal systems in segments of 8, 16 and 32 and longer than 256
unknowns; unequal spacings and a start other than zero.  Tolerance: 1e-10 of max |phi|, as for the
iterations.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import poisson  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    from paper_1003_4570_gb300 import omen
    return omen.omen_create(0, torch.cuda.current_stream().cuda_stream)


GRIDS = [
    (1, 1, 2), (2, 1, 3), (1, 2, 9), (2, 2, 300), (3, 5, 8), (11, 11, 40), (13, 34, 7), (16, 15, 33), (9, 64, 6),
    (1, 97, 12), (48, 64, 4),                        # planes at once
    (64, 49, 5), (49, 64, 4), (256, 13, 3), (17, 211, 4), (2048, 2, 3), (3, 1025, 5),   # lines, segments of 8
    (121, 41, 4), (63, 128, 5),                      # segments of 16
    (128, 80, 4), (101, 99, 3),                      # segments of 32
]


@pytest.mark.parametrize("n", GRIDS, ids=["x".join(map(str, g)) for g in GRIDS])
def test_direct_corrections_match_sparse_solve(ctx, n):
    from paper_1003_4570_gb300 import omen
    g = poisson.Grid(*n, 0.21 * n[0], 0.17 * n[1], 0.3 * n[2])
    rng = np.random.default_rng(sum(n))
    rho = rng.normal(size=g.shape) * 1e6 + 2e5
    ref = poisson.solve_direct(g, rho)
    for prec in (omen.OMEN_F64, omen.OMEN_F32_REFINE64):
        phi = torch.from_numpy(rng.normal(size=g.shape) * np.abs(ref).max()).cuda()
        info = omen.omen_poisson(ctx, g, torch.from_numpy(rho).cuda(), phi, rtol=1e-12, precision=prec)
        assert info["converged"] == 1 and info["rel_residual"] <= 1e-12
        np.testing.assert_allclose(phi.cpu().numpy(), ref, atol=1e-10 * np.abs(ref).max(), rtol=0)
        # already solved: nothing is done
        again = phi.clone()
        info = omen.omen_poisson(ctx, g, torch.from_numpy(rho).cuda(), again, rtol=1e-8, precision=prec)
        assert info["iterations"] == 0 and torch.equal(again, phi)


@pytest.mark.parametrize("n", [(3, 5, 8), (64, 49, 5), (33, 100, 6)], ids=["planes", "lines", "odd_lines"])
def test_from_the_zero_field(ctx, n):
    """The first residual from a zero start is the right-hand side; one component that is not zero
    must send it the general way."""
    from paper_1003_4570_gb300 import omen
    g = poisson.Grid(*n, 0.2 * n[0], 0.2 * n[1], 0.2 * n[2])
    rho = np.random.default_rng(5).normal(size=g.shape) * 1e6
    ref = poisson.solve_direct(g, rho)
    for last in (0.0, 1e6 * np.abs(ref).max()):
        phi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        phi[-1, -1, -1] = last
        omen.omen_poisson(ctx, g, torch.from_numpy(rho).cuda(), phi, rtol=1e-12)
        np.testing.assert_allclose(phi.cpu().numpy(), ref, atol=1e-10 * np.abs(ref).max(), rtol=0)


def test_iteration_limit_is_kept(ctx):
    from paper_1003_4570_gb300 import omen
    g = poisson.Grid(7, 6, 20, 1.4, 1.2, 4.0)
    rho = torch.from_numpy(np.random.default_rng(1).normal(size=g.shape) * 1e6).cuda()
    for limit in (1, 2, 4):
        phi = torch.zeros_like(rho)
        with pytest.raises(omen.OmenError) as e:
            omen.omen_poisson(ctx, g, rho, phi, rtol=1e-200, max_iter=limit)
        assert e.value.status == omen.OMEN_ENOCONV
