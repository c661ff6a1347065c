"""Calls of omen_poisson by the form of solve they take.

Checked by the residual b - A x with the oracle's matrix, whose bound does not depend on the grid's
condition (twice the tolerance asked for: the rest is the rounding of b - A x), and against the
oracle's sparse solve within the error that this residual allows, ||r|| / lambda_min."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import poisson  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    from paper_1003_4570_gb300 import omen
    return omen.omen_create(0, torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("n", [(8, 6, 20), (64, 50, 5)], ids=["planes", "lines"])
def test_lateral_spacing_far_below_the_vertical_one(ctx, n):
    """Charge without a lateral mean on a grid a thousand times finer in x and y than in z: pivots
    exact to rounding solve it to 1e-12 in one correction."""
    from paper_1003_4570_gb300 import omen
    g = poisson.Grid(*n, 1e-3 * n[0], 1e-3 * n[1], 1.0 * n[2])
    rho = np.random.default_rng(8).normal(size=g.shape) * 1e6
    rho -= rho.mean(axis=(1, 2), keepdims=True)
    phi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    info = omen.omen_poisson(ctx, g, torch.from_numpy(rho).cuda(), phi, rtol=1e-12)
    assert info["converged"] == 1 and info["iterations"] == 1
    # the laterally constant mode is a million times softer: the residual is what is well defined
    b = rho.ravel() / (poisson.EPS0 * g.eps_r)
    r = b - poisson.laplacian(g) @ phi.cpu().numpy().ravel()
    assert np.linalg.norm(r) <= 2e-12 * np.linalg.norm(b)


def residual(g, rho, phi):
    """||b - A phi|| and ||b||."""
    b = rho.ravel() / (poisson.EPS0 * g.eps_r)
    return np.linalg.norm(b - poisson.laplacian(g) @ phi.cpu().numpy().ravel()), np.linalg.norm(b)


# lines of more than 2,048 points, more than 1,024 planes, and few planes of lines with a large prime
@pytest.mark.parametrize("n", [(1, 1, 1100), (3, 2, 1027), (2050, 1, 4), (1, 2053, 3), (2049, 3, 12), (2039, 16, 3), (1021, 64, 3)],
                         ids=lambda n: "x".join(map(str, n)))
def test_iterated_grids_match_sparse_solve(ctx, n):
    """Conjugate gradients in both precisions, narrow and wide rows."""
    from paper_1003_4570_gb300 import omen
    g = poisson.Grid(*n, 0.21 * n[0], 0.17 * n[1], 0.3 * n[2])
    rho = np.random.default_rng(sum(n)).normal(size=g.shape) * 1e6
    ref = poisson.solve_direct(g, rho)
    rho_d = torch.from_numpy(rho).cuda()
    for rtol in (1e-10, 1e-8):
        for prec in (omen.OMEN_F64, omen.OMEN_F32_REFINE64):
            phi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
            info = omen.omen_poisson(ctx, g, rho_d, phi, rtol=rtol, precision=prec)
            assert info["converged"] == 1 and info["rel_residual"] <= rtol
            if max(n[:2]) > 2048 or n[2] > 1025:           # else the faster form is taken
                assert info["iterations"] > 2
            r, b = residual(g, rho, phi)
            assert r <= 2 * rtol * b
            smallest = 4 * np.sin(np.pi / (2 * g.nz)) ** 2 / g.h_m[2] ** 2
            assert np.linalg.norm(phi.cpu().numpy() - ref) <= 2 * rtol * b / smallest


# line by line with several runs of 64 pivots and chains of several segments: 16 unknowns a thread, 32 a
# thread with up to 256 and with more unknowns; planes at once with more than 256
@pytest.mark.parametrize("n", [(64, 49, 150), (128, 81, 200), (64, 80, 300), (9, 64, 400)], ids=lambda n: "x".join(map(str, n)))
def test_deep_grids(ctx, n):
    from paper_1003_4570_gb300 import omen
    g = poisson.Grid(*n, 0.21 * n[0], 0.17 * n[1], 0.3 * n[2])
    rho = np.random.default_rng(sum(n)).normal(size=g.shape) * 1e6 + 2e5
    rho_d = torch.from_numpy(rho).cuda()
    for prec in (omen.OMEN_F64, omen.OMEN_F32_REFINE64):
        phi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        info = omen.omen_poisson(ctx, g, rho_d, phi, rtol=1e-11, precision=prec)
        assert info["converged"] == 1 and info["iterations"] <= 2
        r, b = residual(g, rho, phi)
        assert r <= 2e-11 * b
