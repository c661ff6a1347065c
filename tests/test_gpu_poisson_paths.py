"""Calls of omen_poisson by the form of solve they take."""
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
