"""3D prior and mass solves of blocks large enough for the z-marching kernel on grids that fill its
xy tiles badly, where the prior keeps the row kernels and the mass matrix's Chebyshev iteration still
marches: each reaches its FP64 residual and agrees with the columns solved one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-10


@pytest.mark.parametrize("N,cols", [(20, 221), (36, 42)])
def test_prior_and_mass_solves(N, cols):
    from paper_1909_03948_gb300 import Problem
    P = Problem(3, N, 0.07, 0.6, 0.01, np.zeros((0, 3)), rtol=RTOL)
    B = torch.tensor(np.random.default_rng(N).standard_normal((cols, P.n)), device="cuda")
    for solve, apply in ((P.prior_solve, P.prior_apply), (P.mass_solve, P.mass_apply)):
        X, _ = solve(B)
        rel = torch.linalg.norm(B - apply(X), dim=1) / torch.linalg.norm(B, dim=1)
        assert float(rel.max()) <= RTOL * (1 + 1e-3) + 1e-13, float(rel.max())
        x1, _ = solve(B[cols - 1])
        assert float(torch.linalg.norm(X[-1] - x1) / torch.linalg.norm(x1)) <= 1e-8
    P.close()
