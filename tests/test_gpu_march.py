"""3D prior and mass solves whose FP32 stencils run as the z-marching kernel (blocks with enough
values), on grids with one tile, a last tile of every width and several, segments of 8 and 16
planes, groups with empty columns, an anisotropic prior with a Robin boundary (the coupling
coefficients then differ per direction and at the boundary): each solve reaches its FP64
residual, at multigrid's rate, and agrees with the same solve run in column chunks small
enough for the row kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
RTOL = 1e-10


@pytest.mark.parametrize("N,cols", [(24, 130), (32, 56), (32, 121), (40, 30), (48, 18), (64, 7), (64, 29)])
@pytest.mark.parametrize("aniso", [False, True])
@pytest.mark.parametrize("nu", [3, 1])
def test_prior_and_mass_solves(N, cols, aniso, nu):
    from paper_1909_03948_gb300 import Problem
    kw = {}
    if aniso:
        kw = {"theta": np.array([[2.0, 0.3, -0.2], [0.3, 1.0, 0.1], [-0.2, 0.1, 0.7]]), "robin_beta": 0.8}
    P = Problem(3, N, 0.07, 0.6, 0.01, np.zeros((0, 3)), rtol=RTOL, **kw)
    B = torch.tensor(np.random.default_rng(N + cols).standard_normal((cols, P.n)), device=DEV)
    nb = torch.linalg.norm(B, dim=1)
    P.set_tuning(nu=nu)
    for solve, apply in ((P.prior_solve, P.prior_apply), (P.mass_solve, P.mass_apply)):
        P.set_tuning(nu=nu)
        X, st = solve(B)
        rel = torch.linalg.norm(B - apply(X), dim=1) / nb
        assert float(rel.max()) <= RTOL * (1 + 1e-3) + 1e-13, float(rel.max())
        P.set_tuning(nu=nu, col_chunk=1)             # one column at a time: row kernels
        X1, st1 = solve(B[:2])
        assert float(torch.linalg.norm(X[:2] - X1) / torch.linalg.norm(X1)) <= 1e-8
        assert st["iterations"] <= st1["iterations"] + 2 * st["outer"], (st, st1)
    P.close()
