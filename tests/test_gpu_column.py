"""FP32 solves whose work runs with one CTA per column: the whole PCG of problems of up to
5,120 nodes (2D and 3D, with and without multigrid levels, coarsest grids that fit in shared
memory and ones that do not), and the coarse end of larger problems' V-cycles.  Every solve
reaches its FP64 relative residual, and a block's columns equal the same columns solved one by
one bit for bit (the two differ in the vectors' layout and in nothing else)."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
RTOL = 1e-10


@pytest.mark.parametrize("dim,N", [(2, 1), (2, 3), (2, 16), (2, 17), (2, 30), (2, 33), (2, 48), (2, 64), (2, 70),
                                   (2, 72), (2, 100), (3, 1), (3, 4), (3, 5), (3, 8), (3, 9), (3, 12), (3, 16),
                                   (3, 20), (3, 24)])
@pytest.mark.parametrize("nu,nu_coarse", [(3, 0), (1, 0), (2, 4)])
def test_residuals_and_columns(dim, N, nu, nu_coarse):
    from paper_1909_03948_gb300 import Problem
    w = W.make_workload(dim, N, 10, seed=211)
    P = Problem(dim, N, w.gamma, w.delta, 0.01, W.draws(w).obs_xyz, rtol=RTOL)
    rng = np.random.default_rng(dim * 1000 + N)
    P.set_tuning(nu=nu, nu_coarse=nu_coarse)
    P.set_point(0.4 * torch.tensor(rng.standard_normal(P.n), device=DEV))
    s = 7
    B = torch.tensor(rng.standard_normal((s, P.n)), device=DEV)
    B[4] = 0.0                                       # a column that starts converged
    np_ = N + 1
    free = torch.ones(P.n, dtype=torch.float64, device=DEV)
    face = np_ ** (dim - 1)
    free[:face] = 0.0
    free[-face:] = 0.0
    for solve, apply, mask in ((P.state_solve, P.stiffness_apply, free), (P.prior_solve, P.prior_apply, None),
                               (P.mass_solve, P.mass_apply, None)):
        X, st = solve(B)
        b = B if mask is None else B * mask
        r = b - (apply(X) if mask is None else apply(X) * mask)
        nb = torch.linalg.norm(b, dim=1)
        nr = torch.linalg.norm(r, dim=1)
        # the solver's own test, evaluated anew in FP64 (its rounding: n ulps of |A| |x|)
        assert bool((nr <= RTOL * nb * (1 + 1e-3) + 1e-13 * nb).all()), (solve.__name__, (nr / nb).max())
        assert float(X[4].abs().max()) == 0.0
        assert st["iterations"] > 0 or float(nb.max()) == 0.0
        for j in (0, s - 1):
            x1, _ = solve(B[j])
            assert torch.equal(x1, X[j]), (solve.__name__, j)
    P.close()


def test_more_columns_than_sms():
    from paper_1909_03948_gb300 import Problem
    P = Problem(2, 32, 0.1, 0.5, 0.01, np.zeros((0, 2)), rtol=RTOL)
    B = torch.tensor(np.random.default_rng(5).standard_normal((321, P.n)), device=DEV)
    X, _ = P.prior_solve(B)
    r = B - P.prior_apply(X)
    assert float((torch.linalg.norm(r, dim=1) / torch.linalg.norm(B, dim=1)).max()) <= RTOL * (1 + 1e-3) + 1e-13
    assert torch.equal(P.prior_solve(B[320])[0], X[320])
    P.close()
