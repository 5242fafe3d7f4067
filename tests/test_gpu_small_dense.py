"""The dense kernels of the eigensolver (Cholesky and triangular inverse of the R-Gram matrix,
Jacobi eigensolve of the projected operator) at widths from 1 to beyond each kernel's range (90: the
eigenvectors leave shared memory, 144: the Cholesky in shared memory ends), odd and
even: V is R-orthonormal and diagonalises the misfit Hessian.  The solves run at 1e-10, so the
Hessian's projection is within 1e-8 of diag(lambda), relative to the largest; 1e-7 is
the eigensolver's own bound on V^T R V."""
import numpy as np
import pytest

import workloads as W
from oracle.inverse import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def problem():
    from paper_1909_03948_gb300 import Problem
    w = W.WORKLOADS["small2d"]
    orc, m_true, _ = make_problem(w, W.draws(w))
    P = Problem(w.dim, w.N, w.gamma, w.delta, orc.sigma, orc.obs_xyz, d_obs=orc.d_obs, rtol=1e-10)
    yield P, torch.tensor(m_true, device=DEV)
    P.close()


@pytest.mark.parametrize("k,p", [(1, 0), (1, 1), (2, 1), (5, 2), (20, 13), (40, 20), (41, 20), (71, 20), (127, 20),
                                 (140, 20)])
def test_eigenpairs(problem, k, p):
    P, m = problem
    Om = torch.tensor(np.random.default_rng(k).standard_normal((k + p, P.n)), device=DEV)
    lam, V, _ = P.lowrank_eig(m, k, p, Om)
    P.set_point(m)
    eye = torch.eye(k, dtype=torch.float64, device=DEV)
    assert float((V @ P.R_apply(V).T - eye).abs().max()) <= 1e-7
    T = V @ P.hessian_apply(V)[0].T
    assert float((T - torch.diag(lam)).abs().max()) <= 1e-8 * float(lam[0])
    assert bool((lam[1:] <= lam[:-1]).all())
