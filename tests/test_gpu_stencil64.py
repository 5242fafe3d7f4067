"""FP64 stencils of column blocks (K, A, M, C, C^T) over the flattened grid, against the FP64
oracle: node counts around a block's 256, odd column counts (a thread takes two columns), and
enough columns that a block makes several passes over the nodes.  K, A and M differ from the
oracle's products by rounding order only (1e-12); C and C^T also by the state they are
linearised at, which is solved at 1e-11 (1e-9).  Then solves whose right-hand sides have entries from
1 down to 1e-60 and zeros, which the FP64 -> FP32 conversion rounds to denormals and zeros: each
reaches its residual in FP64."""
import numpy as np
import pytest

import workloads as W
from oracle.inverse import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


def _t(X):
    return torch.tensor(np.ascontiguousarray(X.T), device=DEV)


def _err(Y, ref):
    Y = Y.cpu().numpy().T
    return float((np.linalg.norm(Y - ref, axis=0) / np.linalg.norm(ref, axis=0)).max())


@pytest.mark.parametrize("dim,N,cols", [(2, 14, 1), (2, 15, 3), (2, 16, 2), (2, 44, 5), (3, 5, 3), (3, 6, 1),
                                        (3, 12, 4), (3, 16, 1001)])
def test_stencils_against_the_oracle(dim, N, cols):
    from paper_1909_03948_gb300 import Problem
    w = W.make_workload(dim, N, 6, seed=W.SEED_BASE + 900 + N)
    dr = W.draws(w)
    orc, m_true, _ = make_problem(w, dr)
    P = Problem(dim, N, w.gamma, w.delta, orc.sigma, dr.obs_xyz, d_obs=orc.d_obs, rtol=1e-11)
    m = 0.7 * m_true
    P.set_point(torch.tensor(m, device=DEV))
    P.set_tuning(refine_df=0)
    X = W.random_block(orc.n, cols, 7)
    K = orc.stiffness(m).tolil()
    d = np.flatnonzero(orc.dmask)
    K[d, :] = 0
    K[:, d] = 0
    K[d, d] = 1.0
    assert _err(P.stiffness_apply(_t(X)), K.tocsr() @ X) < 1e-12
    assert _err(P.prior_apply(_t(X)), orc.A @ X) < 1e-12
    assert _err(P.mass_apply(_t(X)), orc.M @ X) < 1e-12
    u = orc.forward(m)
    assert _err(P.C_apply(_t(X)), orc.C_apply(m, u, X)) < 1e-9
    X[orc.dmask] = 0.0
    assert _err(P.Ct_apply(_t(X)), orc.Ct_apply(m, u, X)) < 1e-9
    P.close()


@pytest.mark.parametrize("dim,N", [(2, 48), (2, 96), (3, 32)])
def test_right_hand_sides_of_many_magnitudes(dim, N):
    from paper_1909_03948_gb300 import Problem
    P = Problem(dim, N, 0.07, 0.6, 0.01, np.zeros((0, dim)), rtol=1e-10)
    rng = np.random.default_rng(N)
    B = rng.standard_normal((5, P.n)) * 10.0 ** rng.uniform(-60, 0, (5, P.n)) * (rng.random((5, P.n)) > 0.2)
    B *= np.array([1.0, 1e-100, 1e100, 1e-30, 1e30])[:, None]
    B = torch.tensor(B, device=DEV)
    for solve, apply in ((P.prior_solve, P.prior_apply), (P.mass_solve, P.mass_apply)):
        X, _ = solve(B)
        rel = torch.linalg.norm((B - apply(X)) / B.abs().amax(1, True), dim=1) / torch.linalg.norm(
            B / B.abs().amax(1, True), dim=1)
        assert float(rel.max()) <= 1e-10 * (1 + 1e-3) + 1e-13, rel
    P.close()
