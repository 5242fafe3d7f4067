"""FP64 stencils (K, A, M, C, C^T) of blocks with an odd column count, whose last column a thread takes
alone: every column equals the same column applied by itself bit for bit, with one block of nodes,
several, and so many columns that a block makes several passes."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("dim,N,cols", [(2, 8, 3), (2, 33, 5), (3, 5, 3), (3, 18, 7), (3, 24, 1203)])
def test_columns_equal_single_columns(dim, N, cols):
    from paper_1909_03948_gb300 import Problem
    w = W.make_workload(dim, N, 6, seed=431)
    P = Problem(dim, N, w.gamma, w.delta, 0.01, W.draws(w).obs_xyz, rtol=1e-8)
    P.set_tuning(refine_df=0)
    rng = np.random.default_rng(N)
    P.set_point(0.4 * torch.tensor(rng.standard_normal(P.n), device=DEV))
    X = torch.tensor(rng.standard_normal((cols, P.n)), device=DEV)
    for apply in (P.stiffness_apply, P.prior_apply, P.mass_apply, P.C_apply, P.Ct_apply):
        Y = apply(X)
        for j in (0, 1, cols - 2, cols - 1):
            assert torch.equal(apply(X[j]), Y[j]), (apply.__name__, j)
    P.close()
