"""Solves whose multigrid levels run several steps per launch (a 2D level's two legs, the coarse
end of the V-cycle in one CTA per column, the whole PCG of a column in one) against the same solves
with one launch per step (smem_tail 15): every value and every FP32 partial sum is formed by
the same operations in the same order, so the solutions, the iteration counts and the refinement
steps are equal bit for bit.  Grids around the legs' 32 x 16 tile and the one-CTA limits, coarsest
grids of several sizes, one column (scalar layout) and groups of four with empty places, one to
four sweeps, stiffness (axis stencil), prior (all Kuhn edges) and mass, a row grid that is
capped (the <r, z> sums then run over rows far apart), and a level from which on steps are
joined."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
RTOL = 1e-9
# a whole PCG in one CTA, with the coarsest grid's inverse in shared memory (as a triangle) or not
SMALL = [(2, 1), (2, 16), (2, 32), (2, 33), (2, 48), (2, 64), (2, 70), (3, 1), (3, 5), (3, 8), (3, 12), (3, 16)]
LARGER = [(2, 72), (2, 88), (2, 104), (2, 112), (2, 128), (2, 160), (3, 20), (3, 24), (3, 36)]


def solves(P, cols, settings):
    rng = np.random.default_rng(P.n + cols)
    m = 0.4 * torch.tensor(rng.standard_normal(P.n), device=DEV)
    B = torch.tensor(rng.standard_normal((cols, P.n) if cols > 1 else P.n), device=DEV)
    if cols > 2:
        B[1] = 0.0
    out = []
    for kw in settings:
        P.set_tuning(**kw)
        P.set_point(m)
        out.append([s(B) for s in (P.state_solve, P.prior_solve, P.mass_solve)])
    for other in out[1:]:
        for i, ((x0, s0), (x1, s1)) in enumerate(zip(out[0], other)):
            assert torch.equal(x0, x1), (i, float((x0 - x1).abs().max()), s0, s1)
            assert s0 == s1, (i, s0, s1)


@pytest.mark.parametrize("dim,N", SMALL + LARGER)
@pytest.mark.parametrize("cols,nu,nu_coarse", [(1, 3, 0), (1, 2, 1), (6, 3, 0), (6, 1, 0), (6, 2, 4), (5, 4, 2)])
def test_same_bits_as_one_launch_per_step(dim, N, cols, nu, nu_coarse):
    from paper_1909_03948_gb300 import Problem
    w = W.make_workload(dim, N, 10, seed=411)
    P = Problem(dim, N, w.gamma, w.delta, 0.01, W.draws(w).obs_xyz, rtol=RTOL)
    kw = {"nu": nu, "nu_coarse": nu_coarse}
    solves(P, cols, [dict(kw), dict(kw, smem_tail=15), dict(kw, smem_tail=2)])
    P.close()


@pytest.mark.parametrize("N,cols,max_blocks", [(128, 40, 256), (96, 9, 64)])
def test_same_bits_with_a_capped_grid(N, cols, max_blocks):
    from paper_1909_03948_gb300 import Problem
    w = W.make_workload(2, N, 10, seed=413)
    P = Problem(2, N, w.gamma, w.delta, 0.01, W.draws(w).obs_xyz, rtol=RTOL)
    solves(P, cols, [{"max_blocks": max_blocks}, {"max_blocks": max_blocks, "smem_tail": 15}])
    P.close()


def test_same_bits_after_a_change_of_precision():
    """The coarse inverse made in FP64 (plain FP64 solves) serves FP32 solves afterwards."""
    from paper_1909_03948_gb300 import Problem
    w = W.make_workload(2, 48, 10, seed=415)
    P = Problem(2, 48, w.gamma, w.delta, 0.01, W.draws(w).obs_xyz, rtol=RTOL, precision="fp64")
    P.set_point(torch.zeros(P.n, dtype=torch.float64, device=DEV))
    P.set_precision("fp32_ir")
    solves(P, 3, [{}, {"smem_tail": 15}])
    P.close()


@pytest.mark.parametrize("N,cols", [(32, 330), (38, 700), (72, 250), (100, 45)])
def test_same_bits_for_many_columns(N, cols):
    """Column counts past the limits of the one-CTA PCG and of badly filled leg tiles (part of the
    levels, or all, then run one launch per step)."""
    from paper_1909_03948_gb300 import Problem
    P = Problem(2, N, 0.1, 0.5, 0.01, np.zeros((0, 2)), rtol=RTOL)
    solves(P, cols, [{}, {"smem_tail": 15}, {"smem_tail": 2}])
    P.close()
