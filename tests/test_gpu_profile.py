"""Profiling times every level-0 launch of a solve, in whichever form the solve runs it: a 2D
V-cycle's legs or its separate steps, a whole PCG in one CTA per column, the mass matrix's CG and its
Chebyshev iteration; and the legs can be replayed like the other kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"
STEPS = ("smooth", "resid_mg", "presmooth")


def profile(dim, N, cols, solve, **tuning):
    from paper_1909_03948_gb300 import Problem
    P = Problem(dim, N, 0.1, 0.5, 0.01, np.zeros((0, dim)), rtol=1e-8)
    P.set_tuning(**tuning)
    P.set_point(torch.zeros(P.n, dtype=torch.float64, device=DEV))
    B = torch.tensor(np.random.default_rng(N).standard_normal((cols, P.n)), device=DEV)
    P.profile_enable(True)
    _, st = getattr(P, solve)(B)
    prof = P.profile_read()
    P.profile_enable(False)
    P.close()
    assert all((cnt > 0) == (ms > 0.0) for cnt, ms in prof.values()), prof
    return {k: v[0] for k, v in prof.items()}, st


@pytest.mark.parametrize("solve", ["state_solve", "prior_solve"])
def test_level_legs_and_separate_steps(solve):
    c, st = profile(2, 128, 6, solve)
    assert c["leg_down"] == c["leg_up"] == c["vcycle"] == c["matvec"] == c["cg_update"] == st["iterations"]
    assert all(c[k] == 0 for k in STEPS + ("columns",))
    c, st = profile(2, 128, 6, solve, smem_tail=15)
    assert c["presmooth"] == c["resid_mg"] == c["vcycle"] == st["iterations"] and c["smooth"] == 4 * c["vcycle"]
    assert c["leg_down"] == c["leg_up"] == 0


def test_one_cta_per_column():
    c, st = profile(2, 32, 6, "state_solve")
    assert c["columns"] == st["outer"] and all(c[k] == 0 for k in STEPS + ("matvec", "vcycle", "cg_update"))


def test_mass_solves():
    c, st = profile(2, 128, 6, "mass_solve")
    assert c["matvec"] == c["cg_update"] == st["iterations"] and c["cheb_step"] == 0
    c, st = profile(3, 32, 60, "mass_solve")
    assert c["cheb_step"] == st["iterations"] and c["matvec"] == c["cg_update"] == 0


def test_replay_of_legs():
    from paper_1909_03948_gb300 import HPError, Problem
    for dim, N, nu, ok in ((2, 128, 3, True), (2, 64, 1, True), (2, 64, 4, False), (3, 16, 3, False)):
        P = Problem(dim, N, 0.1, 0.5, 0.01, np.zeros((0, dim)), rtol=1e-8)
        P.set_tuning(nu=nu)
        P.set_point(torch.zeros(P.n, dtype=torch.float64, device=DEV))
        B = torch.tensor(np.random.default_rng(N).standard_normal((6, P.n)), device=DEV)
        x0, _ = P.state_solve(B)
        for fam in ("leg_down", "leg_up"):
            if ok:
                assert 0.0 < P.replay_kernel(fam, 5)[0] < 1e4 and 0.0 < P.replay_kernel_graph(fam, 5) < 1e4
            else:
                with pytest.raises(HPError):
                    P.replay_kernel(fam, 5)
                with pytest.raises(HPError):
                    P.replay_kernel_graph(fam, 5)
        assert torch.equal(P.state_solve(B)[0], x0)
        P.close()


def test_samples_keep_cg():
    """The sampling update's mass solve runs by CG, the mass solves before and after it do not."""
    from paper_1909_03948_gb300 import Problem
    P = Problem(3, 32, 0.1, 0.5, 0.01, np.zeros((0, 3)), rtol=1e-8)
    B = torch.tensor(np.random.default_rng(1).standard_normal((60, P.n)), device=DEV)
    m = torch.zeros(P.n, dtype=torch.float64, device=DEV)
    lam, V = torch.ones(2, dtype=torch.float64, device=DEV), B[:2].clone()
    P.profile_enable(True)
    for call, cheb in ((lambda: P.mass_solve(B), True),
                       (lambda: P.laplace_sample(m, lam, V, want_prior=False, seed=3, nsamples=60), False),
                       (lambda: P.mass_solve(B), True)):
        call()
        assert (P.profile_read()["cheb_step"][0] > 0) == cheb
    P.close()
