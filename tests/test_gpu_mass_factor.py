"""3D prior samples whose normals are drawn inside the mass factor equal the samples of the same
normals drawn first and passed in, at grid sizes around its tiles (one cell; one tile; last
tiles of every width; several z segments) and past one chunk of 64 samples: to 1e-8, the bound
the sampler's parity with the oracle has for identical normals."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,ns", [(1, 3), (2, 2), (3, 2), (5, 2), (8, 67), (16, 5), (24, 3), (32, 3), (40, 2), (64, 2)])
def test_drawn_and_given_normals_agree(N, ns):
    from paper_1909_03948_gb300 import Problem, philox_normals
    P = Problem(3, N, 0.1, 0.5, 0.01, np.zeros((0, 3)), rtol=1e-11)
    seed = 0x1234567_89abcdef
    eta = philox_normals(seed, 0, ns, P.nelems * 4)
    a, _, _ = P.laplace_sample(None, None, None, eta, want_post=False)
    b, _, _ = P.laplace_sample(None, None, None, want_post=False, seed=seed, nsamples=ns)
    rel = torch.linalg.norm(a - b, dim=1) / torch.linalg.norm(a, dim=1)
    assert float(rel.max()) <= 1e-8, rel
    P.close()
