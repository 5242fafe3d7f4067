"""The sums over pixels in the network's weight and bias gradients are wider than FP32: with layers
set up so that every term is a known float (dL/dz = dz at each pixel of the last two layers,
their inputs 1), two large terms of opposite sign in different columns of an image cancel without
taking the small terms' digits with them, and terms whose sum leaves the float range give an
infinity, not a NaN.  Every expected value is exact."""
import numpy as np
import pytest

from oracle import unet as O
from test_gpu_unet import dev, unpack

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
S = 64


def gradients(dz):
    """Gradients of the last two layers for dL/dy = dz (zero on the image's border)."""
    from paper_1909_03948_gb300 import UNet
    ps = []
    for name, ci, co, k in O.LAYERS:
        w, b = np.zeros((co, ci, k, k), np.float32), np.zeros(co, np.float32)
        if name in ("dec1a", "dec1b"):
            b[:] = 1.0                      # inputs of dec1b and out: 1 everywhere
        if name == "out":
            w[:], b[:] = 1.0, -16.0         # y = 0, so that the residual is b
        ps.append(np.concatenate([w.ravel(), b]))
    net = UNet(S, S, batch_cap=1)
    net.set_params(np.concatenate(ps))
    x = np.zeros((1, 3, S, S), np.float32)
    x[0, 2] = 1.0
    sign = np.where(dz < 0, 1.0, -1.0)      # dL/dy = -diag w b with w = 1 / |b|^2, w |b| = 1
    aux = np.zeros((1, 4, S, S), np.float32)
    aux[0, 0] = sign * 2.0 ** -12
    aux[0, 1] = np.abs(dz)
    _, g = net.loss_grad(dev(x), dev(aux))
    net.close()
    return unpack(np.asarray(g))[-2:]


@pytest.mark.parametrize("big", [0.0, 2.0 ** 30])
def test_large_terms_cancel(big):
    rng = np.random.default_rng(3)
    dz = np.zeros((S, S))
    dz[1:-1, 1:-1] = rng.choice([-1.0, 1.0], (S - 2, S - 2))
    dz[:, 10] = dz[:, 20] = 0.0             # no other term beside a large one in its column
    dz[5, 10], dz[9, 20] = big, -big
    want = dz.sum()
    for gw, gb in gradients(dz):
        assert np.array_equal(gw, np.full(gw.shape, want)), (np.unique(gw), want)
        assert np.array_equal(gb, np.full(gb.shape, want)), (np.unique(gb), want)


def test_overflow_is_infinite():
    dz = np.zeros((S, S))
    dz[5, 10], dz[9, 20] = -(2.0 ** 127), -(2.0 ** 127)
    for gw, gb in gradients(dz):
        assert np.all(gw == -np.inf) and np.all(gb == -np.inf), (np.unique(gw), np.unique(gb))
