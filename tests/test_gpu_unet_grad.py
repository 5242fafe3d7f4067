"""Weight and bias gradients of the warm-start network's convolutions at the sizes where their
tiling has edges: images narrower than a warp on every level (down to one pixel), columns
that leave part of the last strip or unit empty, row counts around the 18-row units, batches
that leave part of the last set of units empty, and enough images for several sets per warp.
Bounds as in test_gpu_unet.py (ten times the error of the FP32-evaluated oracle plus 1e-4
relative, FP32 pipes)."""
import numpy as np
import pytest

from oracle import unet as O
from test_gpu_unet import batch, dev, make_params, unpack

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W", [(1, 8, 8), (3, 8, 8), (17, 16, 16), (1, 16, 136), (2, 144, 8), (5, 40, 72)])
def test_gradients_match_oracle(N, H, W):
    from paper_1909_03948_gb300 import UNet
    packed, ops = make_params(21)
    net = UNet(H, W, batch_cap=N, tensor_cores=False)
    net.set_params(packed)
    x, aux = batch(22, N, H, W)
    _, g = net.loss_grad(dev(x), dev(aux))
    net.close()

    def oracle(ps, xx, aa):
        y, cache = O.forward(ps, xx)
        _, dy = O.residual_loss(y, xx, aa)
        return O.backward(ps, cache, dy.astype(xx.dtype))
    go = oracle(ops, x.astype(np.float64), aux.astype(np.float64))
    g32 = oracle([(w.astype(np.float32), b.astype(np.float32)) for w, b in ops], x, aux)
    nrm = np.linalg.norm
    for (gw, gb), (ow, ob), (w32, b32), (name, *_) in zip(unpack(g.astype(np.float64)), go, g32, O.LAYERS):
        assert nrm(gw - ow) <= 10 * nrm(w32 - ow) + 1e-4 * nrm(ow), name
        assert nrm(gb - ob) <= 10 * nrm(b32 - ob) + 1e-4 * nrm(ob), name
