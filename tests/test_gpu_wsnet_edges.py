"""Forward and gradients of the warm-start network at the edges of its
kernels' tiles: 256-pixel convolution tiles, 64- and 32-column segments and
strips of up to 16 rows of the weight gradient, dilations up to 64 wider than
the image, single rows and columns."""
import numpy as np
import pytest

from helpers import to_dev, to_np
from oracle import wsnet as ON

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W_,B,dil", [
    (1, 1, 1, (1, 1, 2, 33, 64, 1)), (3, 257, 1, (1, 4, 16, 64, 4, 1)), (70, 31, 2, (2, 33, 1, 32, 5, 3)),
    (17, 64, 3, (1, 1, 1, 1, 1, 1)), (40, 65, 2, (64, 64, 64, 64, 64, 64)), (130, 128, 1, (1, 4, 16, 64, 4, 1))])
@pytest.mark.parametrize("loss", ["mse", "energy"])
def test_gradients_at_edges(gk, H, W_, B, dil, loss):
    """Against the oracle in FP64: an FP32 sum of n products errs by about
    sqrt(n) 2^-24 of the terms' root mean square, and six layers of 288
    products follow one another, so 1e-4 of a group's norm is a loose bound
    (the bar of the network's other gradient tests); the loss 1e-5."""
    net = gk.WsNet(H, W_, B, dilations=dil)
    params = ON.init_params(5)
    net.set_params(ON.flatten(params).astype(np.float32))
    params = ON.unflatten(ON.flatten(params).astype(np.float32).astype(np.float64))
    net.set_loss(loss)
    rng = np.random.default_rng(H * W_)
    x = rng.standard_normal((B, 2, H, W_)).astype(np.float32)
    t = rng.standard_normal((B, 1, H, W_)).astype(np.float32)
    out, acts = ON.forward(params, x.astype(np.float64), dil)
    y = to_dev(np.zeros((B, 1, H, W_), dtype=np.float32))
    net.forward(to_dev(x), y)
    assert np.linalg.norm(to_np(y) - out) <= 1e-5 * np.linalg.norm(out)
    if loss == "mse":
        ref_loss, dout = ON.mse(out, t.astype(np.float64))
    else:
        ref_loss, dout = ON.energy(out, t.astype(np.float64), x[:, 0].astype(np.float64))
    grads = ON.backward(params, acts, dout, dil)
    value, g = net.gradients(to_dev(x), to_dev(t))
    assert value == pytest.approx(ref_loss, rel=1e-5)
    for l, ((gw, gb), (rw, rb)) in enumerate(zip(ON.unflatten(g.astype(np.float64)), grads)):
        assert np.linalg.norm(gw - rw) <= 1e-4 * np.linalg.norm(rw), l
        assert np.linalg.norm(gb - rb) <= 1e-4 * np.linalg.norm(rb) + 1e-12, l
