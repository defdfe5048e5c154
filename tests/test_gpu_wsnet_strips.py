"""The warm-start network at sizes where its kernels' blocks take several work
items and strips of several rows, as training on 16 and serving 64 images of
256 x 256 do: the weight gradient's ring of staged rows is reused and its sums
are added to a slot that holds earlier ones; inference's ring of staged rows
wraps, its accumulators are given back, two rows share a read of the folded
last layer's weights, and the first layer's double buffers alternate.
Against the same network in plain torch in FP64."""
import numpy as np
import pytest

from helpers import to_dev, to_np
from oracle import wsnet as ON

pytestmark = pytest.mark.gpu

SMS = 152


def _layers(vec):
    import torch
    out, k = [], 0
    for ci, co in zip(ON.CHANNELS[:-1], ON.CHANNELS[1:]):
        w = vec[k:k + co * ci * 9].view(co, ci, 3, 3)
        k += co * ci * 9
        out.append((w, vec[k:k + co]))
        k += co
    assert k == vec.numel() and isinstance(vec, torch.Tensor)
    return out


def _forward(layers, x, dil, rounded=False):
    """Tap by tap; rounded: activations to BF16 after every layer but the last."""
    import torch
    H, W = x.shape[-2:]
    for l, ((w, bias), d) in enumerate(zip(layers, dil)):
        p = torch.nn.functional.pad(x, (d, d, d, d))
        y = bias.view(1, -1, 1, 1).expand(x.shape[0], -1, H, W)
        for ky in range(3):
            for kx in range(3):
                tap = p[:, :, ky * d:ky * d + H, kx * d:kx * d + W]
                y = y + torch.einsum("oc,bchw->bohw", w[:, :, ky, kx], tap)
        if l < len(layers) - 1:
            y = torch.relu(y)
            if rounded:
                y = y.bfloat16().double()
        x = y
    return x


def _params(seed):
    """Random weights and, so that they are seen, biases."""
    p = ON.init_params(seed)
    rng = np.random.default_rng(seed + 1)
    return ON.flatten([(w, 0.1 * rng.standard_normal(b.shape)) for w, b in p]).astype(np.float32)


def _rows_per_strip(B, H, W, d):
    """Of the 32 -> 32 weight gradient, and its blocks' items."""
    seg = 32 if d > 32 else 64
    columns, per_class = B * -(-W // seg), -(-H // d)
    rows = min(max(1, min(16, columns * H // (12 * SMS))), per_class)
    return rows, columns * d * -(-per_class // rows) / (2 * SMS)


@pytest.mark.parametrize("B,H,W_,dil", [
    (16, 256, 256, (1, 4, 16, 64, 4, 1)), (7, 250, 261, (2, 1, 33, 64, 5, 3)), (12, 201, 130, (1, 3, 40, 8, 2, 7))])
def test_gradients(gk, B, H, W_, dil):
    """The targets lie to one side of the outputs, so that a gradient's terms
    add up instead of cancelling: activations whose sign an FP32 forward pass
    gets wrong (some 1e-6 of them) then count for 1e-6 of it, and n products'
    rounding for about 2^-24.  Six layers follow one another; the bars of the
    network's other gradient tests, 1e-4 of a group's norm and 1e-5 for the
    loss, are loose, and one segment's row left out of the sums (64 of 313,000
    to 1,050,000 columns) is of that size.  Every element within 1e-3 of its
    group's largest."""
    import torch
    strips = [_rows_per_strip(B, H, W_, d) for d in dil[1:5]]
    assert max(r for r, _ in strips) > 2 and min(i for _, i in strips) > 2
    net = gk.WsNet(H, W_, B, dilations=dil)
    flat = _params(3)
    net.set_params(flat)
    rng = np.random.default_rng(B)
    x = to_dev(rng.standard_normal((B, 2, H, W_)).astype(np.float32))
    t = to_dev((8.0 + rng.standard_normal((B, 1, H, W_))).astype(np.float32))
    value, g = net.gradients(x, t)
    value2, g2 = net.gradients(x, t)
    assert value == value2 and np.array_equal(g, g2)
    # FP64, a sample at a time: the losses are means over all outputs
    vec = torch.from_numpy(flat).cuda().double().requires_grad_(True)
    grads, total = torch.zeros_like(vec), 0.0
    for k in range(B):
        out = _forward(_layers(vec), x[k:k + 1].double(), dil)
        lk, dout = ON.mse(out.detach().cpu().numpy(), to_np(t[k:k + 1]).astype(np.float64))
        total += lk / B
        grads += torch.autograd.grad(out, vec, torch.from_numpy(dout / B).cuda())[0]
    assert value == pytest.approx(total, rel=1e-5)
    got, ref = ON.unflatten(g.astype(np.float64)), ON.unflatten(grads.cpu().numpy())
    for l, (a, b) in enumerate(zip(got, ref)):
        for u, v in zip(a, b):
            assert np.linalg.norm(u - v) <= 1e-4 * np.linalg.norm(v), (l, np.linalg.norm(u - v), np.linalg.norm(v))
            assert np.abs(u - v).max() <= 1e-3 * np.abs(v).max(), l


@pytest.mark.parametrize("B,H,W_,dil", [
    (64, 256, 256, (1, 4, 16, 64, 4, 1)), (33, 250, 261, (2, 1, 33, 64, 5, 3)), (77, 251, 130, (3, 2, 7, 16, 5, 1))])
def test_bf16_inference(gk, B, H, W_, dil):
    """Bars of test_bf16_inference_tiles_and_edges: per element 2 % of the
    output's scale plus 1 % of the element (an element may differ by the BF16
    rounding of its inputs), 1 % of the norm."""
    import torch
    tiles = B * H * -(-W_ // 128)
    assert tiles >= 8 * 3 * SMS  # strips of two rows or more in the middle layers
    net = gk.WsNet(H, W_, B, dilations=dil)
    flat = _params(6)
    net.set_params(flat)
    x = to_dev(np.random.default_rng(B).standard_normal((B, 2, H, W_)).astype(np.float32))
    y = to_dev(np.full((B, 1, H, W_), np.nan, dtype=np.float32))
    net.infer_bf16(x, y)
    net.check()
    y2 = to_dev(np.zeros((B, 1, H, W_), dtype=np.float32))
    net.infer_bf16(x, y2)
    assert torch.equal(y, y2)
    layers = _layers(torch.from_numpy(flat).cuda().bfloat16().double())
    ref = torch.cat([_forward(layers, x[k:k + 2].bfloat16().double(), dil, rounded=True) for k in range(0, B, 2)])
    err = (y.double() - ref).abs()
    assert bool(torch.isfinite(y).all())
    assert bool((err <= 2e-2 * ref.abs().max() + 1e-2 * ref.abs()).all()), err.max()
    assert float(err.norm()) <= 1e-2 * float(ref.norm())
