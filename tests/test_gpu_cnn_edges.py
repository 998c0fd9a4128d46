"""Warm-start network at the edges of its 128-pixel tiles and of the loss's cluster of CTAs.

Bars: five layers forward and five back, each rounding its operands to BF16 (relative 2^-9, up to 0.4 %
per layer with nothing averaged on an image of a few pixels), add up to 4 %: 6e-2 in relative L2.  The
loss sums in FP64 and is rounded to FP32; the prediction it is compared through is the same FP32 array:
1e-5.  The output gradient is FP32 arithmetic on that array, and every sum of the backward pass runs in a
fixed order: the gradient of the loss equals that of the same output gradient computed outside, bit for
bit.  (One that differs in its last bits turns BF16 roundings over, each worth 2^-9 of one pixel's value
in one channel: 1.4e-4 of the gradient at 128 pixels.)"""
import numpy as np
import pytest

from oracle import cnn as ref

torch = pytest.importorskip("torch")


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))


@pytest.mark.gpu
@pytest.mark.parametrize("k,B", [(1, 2), (5, 3), (8, 2), (16, 8), (33, 40)])
def test_network_at_tile_edges(k, B):
    """2 pixels, 75, exactly one tile, 16 tiles, and 341 tiles with a ragged last one (second tiles on
    some of 304 CTAs); images smaller than one CTA's share of the loss and larger than a cluster's."""
    from paper_2206_11009_gb300 import learn
    th = learn.init_params(7)
    rng = np.random.default_rng(k)
    for e in ref.param_layout()[0]:
        th[e["b"]:e["b"] + e["cout"]] = 0.1 * rng.standard_normal(e["cout"])
    net = learn.WarmNet(th)
    x, tgt, dy = (rng.standard_normal((B, 2, k, k)).astype(np.float32) for _ in range(3))
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    gx = torch.empty((B, 2, k, k), dtype=torch.float32, device="cuda")
    y = net.forward(cu(x)).cpu().numpy()
    g = net.backward(cu(x), cu(dy), gx).cpu().numpy()
    y_ref, cache = ref.forward(th.astype(np.float64), x.astype(np.float64))
    g_ref, gx_ref = ref.backward(th.astype(np.float64), cache, dy.astype(np.float64))
    assert _rel(y, y_ref) < 6e-2
    assert _rel(g, g_ref) < 6e-2
    assert _rel(gx.cpu().numpy(), gx_ref) < 6e-2
    loss = net.loss_and_grad(cu(x), cu(tgt))
    g1 = net.grad.cpu().numpy().copy()
    e = y.astype(np.float64) - tgt
    t = (e[:, 0] - e[:, 1]).mean(axis=(1, 2), keepdims=True) / 2
    r = np.stack([e[:, 0] - t, e[:, 1] + t], 1)
    want = (r * r).sum() / (2 * B * k * k)
    assert abs(loss - want) <= 1e-5 * want
    e = y - tgt   # FP32 from here, as the library forms it
    t = ((e[:, 0].astype(np.float64) - e[:, 1]).sum(axis=(1, 2), keepdims=True) / (2.0 * k * k)).astype(np.float32)
    inv = np.float32(1) / np.float32(B * k * k)
    g2 = net.backward(cu(x), cu(np.stack([(e[:, 0] - t) * inv, (e[:, 1] + t) * inv], 1))).cpu().numpy()
    assert np.array_equal(g1, g2)
