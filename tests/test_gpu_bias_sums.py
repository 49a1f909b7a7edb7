"""Bias gradients are FP32 sums, rounded to nearest.

A 4-layer network with zero hidden weights and biases of 1 has activations of
1 everywhere, and with one tap of powers of two in its last layer its output
gradient reaches the layer before unrounded: with a power of two of pixels and
a BF16 misfit, layer 2's bias gradient is the exact sum of known numbers.
About 64 additions reach one sum (16 of a row, the rows with a correction, 8
lanes, at most 38 groups and 4 threads), each off by 0.58 of 2^-25 of a sum of
terms of one sign: 8 x 0.58 x 2^-25 < 2^-22, of the sum of magnitudes.  (Sums
in the tensor core, which cuts off, were up to 2^-19.8 away.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LAYERS = 4


@pytest.mark.parametrize("B,H,W", [(1, 1, 1), (2, 4, 16), (32, 64, 64), (2, 8, 128), (1, 16, 256), (1, 512, 512),
                                   (16, 256, 256)])
@pytest.mark.parametrize("mean", [0.0, 1.0])
def test_bias_gradient_is_the_exact_sum(B, H, W, mean):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    rng = np.random.default_rng(B + H + W)
    w = np.zeros((9, 64), np.float32)
    w[4] = 2.0 ** rng.integers(-3, 3, 64) * rng.choice([1, -1], 64)
    bias = [np.ones(64, np.float32)] * (LAYERS - 1) + [np.float32([-w.sum()])]      # f = 0
    weights = [np.zeros(576, np.float32)] + [np.zeros(9 * 64 * 64, np.float32)] * (LAYERS - 2) + [w.reshape(-1)]
    flat = np.concatenate([v for pair in zip(weights, bias) for v in pair])
    r = torch.as_tensor(mean + rng.standard_normal((B, H, W))).bfloat16().float().cuda()
    with dg.CNN(LAYERS) as net:
        net.set_params(flat)
        _, grad = net.gradients(r, torch.zeros_like(r), np.ones(B, np.float32))
    at = 576 + 64 + (9 * 64 * 64) + 64 + 9 * 64 * 64
    got = grad[at:at + 64].astype(np.float64)
    g = r.cpu().numpy().astype(np.float64) * (-2.0 / r.numel())
    want, size = g.sum() * w[4], np.abs(g).sum() * np.abs(w[4])
    assert np.max(np.abs(got - want) / size) <= 2.0 ** -22
