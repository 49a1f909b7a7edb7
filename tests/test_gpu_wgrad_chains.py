"""Weight gradients of the hidden layers: how many additions the tensor core
strings together before a sum moves to FP32.

A 17-layer network with zero hidden weights and biases of 1 has activations of
1, and with one tap of powers of two in its last layer its output gradient
reaches the layer before unrounded, so that layer's weight gradients are exact
sums of known numbers, here mostly of one sign.  The tensor core cuts a running
sum off at about 2^-26 at each step of 16 pixels: S steps lose S 2^-28 of the
sum on average, and the FP32 additions after them 2^-23.  S is a fiftieth of the
layer's steps, at most 320, whatever the number of layers in the launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LAYERS = 17


@pytest.mark.parametrize("B,H,W", [(4, 64, 32), (8, 64, 64), (32, 64, 64), (4, 128, 128), (1, 512, 512),
                                   (16, 256, 256)])
def test_weight_gradient_chains(B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    rng = np.random.default_rng(B + H)
    w = np.zeros((9, 64), np.float32)
    w[4] = 2.0 ** rng.integers(-3, 3, 64) * rng.choice([1, -1], 64)
    bias = [np.ones(64, np.float32)] * (LAYERS - 1) + [np.float32([-w.sum()])]      # f = 0
    weights = [np.zeros(576, np.float32)] + [np.zeros(9 * 64 * 64, np.float32)] * (LAYERS - 2) + [w.reshape(-1)]
    flat = np.concatenate([v for pair in zip(weights, bias) for v in pair])
    r = torch.as_tensor(1 + rng.standard_normal((B, H, W))).bfloat16().float().cuda()
    with dg.CNN(LAYERS) as net:
        net.set_params(flat)
        _, grad = net.gradients(r, torch.zeros_like(r), np.ones(B, np.float32))
    at = 576 + 64 + (LAYERS - 3) * (9 * 64 * 64 + 64)
    got = grad[at:at + 9 * 4096].reshape(9, 64, 64).astype(np.float64)
    g = r.cpu().numpy().astype(np.float64) * (-2.0 / r.numel())
    steps = min(320, -(-B * H * sum(-(-min(W - x, 128) // 16) for x in range(0, W, 128)) // 50))
    for tap in range(9):
        dy, dx = tap // 3 - 1, tap % 3 - 1
        m = g[:, max(0, -dy):H - max(0, dy), max(0, -dx):W - max(0, dx)]     # pixels whose tap lies in the image
        err = np.abs(got[tap] - m.sum() * w[4]) / (np.abs(m).sum() * np.abs(w[4]))
        assert err.max() <= steps * 2.0 ** -28 + 2.0 ** -23
