"""The tensor-core convolution at the edges of its work split: runs of one,
two and many output rows per CTA, an accumulator ring that wraps, bands whose
last strip is ragged, images narrower than a strip and odd batches, against
the FP64 oracle.

A 3-layer network has one tensor-core layer, so the GPU and the BF16-rounding
oracle differ by FP32 summation order and the few roundings it flips (2^-8 of
an activation each, over 576 terms and 64 channels): 1e-3 relative, the
forward-mode derivative 5e-3 (a mask flips outright)."""
import numpy as np
import pytest

from oracle import cnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(1, 1, 1), (1, 2, 64), (3, 1, 130), (200, 1, 3), (161, 2, 5), (5, 63, 64), (3, 40, 65), (1, 2100, 2),
          (2, 300, 129)]


def rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("B,H,W", SHAPES)
def test_one_hidden_layer_matches_the_oracle(B, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    from paper_1609_04661_gb300.binding import flatten_params
    ws, bs = cnn.init_params(31, layers=3)
    rng = np.random.default_rng(B + 7 * H + 31 * W)
    bs = [np.asarray(rng.standard_normal(b.shape) * 0.05, dtype=np.float32).astype(np.float64) for b in bs]
    r = rng.standard_normal((B, H, W)).astype(np.float32)
    x = rng.standard_normal((B, H, W)).astype(np.float32)
    sig = np.exp(rng.uniform(-2, 0, B)).astype(np.float32)
    rt, xt = torch.as_tensor(r).cuda(), torch.as_tensor(x).cuda()
    with dg.CNN(3) as net:
        net.set_params(flatten_params(ws, bs))
        out = net.denoise(rt, sig).cpu().numpy()
        loss, grad = net.gradients(rt, xt, sig)
        ref = r - sig[:, None, None] * cnn.net_forward(r / sig[:, None, None].astype(np.float64), ws, bs, bf16=True)[0]
        assert rel(out, ref) < 1e-3
        ref_loss, gws, gbs = cnn.loss_and_grads(r, x, sig, ws, bs, bf16=True)
        assert abs(loss - ref_loss) < 1e-3 * abs(ref_loss)
        # the output gradient is rounded to BF16 between the layers (2^-9 each), the sums to FP32
        assert rel(grad, flatten_params(gws, gbs)) < 1e-2
        if B == 1:
            b = rng.standard_normal((H, W)).astype(np.float32)
            d, jb = net.denoise_jvp(rt[0].contiguous(), torch.as_tensor(b).cuda(), float(sig[0]))
            ref_d, ref_jb = cnn.denoise_jvp(r[0], b, float(sig[0]), ws, bs, bf16=True)
            assert rel(d.cpu().numpy(), ref_d) < 1e-3
            assert rel(jb.cpu().numpy(), ref_jb) < 5e-3
