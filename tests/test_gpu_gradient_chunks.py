"""Gradients of batches whose layers' output gradients are not all kept: they
run through 8, 4 and 2 slots in chunks of layers, forwards and backwards in
turn, where one image of the batch takes all its layers at once.

With 2^k images of equal sigma the batch's output gradients are the single
images' scaled by 2^-k, bit for bit, so its gradients are the single ones'
mean up to the sums: each is off by about 1e-5 of its terms' magnitudes, which
cancel by up to ten in a layer's gradient: 1e-4.  A wrong slot is off by 1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B", [4, 8, 16])
def test_chunked_backward_equals_single_images(B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    from paper_1609_04661_gb300.binding import unflatten_params
    gen = torch.Generator(device="cuda").manual_seed(B)
    x = torch.rand((B, 512, 512), generator=gen, device="cuda")
    r = x + 0.25 * torch.randn(x.shape, generator=gen, device="cuda")
    one = np.float32([0.25])
    mean, losses = 0.0, []
    with dg.CNN(17, seed=3) as net:
        for b in range(B):
            loss, g = net.gradients(r[b:b + 1], x[b:b + 1], one)
            mean = mean + g.astype(np.float64) / B
            losses.append(loss)
    with dg.CNN(17, seed=3) as net:
        loss, g = net.gradients(r, x, np.repeat(one, B))
    assert loss == pytest.approx(np.mean(losses), rel=1e-6)
    for got, want in zip(*(unflatten_params(v) for v in (g, mean))):
        for a, b in zip(got, want):
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
