"""A training pass that fits with two gradient slots runs, also where all its
layers' gradients would fit by themselves but leave no room for the rest of
the workspace."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_gradients_fall_back_to_two_slots():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    gen = torch.Generator(device="cuda").manual_seed(1)
    x = torch.rand((2, 512, 512), generator=gen, device="cuda")
    r = x + 0.25 * torch.randn(x.shape, generator=gen, device="cuda")
    s = np.float32([0.25, 0.25])
    with dg.CNN(17, seed=3) as net:
        net.gradients(r[:1, :96, :96].contiguous(), x[:1, :96, :96].contiguous(), s[:1])      # loads every kernel
        torch.cuda.empty_cache()
        before = torch.cuda.mem_get_info()[0]
        loss, g = net.gradients(r, x, s)
        used = before - torch.cuda.mem_get_info()[0]       # 16 slots of 64 MB for the activations and as many for the gradients
    assert used > 28 * (64 << 20)
    with dg.CNN(17, seed=3) as net:
        net.gradients(r[:1, :96, :96].contiguous(), x[:1, :96, :96].contiguous(), s[:1])
        torch.cuda.empty_cache()
        # all but 20 MB of what it took: the gradients still fit after the activations, the 30 MB of sums do not
        fill = torch.empty(torch.cuda.mem_get_info()[0] - used + (20 << 20), dtype=torch.uint8, device="cuda")
        try:
            loss2, g2 = net.gradients(r, x, s)
        finally:
            del fill
            torch.cuda.empty_cache()
    assert loss2 == loss
    assert np.linalg.norm(g2 - g) <= 1e-4 * np.linalg.norm(g)     # the sums' order alone differs
