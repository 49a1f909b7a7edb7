"""V^-1 x is as close to FP64 as one plain complex FP32 transform of the image
each way (scipy's, without the real input's symmetry) brings it; 10% is for
the order of the additions, which differs between the two.  A form that uses
the symmetry loses the share of the rounding that falls into the discarded
imaginary parts and mirrored frequencies, 15% to 25%."""
import numpy as np
import pytest

from oracle import precond
from oracle.geometry import Geometry

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
fft = pytest.importorskip("scipy.fft")


@pytest.mark.parametrize("n", [128, 200, 255])
def test_rounding_of_the_image_filter(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    g = Geometry(n, 3, n)
    k = np.arange(n) - (n - 1) / 2
    err = np.zeros((3, 2))
    for seed in range(3):
        rng = np.random.default_rng(seed)
        x = 0.002 * rng.standard_normal((n, n))
        for _ in range(8):
            cx, cy, a, b = *rng.uniform(-0.3, 0.3, 2), *rng.uniform(0.05, 0.2, 2)
            x += rng.uniform(0, 0.02) * (((k[None] / n - cx) / a) ** 2 + ((k[:, None] / n - cy) / b) ** 2 <= 1)
        x = x.astype(np.float32)
        ref = precond.v_inverse(x, g)
        m = 1 << (2 * n - 1).bit_length()
        f = np.fft.fftfreq(m)
        gain = np.sqrt(np.maximum(np.hypot(f[:, None], f[None]), 1 / (2 * g.P))).astype(np.float32)
        spec = fft.fft2(x.astype(np.complex64), s=(m, m))
        assert spec.dtype == np.complex64
        plain = fft.ifft2(spec * gain).real[:n, :n]
        with dg.Plan(n, 3, n) as pl:
            out = pl.precond_image(torch.as_tensor(x).cuda(), inverse=True).cpu().numpy()
        err[seed] = [np.linalg.norm(v.astype(np.float64) - ref) for v in (out, plain)]
    assert err[:, 0].sum() <= 1.1 * err[:, 1].sum()
