"""The real-input FFT forms at their edges: H of a view as a complex line of
half the length (the shortest and longest lines, odd bin counts, one view), and
the image filter with rows in pairs and half the spectrum (odd sizes, a last
row alone, one to four columns per block), against the FP64 oracle at the
operators' 1e-5."""
import numpy as np
import pytest

from oracle import precond
from oracle.geometry import Geometry

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    return dg


@pytest.mark.parametrize("nv,nd", [(1, 2), (3, 3), (2, 5), (7, 95), (1, 1449), (5, 4096)])
def test_filter_by_half_length_fft(nv, nd):
    dg = _dg()
    s = np.random.default_rng(nd).standard_normal((nv, nd)).astype(np.float32)
    with dg.Plan(4, nv, nd) as pl:
        pl.set_tuning(filter_mode=0)
        t = torch.as_tensor(s).cuda()
        out = pl.filter(t).cpu().numpy().astype(np.float64)
        pl.filter(t, out=t)                                   # in place
        assert np.array_equal(t.cpu().numpy().astype(np.float64), out)
    ref = precond.filter_views(s, Geometry(4, nv, nd))
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [2, 3, 5, 16, 37, 301, 513, 1025])
@pytest.mark.parametrize("inverse", [True, False])
def test_image_filter_by_half_spectrum(n, inverse):
    dg = _dg()
    x = np.random.default_rng(n).standard_normal((n, n)).astype(np.float32)
    g = Geometry(n, 3, max(2, n))
    with dg.Plan(n, 3, max(2, n)) as pl:
        t = torch.as_tensor(x).cuda()
        out = pl.precond_image(t, inverse=inverse).cpu().numpy().astype(np.float64)
        pl.precond_image(t, inverse=inverse, out=t)           # in place
        assert np.array_equal(t.cpu().numpy().astype(np.float64), out)
    ref = precond.v_inverse(x, g) if inverse else precond.v_forward(x, g)
    assert np.linalg.norm(out - ref) <= 1e-5 * np.linalg.norm(ref)
