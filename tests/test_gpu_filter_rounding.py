"""H by FFT is as close to FP64 as a plain complex FP32 transform (scipy's) that
takes two views as one line, also where it matters most: near the highest
frequencies, whose bins are differences of the large low-frequency ones and
meet the largest gain.  10% is for the order of the additions, which differs
between the two; a line of half the length whose two halves are combined in
plain FP32 is 20% further off there."""
import numpy as np
import pytest

import synth
from oracle import precond
from oracle.geometry import Geometry

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
fft = pytest.importorskip("scipy.fft")


def test_rounding_of_the_filter_near_the_highest_frequencies():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    err = np.zeros((2, 2))
    for n, nv, nd in ((64, 30, 95), (160, 32, 221), (295, 30, 427), (512, 64, 729), (640, 30, 909), (1024, 30, 1449)):
        g = Geometry(n, nv, nd)
        z = synth.analytic_sinogram(synth.random_phantom(n, 8, n), synth.view_angles(nv), nd).astype(np.float32)
        ref = precond.filter_views(z, g)
        P = g.P
        f = np.minimum(np.arange(P), P - np.arange(P)) / P
        gain = np.sqrt(np.maximum(f, 1 / (2 * P))).astype(np.float32)
        spec = fft.fft((z[0::2] + 1j * z[1::2]).astype(np.complex64), n=P, axis=1)
        assert spec.dtype == np.complex64
        pair = fft.ifft(spec * gain, axis=1)[:, :nd]
        plain = np.empty_like(z)
        plain[0::2], plain[1::2] = pair.real, pair.imag
        with dg.Plan(n, nv, nd) as pl:
            if pl.tuning()["filter_mode"] != 0:
                pl.set_tuning(filter_mode=0)
            out = pl.filter(torch.as_tensor(z).cuda()).cpu().numpy()
        for k, v in enumerate((out, plain)):
            d = v.astype(np.float64) - ref
            e = np.abs(np.fft.rfft(d, n=P, axis=1)) ** 2
            err[k] += [np.log(e[:, 63 * (P // 2) // 64:].sum()) / 2, np.log((d ** 2).sum()) / 2]
    near, total = np.exp((err[0] - err[1]) / 6)      # geometric means over the sizes
    assert near <= 1.1 and total <= 1.1
