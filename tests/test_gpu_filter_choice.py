"""Reading a plan's tuning and writing it back changes nothing: a solve in the
three-kernel form, whose H a changed filter_mode would replace, stays the same
bit for bit; changing filter_mode does replace it, and the single steps follow
either way."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# the small plans take the Toeplitz form for single steps, the wide one the FFT
@pytest.mark.parametrize("n,nv,nd", [(16, 3, 24), (40, 7, 57), (64, 30, 95), (32, 3, 1449)])
@pytest.mark.parametrize("moments", [0, 1])
def test_writing_the_tuning_back_is_neutral(n, nv, nd, moments):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    ph = synth.random_phantom(n, 4, 9)
    y = synth.poisson_counts(synth.analytic_sinogram(ph, synth.view_angles(nv), nd), 1e4, 10)
    y = torch.as_tensor(y).cuda()
    with dg.Plan(n, nv, nd, c_tv=3.0, k_tv=20, damp_x=0.7, damp_s=0.7, output_moments=moments) as pl:
        pl.set_tuning(sino_fused=0)
        first = pl.solve(y, 1e4, 3)
        pl.set_tuning(**pl.tuning())
        assert torch.equal(pl.solve(y, 1e4, 3), first)
        out = {}
        for mode in (0, 1, 0):
            pl.set_tuning(filter_mode=mode)
            assert pl.tuning()["filter_mode"] == mode
            mu = pl.solve(y, 1e4, 3)
            assert mode not in out or torch.equal(mu, out[mode])
            out[mode] = mu
        assert not torch.equal(out[0], out[1])
        d = (out[0] - out[1]).double().norm() / out[0].double().norm()
        assert float(d) < 1e-3      # two orders of summation of the same operator
        assert np.isfinite(float(d))
