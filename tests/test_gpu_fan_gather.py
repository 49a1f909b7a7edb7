"""The fan-beam back-projection's pixel form (bp_mode 1 where rays lie at least
half a pixel apart) at the edges of its work split: tiles cut by the image's
edge, views that leave a partial staging chunk (32 at a time, sums of 8), a
detector that does not cover the image, a far source; and a ray that is not
finite.

Positions carry 26 fraction bits plus an FP32 correction of about one bin at
most, so a weight is within 2^-21 of the projector's, and FP32 sums: 5e-6
relative against FP64."""
import numpy as np
import pytest

from oracle import fanbeam

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GEOMS = [(17, 1, 30, 40.0, 30.0, 1.95), (50, 37, 72, 88.0, 72.0, 1.95), (100, 40, 60, 176.0, 145.0, 1.95),
         (33, 9, 48, 1e7, 1e7, 2.0), (64, 33, 96, 112.0, 92.0, 1.95)]


def _plan(n, nv, nd, sd, dd, du):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    pl = dg.Plan(n, nv, nd, fan=dict(src_dist=sd, det_dist=dd, det_spacing=du))
    assert pl.tuning()["bp_mode"] == 1
    return pl


@pytest.mark.parametrize("n,nv,nd,sd,dd,du", GEOMS)
def test_pixel_form_matches_the_oracle(n, nv, nd, sd, dd, du):
    s = np.random.default_rng(n).standard_normal((nv, nd)).astype(np.float32)
    with _plan(n, nv, nd, sd, dd, du) as pl:
        out = pl.backproject(torch.as_tensor(s).cuda()).cpu().numpy().astype(np.float64)
    ref = fanbeam.back_project(s, fanbeam.FanGeometry(n, nv, nd, sd, dd, du))
    assert np.linalg.norm(out - ref) <= 5e-6 * np.linalg.norm(ref)


def test_infinite_ray_reaches_only_the_pixels_it_taps():
    n, nv, nd, sd, dd, du = GEOMS[4]
    s = np.random.default_rng(3).standard_normal((nv, nd)).astype(np.float32)
    s[4, 48] = np.inf
    e = np.zeros((nv, nd))
    e[4, 48] = 1.0
    with _plan(n, nv, nd, sd, dd, du) as pl:
        out = pl.backproject(torch.as_tensor(s).cuda()).cpu().numpy()
    w = fanbeam.back_project(e, fanbeam.FanGeometry(n, nv, nd, sd, dd, du))
    assert np.all(out[w > 1e-5] == np.inf)
    assert np.all(np.isfinite(out[w == 0.0]) | np.isinf(out[w == 0.0])) and np.mean(np.isfinite(out[w == 0.0])) > 0.99
