"""The tile back-projection at the edges of its work split: tiles cut by the
image's edge, view counts that leave partial staging chunks (64 views at a
time, partial sums of 8), detectors narrower and wider than the image, explicit
angles in every octant; and rays that are not finite.

Weights within 2^-22 of the projector's (positions of 27 fraction bits) and
FP32 sums of at most a few hundred products: 5e-6 relative against FP64."""
import numpy as np
import pytest

from oracle import joseph
from oracle.geometry import Geometry

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ANG = tuple(np.pi * np.array([0.0, 0.25, 0.5, 0.75, 1.0, 1.25, 1.5, 1.75, 0.1, 0.6, 1.1, 1.6, -0.3, 2.9]))
GEOMS = [(2, 1, 2, None), (16, 8, 24, None), (17, 65, 30, None), (33, 130, 20, None), (100, 9, 400, None),
         (47, 14, 70, ANG), (256, 64, 364, None)]


def _dg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    return dg


@pytest.mark.parametrize("n,nv,nd,ang", GEOMS)
def test_tiles_match_the_oracle(n, nv, nd, ang):
    dg = _dg()
    s = np.random.default_rng(n + nv).standard_normal((nv, nd)).astype(np.float32)
    with dg.Plan(n, nv, nd, angles=ang) as pl:
        pl.set_tuning(bp_mode=1)
        out = pl.backproject(torch.as_tensor(s).cuda()).cpu().numpy().astype(np.float64)
    ref = joseph.back_project(s, Geometry(n, nv, nd, ang))
    assert np.linalg.norm(out - ref) <= 5e-6 * np.linalg.norm(ref)


def test_infinite_ray_reaches_only_the_pixels_it_taps():
    dg = _dg()
    n, nv, nd = 40, 9, 57
    s = np.random.default_rng(3).standard_normal((nv, nd)).astype(np.float32)
    s[4, 28] = np.inf
    e = np.zeros((nv, nd))
    e[4, 28] = 1.0
    with dg.Plan(n, nv, nd) as pl:
        pl.set_tuning(bp_mode=1)
        out = pl.backproject(torch.as_tensor(s).cuda()).cpu().numpy()
    w = joseph.back_project(e, Geometry(n, nv, nd))
    assert np.all(out[w > 1e-5] == np.inf)
    assert np.all(np.isfinite(out[w == 0.0]) | (np.abs(w[w == 0.0]) > 0))
