"""Which fan beams the back-projection's pixel form takes, and how close both
forms of bp_mode 1 come to FP64.

The pixel form is for rays 1/2 to 3 pixels apart inside the image; its
position error is a share of a bin, so at wide spacings it would grow past
that of the ray-driven tiles, which take those.

Ray-driven tiles: a weight's fraction is cut to 23 bits, 2^-23 / sqrt 3 on
average against weights of 0.58 (1.2e-7), and the FP32 products and sums add
0.7e-7: 2e-7 relative allowed.  Pixel form: positions off by at most
17 x 2^-27 bins and the correction (about 2.5 bins beside a close source) by
3 units of 2^-24, times at most 3 pixels, under 2e-6 in a single weight: 1e-6
over the image."""
import math

import numpy as np
import pytest

from oracle import fanbeam

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def pixel_form(n, sd, dd, du, nd):
    """The condition of fan_gather_ok (csrc/fanbeam.cu): (holds, narrowest and widest spacing, slots)."""
    u, R = 0.5 * (nd - 1) * du, n / math.sqrt(2) + 1.0
    Rc, a = R + 12.0, np.pi * np.arange(1025) / 1024
    s, t = sd - Rc * np.cos(a), Rc * np.sin(a)
    slots = 16 * math.sqrt(2) * 1.02 * float(np.max((sd + dd) / du * np.hypot(s, t) / s ** 2)) + 8
    near = du * (sd - R) / math.hypot(sd + dd, u)
    far = du * (sd + R) * math.sqrt(2) / (sd + dd)
    return sd - Rc >= 1 and near >= 0.5 and far <= 3 and slots <= 64, near, far, slots


def _backproject(n, nv, nd, sd, dd, du, s):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    with dg.Plan(n, nv, nd, fan=dict(src_dist=sd, det_dist=dd, det_spacing=du)) as pl:
        assert pl.tuning()["bp_mode"] == 1
        return pl.backproject(torch.as_tensor(s).cuda()).cpu().numpy().astype(np.float64)


# one view and a tile that overhangs by 15 pixels; rays at their closest and at their widest; the
# most slots; a source close to the image
@pytest.mark.parametrize("n,nv,nd,sd,dd,du", [(17, 1, 30, 60.0, 50.0, 1.95), (40, 11, 120, 1e6, 1e6, 1.02),
                                              (40, 33, 40, 1e6, 1e6, 4.2), (64, 40, 96, 120.0, 100.0, 2.5),
                                              (50, 70, 72, 86.0, 72.0, 1.8), (17, 8, 24, 45.0, 25.0, 2.2)])
def test_pixel_form_at_its_limits(n, nv, nd, sd, dd, du):
    assert pixel_form(n, sd, dd, du, nd)[0]
    s = np.random.default_rng(n + nv).standard_normal((nv, nd)).astype(np.float32)
    out = _backproject(n, nv, nd, sd, dd, du, s)
    ref = fanbeam.back_project(s, fanbeam.FanGeometry(n, nv, nd, sd, dd, du))
    assert np.linalg.norm(out - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("du", [3.0, 16.0, 64.0])
def test_wide_rays_keep_the_projectors_weights(du):
    n, nv, sd, dd = 64, 40, 120.0, 100.0
    nd = max(8, int(2.2 * n * (sd + dd) / sd / du))
    assert not pixel_form(n, sd, dd, du, nd)[0]
    s = np.random.default_rng(5).standard_normal((nv, nd)).astype(np.float32)
    out = _backproject(n, nv, nd, sd, dd, du, s)
    ref = fanbeam.back_project(s, fanbeam.FanGeometry(n, nv, nd, sd, dd, du))
    assert np.linalg.norm(out - ref) <= 2e-7 * np.linalg.norm(ref)


def test_infinite_ray_spares_every_pixel_off_its_support():
    n, nv, nd, sd, dd, du = 64, 33, 96, 112.0, 92.0, 1.95
    v, d = 4, 48
    s = np.random.default_rng(3).standard_normal((nv, nd)).astype(np.float32)
    s[v, d] = np.inf
    out = _backproject(n, nv, nd, sd, dd, du, s)
    S, dirs = fanbeam.FanGeometry(n, nv, nd, sd, dd, du).rays()
    (sx, sy), (vx, vy) = S[v, d], dirs[v, d]
    c = (n - 1) / 2
    iy, ix = np.mgrid[:n, :n]
    # distance from the ray along its interpolated axis; rays reach pixels closer than 1
    if abs(vx) >= abs(vy):
        dist = np.abs(iy - (c - (sy + (ix - c - sx) * vy / vx)))
    else:
        dist = np.abs(ix - (sx + (c - iy - sy) * vx / vy + c))
    assert np.all(np.isfinite(out[dist > 1 + 1e-5])) and np.all(np.isinf(out[dist < 1 - 1e-5]))
