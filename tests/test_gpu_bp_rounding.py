"""The tile back-projection rounds no more than FP32 asks for.

Independent errors of a product, in units of 2^-24 of its size: the staged
ray's product 0.4, the weight's own rounding 0.5, its position (27 fraction
bits) and constants 0.5, the two additions into the partial sum 1.1; the
partial sums' additions 1.1 of the result.  Together 1.8 units; 2.2 allowed,
1.3e-7.  (Weights formed from 1 + A and 1 - 2 A, multiples of 2^-22 and 2^-23,
came to 2.8.)"""
import numpy as np
import pytest

from oracle import joseph
from oracle.geometry import Geometry

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nv,nd", [(64, 16, 95), (96, 30, 137), (128, 64, 182), (128, 73, 182), (160, 90, 230)])
def test_tiles_round_like_fp32(n, nv, nd):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1609_04661_gb300 as dg
    s = np.random.default_rng(n + nv).standard_normal((nv, nd)).astype(np.float32)
    with dg.Plan(n, nv, nd) as pl:
        pl.set_tuning(bp_mode=1)
        out = pl.backproject(torch.as_tensor(s).cuda()).cpu().numpy().astype(np.float64)
    ref = joseph.back_project(s, Geometry(n, nv, nd))
    assert np.linalg.norm(out - ref) <= 2.2 * 2.0 ** -24 * np.linalg.norm(ref)
