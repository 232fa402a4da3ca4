"""Ray sums of 16-bit volumes are compensated term by term (include/cbct.h,
cbct_project): a ray through 64 voxels, a large one, 62 small ones each below
half an ulp of the running sum, and the large one's negative.

All lengths and products here are exact (angle 0, voxels of 1, DSD 1024), so
the compensated sum is off by at most one rounding at the size of the largest
partial sum: an ulp of 61440 / 1024 = 60, 2^-18, times the ray's length 1024,
that is 2^-8, plus the 16-bit rounding of the result.  A plain sum loses the
small terms that follow the large one."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

LARGE, SMALL = 61440.0, 2.0 ** -10               # exact in FP16 and BF16


@pytest.fixture(scope="module")
def cbct():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_14212_gb300 import cbct as mod
    return mod


@pytest.mark.parametrize("nz,nv", [(1, 1), (3, 40)])
@pytest.mark.parametrize("dtype", ["float16", "bfloat16"])
def test_small_terms_are_kept(cbct, dtype, nz, nv):
    import torch
    # detector rows of 2^-6: all rays stay in the middle slab
    g = synth.Geometry(64, 1, nz, 1.0, 1.0, 1.0, 1, nv, 1.0, 2.0 ** -6, 512.0, 1024.0, np.array([0.0]))
    x = np.full(g.vol_shape, SMALL, np.float32)
    x[..., 0], x[..., -1] = LARGE, -LARGE
    exact = 62 * SMALL
    ulp16 = 2.0 ** (-11 if dtype == "float16" else -8) * exact
    gm = cbct.Geometry(g)
    for rows in cbct.FWD_ROWS:
        cbct.set_launch(gm, rows, 0)
        y = cbct.project(gm, torch.from_numpy(x).to(getattr(torch, dtype)).cuda()).float().cpu().numpy()
        assert np.abs(y - exact).max() <= 2.0 ** -8 + ulp16, (rows, y.ravel()[:4], exact)
