"""The transpose where a detector row lies in the plane between two slabs (an
odd number of rows, an even number of slabs): the row belongs to the slab that
the oracle and the forward projector give it, which for these spacings is the
lower one (nz / 2 * dz / dz rounds below nz / 2), and for `upper` the upper.

The cases reach each walk of the patch tile: rays going both ways in one stack
(24 and 96 slabs), stacks that meet at the mid-plane (384 slabs), one row or
several passing a plane inside a patch.  Bars as in tests/test_gpu_projector.py."""
import math

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

REL_L2 = 1e-5


@pytest.fixture(scope="module")
def cbct():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_14212_gb300 import cbct as mod
    return mod


def geom(nx, ny, nz, vox, nu, nv, pix, dso, dsd):
    return synth.Geometry(nx, ny, nz, vox, vox, vox, nu, nv, pix, pix, dso, dsd, synth.circular_angles(11) + 0.007)


CASES = {
    "near_24": geom(31, 31, 24, 100 / 31, 55, 39, 11.48, 200.0, 1200.0),
    "far_24": geom(10, 9, 24, 100 / 31, 24, 39, 4.0, 1000.0, 1500.0),
    "far_24_fine": geom(10, 9, 24, 100 / 31, 40, 79, 2.0, 1000.0, 1500.0),
    "stacks_96": geom(7, 6, 96, 100 / 36, 20, 121, 5.0, 1000.0, 1500.0),
    "stacks_384": geom(5, 4, 384, 100 / 53, 16, 441, 3.2, 4000.0, 6000.0),
    "stacks_384_fine": geom(5, 4, 384, 100 / 53, 40, 1101, 1.3, 4000.0, 6000.0),
    "upper": geom(10, 9, 24, 3.0, 24, 39, 4.0, 1000.0, 1500.0),
}


def check(got, ref):
    got = np.asarray(got, np.float64).reshape(ref.shape)
    assert np.linalg.norm(got - ref) <= REL_L2 * np.linalg.norm(ref)
    bad = np.abs(got - ref) > 4 * REL_L2 * np.abs(ref) + 1e-5 * np.abs(ref).max()
    assert not bad.any(), "%d elements off, worst %g" % (bad.sum(), np.abs(got - ref)[bad].max())


@pytest.mark.parametrize("name", list(CASES))
def test_middle_row(cbct, name):
    import torch
    g = CASES[name]
    assert math.floor((0.0 + 0.5 * g.nz * g.dz) / g.dz) == g.nz // 2 - (name != "upper")
    gm = cbct.Geometry(g)
    x = synth.random_volume(g, 61).astype(np.float32)
    check(cbct.project(gm, torch.from_numpy(x).cuda()).cpu().numpy(), oracle.project(g, x.astype(np.float64)))
    y = (synth.random_projections(g, 62) + 0.25).astype(np.float32)
    yd, ref = torch.from_numpy(y).cuda(), oracle.backproject(g, y.astype(np.float64), 8)
    for config in range(len(cbct.BWD_CONFIGS)):
        cbct.set_launch(gm, 1, config)
        check(cbct.backproject(gm, yd).cpu().numpy(), ref)
