"""Projector kernels at the sizes where their tiles, lists and branches end,
against the FP64 oracle (the same bars as tests/test_gpu_projector.py).

The cases cover: x/y cell lists that end just before, at and after a chunk of
32 cells; a single voxel row or column; detectors whose mid-plane row falls in
the middle of a row group (rays going up and down in one warp), on a row
(odd heights) and on a group's edge; detectors taller than the volume's shadow
(rays that leave through the top) and shorter than it; one detector row;
several z blocks of the transpose; voxels that cover many pixels and pixels
that cover many voxels; steep cones with several z crossings per x/y cell."""
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


def geom(nx, ny, nz, nu, nv, du=1.0, dv=1.0, vox=(1.0, 1.0, 1.0), dso=120.0, dsd=200.0, angles=None):
    angles = np.radians([0.0, 31.0, 45.0, 90.0, 163.0, 257.0]) if angles is None else angles
    return synth.Geometry(nx, ny, nz, *vox, nu, nv, du, dv, dso, dsd, angles)


CASES = {
    "cells_31": geom(15, 16, 12, 40, 24),
    "cells_32": geom(16, 16, 12, 40, 24),
    "cells_33": geom(17, 16, 12, 40, 24),
    "cells_65": geom(33, 32, 20, 70, 44),
    "one_row": geom(40, 1, 10, 70, 20),
    "one_column": geom(1, 40, 10, 70, 20),
    "one_slice": geom(24, 24, 1, 50, 9),
    "mid_row_65": geom(20, 20, 40, 40, 65),
    "mid_row_129": geom(12, 14, 70, 30, 129),
    "mid_group_200": geom(12, 14, 90, 30, 200, dv=0.9),
    "tall_detector": geom(24, 20, 10, 44, 150, dv=0.7),
    "short_detector": geom(24, 20, 60, 44, 9),
    "one_detector_row": geom(24, 20, 12, 44, 1),
    "odd_slices": geom(18, 22, 33, 44, 61, vox=(1.0, 0.9, 0.8)),
    "z_blocks": geom(6, 7, 300, 14, 330, dv=1.5, dso=400.0, dsd=640.0),
    "many_pixels": geom(9, 8, 7, 150, 110, du=0.15, dv=0.15, dso=60.0, dsd=100.0),
    "many_voxels": geom(48, 44, 40, 9, 8, du=9.0, dv=9.0),
    "steep_cone": geom(16, 16, 60, 30, 90, dv=2.5, vox=(1.0, 1.0, 0.25), dso=20.0, dsd=60.0),
    "steep_cone_odd": geom(15, 16, 61, 31, 91, dv=2.5, vox=(1.0, 1.0, 0.2), dso=20.0, dsd=60.0),
    "many_angles": geom(10, 9, 34, 20, 40, angles=synth.circular_angles(97)),
}


def check(got, ref):
    got = np.asarray(got, np.float64).reshape(ref.shape)
    assert np.linalg.norm(got - ref) <= REL_L2 * np.linalg.norm(ref)
    bad = np.abs(got - ref) > 4 * REL_L2 * np.abs(ref) + 1e-5 * np.abs(ref).max()
    assert not bad.any(), "%d elements off, worst %g" % (bad.sum(), np.abs(got - ref)[bad].max())


@pytest.mark.parametrize("name", list(CASES))
def test_every_shape_at_the_edges(cbct, name):
    import torch
    g = CASES[name]
    gm = cbct.Geometry(g)
    x = synth.random_volume(g, 41).astype(np.float32)
    y = (synth.random_projections(g, 42) + 0.25).astype(np.float32)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    y_ref, x_ref = oracle.project(g, x.astype(np.float64)), oracle.backproject(g, y.astype(np.float64), 8)
    for rows in cbct.FWD_ROWS:
        cbct.set_launch(gm, rows, 0)
        check(cbct.project(gm, xd).cpu().numpy(), y_ref)
    for config in range(len(cbct.BWD_CONFIGS)):
        cbct.set_launch(gm, 1, config)
        check(cbct.backproject(gm, yd).cpu().numpy(), x_ref)
