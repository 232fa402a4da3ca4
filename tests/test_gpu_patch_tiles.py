"""The transpose's patch tiles where their stacks, lists, rows and crossings
end, in every tile configuration, against the FP64 oracle (the bars of
tests/test_gpu_projector.py), and the voxel-driven backprojector where its
tiles and the detector end.

The cases cover: depths just past one, two and four stacks of 64 voxels; an odd
number of slices (a slab around the mid-plane) and of rows; fewer angles than
angle ranges; a single voxel column; detectors shorter and narrower than the
volume's shadow; voxels of one to seven rows, and planes that one, two and
three rows pass inside a patch; patches that reach out of the volume; more than
eight and sixteen detector columns across a patch; three detector rows."""
import numpy as np
import pytest

import oracle
import synth
from oracle import krylov

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


def geom(nx, ny, nz, nu, nv, du=1.0, dv=1.0, vox=(1.0, 1.0, 1.0), dso=300.0, dsd=480.0, angles=None):
    angles = np.radians([0.0, 31.0, 45.0, 90.0, 117.0, 163.0, 200.5, 257.0, 300.0]) if angles is None else angles
    return synth.Geometry(nx, ny, nz, *vox, nu, nv, du, dv, dso, dsd, angles)


CASES = {
    "stack_65": geom(7, 6, 65, 16, 120),
    "stack_129": geom(6, 7, 129, 16, 220, dso=500.0, dsd=800.0),
    "stack_257": geom(5, 4, 257, 12, 430, dso=900.0, dsd=1440.0),
    "odd_slices": geom(11, 10, 33, 25, 51),
    "three_angles": geom(10, 9, 20, 24, 40, angles=np.radians([3.0, 100.0, 222.0])),
    "seventeen_angles": geom(10, 9, 70, 24, 120, angles=synth.circular_angles(17)),
    "one_column": geom(1, 1, 40, 9, 70),
    "short_detector": geom(12, 11, 80, 26, 61),
    "narrow_detector": geom(20, 18, 24, 17, 40),
    "one_row_voxels": geom(14, 12, 40, 28, 50, dv=1.7),
    "three_row_voxels": geom(14, 12, 40, 28, 150, dv=0.6),
    "seven_row_voxels": geom(10, 9, 16, 70, 130, du=0.45, dv=0.36, vox=(1.5, 1.5, 1.5)),
    "two_rows_pass": geom(12, 12, 56, 30, 130, dso=120.0, dsd=200.0),
    "three_rows_pass": geom(12, 12, 90, 30, 190, dso=120.0, dsd=200.0),
    "columns_9_to_16": geom(9, 8, 12, 90, 40, du=0.4),
    "columns_17_up": geom(9, 8, 12, 150, 40, du=0.25),
    "three_rows": geom(12, 10, 9, 24, 3, dv=4.0),
}


def check(got, ref):
    got = np.asarray(got, np.float64).reshape(ref.shape)
    assert np.linalg.norm(got - ref) <= REL_L2 * np.linalg.norm(ref)
    bad = np.abs(got - ref) > 4 * REL_L2 * np.abs(ref) + 1e-5 * np.abs(ref).max()
    assert not bad.any(), "%d elements off, worst %g" % (bad.sum(), np.abs(got - ref)[bad].max())


@pytest.mark.parametrize("name", list(CASES))
def test_transpose(cbct, name):
    import torch
    g = CASES[name]
    gm = cbct.Geometry(g)
    y = (synth.random_projections(g, 52) + 0.25).astype(np.float32)
    yd = torch.from_numpy(y).cuda()
    ref = oracle.backproject(g, y.astype(np.float64), 8)
    for config in range(len(cbct.BWD_CONFIGS)):
        cbct.set_launch(gm, 1, config)
        check(cbct.backproject(gm, yd).cpu().numpy(), ref)


@pytest.mark.parametrize("name", list(CASES))
def test_voxel_driven(cbct, name):
    import torch
    g = CASES[name]
    y = synth.random_projections(g, 53).astype(np.float32)
    got = cbct.backproject_voxel_driven(cbct.Geometry(g), torch.from_numpy(y).cuda()).cpu().numpy()
    check(got, krylov.VoxelDrivenBackprojector(g)(y.astype(np.float64)).reshape(g.vol_shape))
