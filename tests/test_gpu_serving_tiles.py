"""Served iterates of scans that take every transpose tile of the server, in
steps of several scans and in steps of one, against the single-request solver
at the same tiles and against the FP64 oracle.

The server and the solver sum every ray and voxel in the same order and group
only the FP64 sums of the norms differently, so their iterates differ by far
less than FP32 rounding grows to in 30 iterations: MIX_TOL.  The oracle is met
at k = 10, as in tests/test_gpu_serving.py."""
import numpy as np
import pytest

import oracle
import synth
from oracle import krylov

pytestmark = pytest.mark.gpu

MIX_TOL = 1e-5
ITER_TOL = 1e-4


@pytest.fixture(scope="module")
def cbct():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_14212_gb300 import cbct as mod
    return mod


def rel(a, b):
    a = np.asarray(a, np.float64).ravel()
    b = np.asarray(b, np.float64).ravel()
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def geom(nx, ny, nz, vox, nu, nv, pix, dso=1000.0, dsd=1536.0, angles=40):
    return synth.Geometry(nx, ny, nz, vox, vox, vox, nu, nv, pix, pix, dso, dsd, synth.circular_angles(angles) + 0.003)


# one patch a tile; two; two stacks; four stacks; one patch and several tiles
# along z; more than 12 columns across a patch; a steep cone, which no patch
# tile takes
SCANS = {
    "small": geom(20, 18, 24, 8.0, 40, 48, 8.0),
    "stack_64": geom(52, 50, 40, 5.0, 80, 70, 5.0),
    "stacks_70": geom(64, 64, 70, 3.0, 110, 150, 3.0),
    "stacks_130": geom(64, 64, 130, 2.0, 110, 230, 2.0),
    "deep_small": geom(14, 12, 130, 2.0, 40, 290, 1.5),
    "columns_17": geom(24, 20, 30, 8.0, 300, 70, 1.5 * 8.0 * 1.536 / 8.2),
    "steep": geom(20, 20, 30, 2.0, 40, 60, 6.0, dso=45.0, dsd=120.0),
}


def data(g, seed):
    b = oracle.project(g, synth.ellipsoid_phantom(g, 8, seed=seed).astype(np.float64))
    return b.astype(np.float32).astype(np.float64).ravel()


@pytest.fixture(scope="module")
def problems():
    return {n: (g, data(g, 70 + i), "lsqr" if i % 2 else "lsmr") for i, (n, g) in enumerate(SCANS.items())}


@pytest.mark.parametrize("iters", [10, 30])
def test_mixed_step_equals_solver(cbct, problems, iters):
    with cbct.Server(16 << 30, max_slots=8, schedule="share") as srv:
        ids = {n: srv.submit(g, b, solver, iters) for n, (g, b, solver) in problems.items()}
        mixed = {n: srv.wait(i, timeout=300).x for n, i in ids.items()}
    off = {}
    for n, (g, b, solver) in problems.items():
        xs, _ = getattr(cbct, solver)(cbct.Geometry(g), b.astype(np.float32), iters)
        off[n] = rel(mixed[n], xs)
        if iters == 10:
            ref, _ = getattr(krylov, solver)(oracle.Operator(g), b, iters)
            assert rel(mixed[n], ref) <= ITER_TOL, n
    assert max(off.values()) <= MIX_TOL, off


@pytest.mark.parametrize("g", [
    synth.Geometry(128, 128, 128, 2.0, 2.0, 2.0, 256, 256, 1.6, 1.6, 1000.0, 1536.0, synth.circular_angles(180)),
    synth.Geometry(48, 48, 48, 5.0, 5.0, 5.0, 256, 256, 1.6, 1.6, 1000.0, 1536.0, synth.circular_angles(90)),
    synth.Geometry(40, 40, 150, 2.0, 2.0, 2.0, 128, 400, 1.2, 1.2, 1000.0, 1536.0, synth.circular_angles(90))],
    ids=["128", "columns_above_12", "stacks_150"])
def test_step_of_one_scan_equals_solver(cbct, g):
    """Scans that fill a step alone: the single-request kernels, captured, from
    the same start, so every bit is the solver's, the FP64 norms included."""
    b = data(g, 90)
    with cbct.Server(16 << 30, max_slots=4) as srv:
        res = srv.wait(srv.submit(g, b, "lsqr", 30), timeout=300)
    xs, rep = cbct.lsqr(cbct.Geometry(g), b.astype(np.float32), 30)
    assert np.array_equal(np.asarray(res.report.resid), np.asarray(rep.resid))
    assert np.array_equal(res.x, np.asarray(xs).reshape(res.x.shape))
