"""CGLS in FP32 against the FP64 oracle on the same data, at sizes where 20
iterations are past the first converged directions, so that an error of a step
along itself is multiplied by the later steps.

Bar, from the roundings that remain: each of the 2 x 20 products carries a
relative error of at most about 1.5e-7 (FP32 lengths and sums at these sizes),
independent of one another, so they add up to sqrt(40) x 1.5e-7 = 9.5e-7."""
import numpy as np
import pytest

import oracle
import synth
from oracle import krylov

pytestmark = pytest.mark.gpu

BAR = 1e-6


@pytest.fixture(scope="module")
def cbct():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_14212_gb300 import cbct as mod
    return mod


def test_twenty_iterations(cbct):
    import torch
    g = synth.Geometry(32, 32, 32, 1.0, 1.0, 1.0, 64, 64, 1.2, 1.2, 1000.0, 1500.0, synth.circular_angles(60))
    op, gm = oracle.Operator(g), cbct.Geometry(g)
    worst = {}
    for seed in range(1, 9):
        x = synth.ellipsoid_phantom(g, 10, seed=seed, scale=0.16)
        b = synth.poisson_log_noise(oracle.project(g, x.astype(np.float64)), 1e5, seed=100 + seed).astype(np.float32)
        ref, _ = krylov.cgls(op, b.astype(np.float64).ravel(), 20)
        got, _ = cbct.cgls(gm, torch.from_numpy(np.ascontiguousarray(b.reshape(g.proj_shape))).cuda(), 20)
        got = got.cpu().numpy().astype(np.float64).ravel()
        worst[seed] = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    assert max(worst.values()) <= BAR, worst
