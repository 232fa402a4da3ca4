"""The roofline's ncu counters belong to the code they were taken on (CPU)."""
import os
import re

import bench
import synth


def test_hash_covers_every_projector_kernel_source():
    """Every header that holds projector kernels or their tiles changes the hash."""
    csrc = os.path.join(bench.ROOT, "paper_2211_14212_gb300", "csrc")
    names = [n for n in sorted(os.listdir(csrc)) if n in ("projector.cu", "transpose.cuh") or
             re.search(r"\b(patch_tile|forward_tile|backward_tile)\(const DevGeom", open(os.path.join(csrc, n)).read())]
    base = {n: "int f();\n" for n in names}
    assert "patch_tile.cuh" in names and "projector_device.cuh" in names
    for n in names:
        assert bench.projector_hash(dict(base, **{n: "int g();\n"})) != bench.projector_hash(base), n


def test_no_bound_is_named_without_the_issue_term(monkeypatch):
    g = synth.config("c2")
    monkeypatch.setattr(bench, "NCU_COUNTERS", {})
    rl = bench.roofline_block(g, 2.8e10, 13.0, 12.5, {"sm_mhz": 2070.0}, (4, 7))
    assert rl["t_bound"]["issue_ms"] is None and rl["t_bound"]["binding"] is None
