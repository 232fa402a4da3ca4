"""A launch-shape cache written when other kernels ran behind the same shapes
reads as empty (CPU; no library call)."""
import json

from paper_2211_14212_gb300 import cbct

PARAMS = dict(nx=32, ny=32, nz=32, dx=1.0, dy=1.0, dz=1.0, nu=64, nv=64, du=1.2, dv=1.2, dso=1000.0, dsd=1500.0)


def test_choices_timed_with_the_column_tiles_are_not_taken(tmp_path):
    """Version 1 files were timed with column tiles behind every shape; the
    shapes' names, and so the keys, are the same."""
    path = tmp_path / "tune.json"
    key = cbct.tune_key(PARAMS, 60, "a device")
    path.write_text(json.dumps({"version": 1, "entries": {key: {"fwd_rows": 2, "bwd_config": 8}}}))
    store = cbct.TuneCache(path)
    assert store.get(key) is None
    store.put(key, {"fwd_rows": 4, "bwd_config": 5})
    assert store.get(key) == {"fwd_rows": 4, "bwd_config": 5}
    assert json.loads(path.read_text())["version"] == cbct.TUNE_CACHE_VERSION
