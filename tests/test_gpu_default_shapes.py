"""The transpose tile a scan gets by default: deep stacks only where there are
tiles enough for every SM (a 2 x 2 x 256 volume in four stacks is one block)."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,config", [(2, 256, 3), (24, 512, 3), (40, 65, 3), (64, 65, 5), (48, 200, 5), (32, 512, 5),
                                         (64, 200, 7), (48, 512, 7)])
def test_depth_by_number_of_tiles(n, nz, config):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2211_14212_gb300 import cbct
    g = synth.Geometry(n, n, nz, 1.0, 1.0, 1.0, 2 * n, 2 * nz, 0.8, 0.8, 1000.0, 1536.0, synth.circular_angles(3))
    assert cbct.get_launch(cbct.Geometry(g))[1] == config
