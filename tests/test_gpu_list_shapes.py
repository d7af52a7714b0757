"""Neighbour lists in mixed precision under every number of lanes per sink: the
chunk scan reads the pair records of the force pass, padded from eight lanes on
and shared by several warps above 32, with and without prediction in place."""
import numpy as np
import pytest

from _parity import state
from test_gpu_neighbours import _check_lists, _run

pytestmark = pytest.mark.gpu
SHAPES = [(64, 1, 16), (128, 2, 128), (256, 4, 64), (64, 8, 64), (256, 16, 256), (32, 32, 256), (128, 64, 512),
          (256, 128, 1024)]


@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("n_i", [2, 300])
@pytest.mark.parametrize("threads,j_lanes,j_tile", SHAPES)
def test_mixed_lists_at_every_lane_count(oracle_mod, threads, j_lanes, j_tile, n_i, order):
    from paper_1510_04068_gb300 import sp2
    n = 1501
    s = state(n, 17, order=order)
    idx = np.sort(np.random.default_rng(n_i).choice(n, n_i, replace=False)).astype(np.int32)
    h2 = np.random.default_rng(3).uniform(0.005, 0.05, n_i)
    launch = dict(threads=threads, i_per_thread=1, j_lanes=j_lanes, j_tile=j_tile, split_j=3, ctas_per_sm=0)
    if order == 6 and j_tile == 1024 and n_i > threads // j_lanes:  # 276 KB of shared memory
        with pytest.raises(sp2.SP2Error):
            _run(sp2, s, idx, h2, 512, order=order, precision=sp2.SP2_MIXED, eps2=1e-8, launch=launch)
        return
    _, cnt, lst = _run(sp2, s, idx, h2, 512, order=order, precision=sp2.SP2_MIXED, eps2=1e-8, launch=launch)
    assert cnt.max() > 0
    _check_lists(oracle_mod, s, idx, h2, cnt, lst, 512, True)
