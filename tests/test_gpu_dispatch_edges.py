"""Sizes at the edges of the kernels' dispatch rules and tiles, against the oracle."""
import pytest

from paper_2608_26140_b200 import workloads as wl

from test_gpu_predict_commit import test_predict_commit as check_predict_commit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,B,n_blk", [
    (1280, 4, 32),        # 128 rows: the last size of the one-SM kernel
    (1280, 3, 43),        # 129 rows: two SMs per tile, the second row tile nearly empty, K cut between clusters
    (2688, 3, 43),        # an odd number of 128-wide vocabulary units: one SM
    (65536, 5, 29),       # whole tiles, 145 rows
    (16384, 19, 31),      # whole tiles, 589 rows: three row pairs, the last one without a second row tile
])
def test_lm_head_tiles(V, B, n_blk):
    check_predict_commit(wl.TINY, V, B, 64, n_blk)
