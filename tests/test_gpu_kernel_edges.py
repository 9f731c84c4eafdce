"""Kernels at the sizes where their tiling can go wrong: remainders, single tiles, the smallest and largest of a range."""
import numpy as np
import pytest

from tests.test_gpu_parity import TINY, _mlp_case

pytestmark = pytest.mark.gpu


# The row-by-row down projection: every register layout (1, 2, 3-4, 5-8 tokens), channel ranges shorter than a warp's group
# of 32, one group per warp, and several; rates that leave no kept row, a few (an odd last pair) and all of them.
@pytest.mark.parametrize("B,ff", [(1, 32), (2, 96), (3, 2080), (5, 160), (7, 12320), (2, 20512), (8, 20512)])
def test_down_rows_tiles(B, ff):
    cfg = dict(TINY, d_ff=ff)
    rates = [1000, 999, 960, 500, 37, 0, 750, 875]
    _mlp_case(cfg, B, rates[:B], seed=ff + B)
    _mlp_case(cfg, B, rates[::-1][:B], seed=ff + B + 1)
