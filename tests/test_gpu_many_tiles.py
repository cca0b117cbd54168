"""Lists of more tiles than the warp sorter has warps (16 x 152 CTAs of four), one fewer and one more."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import lib_ready
from test_gpu_parity import _gpu_sort

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gx,gy", [(9727, 1), (128, 76), (139, 70), (300, 200)])
def test_lists(gx, gy):
    import torch
    abi = lib_ready()
    rect, depth = synth.random_rects_depths(gx, 60_000, gx, gy, max_span=4, equal_depth_frac=0.05)
    start, lst, _ = oracle.tile_lists(rect, depth.astype(np.float64), gx, gy)
    pg, tr, c, P = _gpu_sort(abi, torch, rect, depth, gx, gy)
    assert c["n_pairs"] == P == len(lst) and c["overflow"] == 0
    assert np.array_equal(pg[:P], lst)
    full = start[1:] > start[:-1]
    assert np.array_equal(tr[full, 0], start[:-1][full]) and np.array_equal(tr[full, 1], start[1:][full])
