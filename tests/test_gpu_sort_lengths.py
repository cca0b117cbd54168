"""Tile lists at the lengths where the sorters change: the warp sorter's 512, the merge sorter's
runs and buffers (4096 in regions; 2048 and 8192 packed) and the network's 16384, with ties and
equal depths, in both list forms."""
import numpy as np
import pytest

from gpu_helpers import cuda, lib_ready, to_np_u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ties", ["none", "some", "all"])
@pytest.mark.parametrize("n", [511, 512, 513, 1024, 1025, 1536, 2047, 2048, 2049, 4095, 4096, 4097,
                               8191, 8192, 8193, 16384, 16385])
def test_list_lengths(n, ties):
    import torch
    abi = lib_ready()
    rng = np.random.default_rng(n)
    depth = rng.uniform(1.0, 50.0, size=n).astype(np.float32)
    if ties == "some":
        depth = depth[rng.integers(0, n, size=n)]
    elif ties == "all":
        depth[:] = 3.0
    key = depth.view(np.uint32)
    gx, gy = 3, 2
    # every Gaussian covers tile (1, 0); the first 600 also the tile to its right
    rect = np.zeros((n, 2), np.uint32)
    rect[:, 0] = 1
    rect[:, 1] = 2 | (1 << 16)
    rect[:600, 1] = 3 | (1 << 16)
    tiles = np.where(np.arange(n) < 600, 2, 1).astype(np.uint32)
    order = np.lexsort((np.arange(n), key))
    want = {1: order, 2: order[order < 600]}
    args = [cuda(a.view(np.int32)) for a in (key, rect, tiles)]
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    ranges = torch.zeros(gx * gy, 2, dtype=torch.int32, device="cuda")
    P = int(tiles.sum())
    for form in ("packed", "regions"):
        counts.zero_()
        if form == "packed":
            pairs = torch.zeros(P, dtype=torch.int32, device="cuda")
            scr = torch.empty(abi.sort_scratch_bytes(n, P, gx * gy), dtype=torch.uint8, device="cuda")
            abi.sort(*args, n, n, gx, gy, pairs, ranges, P, counts, scr)
        else:
            cap = n
            pk = torch.zeros(gx * gy * cap, dtype=torch.int32, device="cuda")
            pairs = torch.zeros(gx * gy * cap, dtype=torch.int32, device="cuda")
            scr = torch.empty(abi.sort_bins_scratch_bytes(gx * gy), dtype=torch.uint8, device="cuda")
            abi.sort_bins(*args, n, n, gx, gy, abi.tile_bins(pk, pairs, cap), ranges, counts, scr)
        got, r = to_np_u32(pairs), to_np_u32(ranges).reshape(-1, 2)
        assert to_np_u32(counts)[2] == P and to_np_u32(counts)[3] == 0
        for t in range(gx * gy):
            lst = got[r[t, 0]:r[t, 1]]
            assert np.array_equal(lst, want.get(t, np.zeros(0))), (form, t)
