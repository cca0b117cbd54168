"""Tile lists of 513 to 1024 entries at the edges of the 128-entry chunks that they are merged from: whole
chunks, one entry more or less, an odd last run, with ties and equal depths, in both list forms."""
import numpy as np
import pytest

from gpu_helpers import cuda, lib_ready, to_np_u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ties", ["none", "some", "all"])
@pytest.mark.parametrize("form", ["packed", "regions"])
def test_chunk_edges(form, ties):
    """One tile per length, all in one call, the Gaussians in random order."""
    import torch
    abi = lib_ready()
    rng = np.random.default_rng(3)
    lens = [513, 514, 527, 576, 639, 640, 641, 767, 768, 769, 895, 896, 897, 960, 1022, 1023, 1024, 1025]
    gx, gy = 6, 3
    tile = rng.permutation(np.repeat(np.arange(len(lens)), lens))
    n = len(tile)
    depth = rng.uniform(1.0, 50.0, size=n).astype(np.float32)
    if ties == "some":
        depth = depth[rng.integers(0, n // 40, size=n)]
    elif ties == "all":
        depth[:] = 3.0
    key = depth.view(np.uint32)
    x, y = (tile % gx).astype(np.uint32), (tile // gx).astype(np.uint32)
    rect = np.stack([x | (y << 16), (x + 1) | ((y + 1) << 16)], 1)
    args = [cuda(a.view(np.int32)) for a in (key, rect, np.ones(n, np.uint32))]
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    ranges = torch.zeros(gx * gy, 2, dtype=torch.int32, device="cuda")
    if form == "packed":
        pairs = torch.zeros(n, dtype=torch.int32, device="cuda")
        scr = torch.empty(abi.sort_scratch_bytes(n, n, gx * gy), dtype=torch.uint8, device="cuda")
        abi.sort(*args, n, n, gx, gy, pairs, ranges, n, counts, scr)
    else:
        cap = 1100
        pk = torch.zeros(gx * gy * cap, dtype=torch.int32, device="cuda")
        pairs = torch.zeros(gx * gy * cap, dtype=torch.int32, device="cuda")
        scr = torch.empty(abi.sort_bins_scratch_bytes(gx * gy), dtype=torch.uint8, device="cuda")
        abi.sort_bins(*args, n, n, gx, gy, abi.tile_bins(pk, pairs, cap), ranges, counts, scr)
    got, r = to_np_u32(pairs), to_np_u32(ranges).reshape(-1, 2)
    assert to_np_u32(counts)[2] == n and to_np_u32(counts)[3] == 0
    order = np.lexsort((np.arange(n), key))
    for t, length in enumerate(lens):
        assert np.array_equal(got[r[t, 0]:r[t, 1]], order[tile[order] == t]), length
