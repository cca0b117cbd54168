"""Packed lists on both sides of the size where their counting and filling go from one round of
Gaussians per CTA to four (8 x 152 CTAs of 256): the lists in regions, which do not share that walk,
hold the same Gaussians in the same order; the per-tile counts given or not."""
import numpy as np
import pytest

import synth
from gpu_helpers import cuda, lib_ready, to_np_u32

pytestmark = pytest.mark.gpu

WAVE = 8 * 152 * 256


@pytest.mark.parametrize("G", [255, 257, WAVE - 1, WAVE, WAVE + 1, WAVE + 1025])
@pytest.mark.parametrize("ext_counts", [False, True])
def test_packed_equals_regions(G, ext_counts):
    import torch
    abi = lib_ready()
    gx, gy, cap = 60, 40, 4096
    rect, depth = synth.random_rects_depths(G, G, gx, gy, max_span=4, equal_depth_frac=0.05)
    area = np.maximum(rect[:, 2] - rect[:, 0], 0) * np.maximum(rect[:, 3] - rect[:, 1], 0)
    key = depth.astype(np.float32).view(np.uint32).copy()
    key[area == 0] = 0xFFFFFFFF
    packed = np.stack([rect[:, 0] | (rect[:, 1] << 16), rect[:, 2] | (rect[:, 3] << 16)], 1)
    packed = np.where(area[:, None] > 0, packed, 0).astype(np.uint32)
    k, r, a = cuda(key.view(np.int32)), cuda(packed.view(np.int32)), cuda(area.astype(np.int32))
    P = int(area.sum())
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    pk, pg = (torch.zeros(gx * gy * cap, dtype=torch.int32, device="cuda") for _ in range(2))
    regions = torch.zeros(gx * gy, 2, dtype=torch.int32, device="cuda")
    scr = torch.empty(abi.sort_bins_scratch_bytes(gx * gy), dtype=torch.uint8, device="cuda")
    abi.sort_bins(k, r, a, G, G, gx, gy, abi.tile_bins(pk, pg, cap), regions, counts, scr)
    assert dict(zip(abi.COUNT_FIELDS, to_np_u32(counts).tolist()))["overflow"] == 0
    want = to_np_u32(regions).reshape(-1, 2).astype(np.int64)
    lens = want[:, 1] - want[:, 0]
    counts.zero_()
    pairs = torch.zeros(P, dtype=torch.int32, device="cuda")
    ranges = torch.zeros(gx * gy, 2, dtype=torch.int32, device="cuda")
    scr = torch.empty(abi.sort_scratch_bytes(G, P, gx * gy), dtype=torch.uint8, device="cuda")
    abi.sort(k, r, a, G, G, gx, gy, pairs, ranges, P, counts, scr,
             tile_count=cuda(lens.astype(np.int32)) if ext_counts else None)
    c = dict(zip(abi.COUNT_FIELDS, to_np_u32(counts).tolist()))
    assert c["overflow"] == 0 and c["n_pairs"] == P == lens.sum()
    got = to_np_u32(ranges).reshape(-1, 2).astype(np.int64)
    assert np.array_equal((got[:, 1] - got[:, 0]), lens)
    flat = to_np_u32(pg)
    expect = np.concatenate([flat[x:y] for x, y in want])
    assert np.array_equal(to_np_u32(pairs), expect)
