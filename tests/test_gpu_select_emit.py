"""Selection where its second pass goes from one tile per CTA to four (more than 3648 tiles of 2048
anchors): the entries, their weights and the counts against the selections of two halves of the
anchors, each of which takes the one-tile form.  Every anchor is judged by itself, so they are equal
bit for bit."""
import numpy as np
import pytest

from gpu_helpers import lib_ready, to_np_u32
import synth

pytestmark = pytest.mark.gpu

TILE, LINE = 2048, 3648


def select(abi, torch, pos, level, dL, cam, cap):
    n = pos.shape[0]
    idx = torch.full((max(cap, 1),), -1, dtype=torch.int32, device="cuda")
    w = torch.zeros(max(cap, 1), device="cuda")
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    scr = torch.empty(abi.lod_select_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    abi.lod_select(pos, level, dL, n, 8, 10, cam, True, idx, w, cap, counts, scr)
    return idx, w, dict(zip(abi.COUNT_FIELDS, to_np_u32(counts).tolist()))


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("tiles,extra", [(LINE, 0), (LINE, 1), (LINE + 2, 5), (LINE + 3, 0)])
def test_tiles_per_cta(tiles, extra, dense):
    import torch
    abi = lib_ready()
    n = tiles * TILE + extra
    g = torch.Generator(device="cuda").manual_seed(n)
    pos = torch.rand(n, 3, device="cuda", generator=g) * 400 - 200
    if dense:                                    # all in view and coarse enough to be kept
        pos = pos * 0.05
    level = torch.randint(0, 1 if dense else 8, (n,), device="cuda", generator=g).to(torch.uint8)
    dL = torch.rand(n, device="cuda", generator=g) * 0.3
    cam = synth.look_at_camera(np.array([150.0, -160.0, 40.0]), np.array([0.0, 0.0, 0.0]), 1920, 1080,
                               d_max=500.0)
    idx, w, c = select(abi, torch, pos, level, dL, cam, n)
    half = (tiles // 2) * TILE
    ia, wa, ca = select(abi, torch, pos[:half], level[:half], dL[:half], cam, half)
    ib, wb, cb = select(abi, torch, pos[half:], level[half:], dL[half:], cam, n - half)
    ma, mb = ca["n_selected"], cb["n_selected"]
    m = ma + mb
    assert m > (n // 2 if dense else n // 1000)
    assert c["n_selected"] == c["need_selected"] == m and c["overflow"] == 0
    assert c["n_gaussians"] == 10 * m
    want = torch.cat([ia[:ma], ib[:mb] + half])
    assert torch.equal(idx[:m], want) and torch.equal(w[:m], torch.cat([wa[:ma], wb[:mb]]))
    cap = m - 1 - m // 3                         # the cut falls inside a CTA's run of tiles
    ic, wc, cc = select(abi, torch, pos, level, dL, cam, cap)
    assert cc["n_selected"] == cap and cc["need_selected"] == m and cc["overflow"] & 1
    assert torch.equal(ic[:cap], want[:cap])
