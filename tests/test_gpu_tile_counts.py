"""Per-tile pair counts where their form changes: a table of corners per CTA from 16 Gaussians per tile,
up to 12288 entries and 256 tiles a side, filled by the projection or, for the fused decode +
projection, by a pass of its own; one atomic per pair otherwise.  The counts must be those of the rectangles written beside them."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, lib_ready, to_np_u32
from test_gpu_fused import GAUSS, NAMES, _bufs

pytestmark = pytest.mark.gpu

GRIDS = [(48, 32, (1, 95, 96, 511, 512, 513, 3000)),          # 6 tiles
         (1920, 1080, (130_559, 130_560, 400_001)),           # 8160 tiles
         (2016, 1520, (194_000,)), (2032, 1520, (194_600,)),   # tables of 127 x 96 = 12192, 128 x 96 = 12288
         (2048, 1520, (200_000,)),                            # 129 x 96: too large
         (4096, 64, (17_000,)), (4112, 64, (17_000,)),        # 256 and 257 tiles a side
         (64, 4096, (17_000,)), (64, 4112, (17_000,))]


def counted(rect, gx, gy):
    """Pairs per tile of rectangles u32[n][2] (corners x | y << 16), by differences."""
    d = np.zeros((gy + 1, gx + 1), np.int64)
    x0, y0 = rect[:, 0] & 0xFFFF, rect[:, 0] >> 16
    x1, y1 = rect[:, 1] & 0xFFFF, rect[:, 1] >> 16
    for y, x, s in ((y0, x0, 1), (y1, x1, 1), (y0, x1, -1), (y1, x0, -1)):
        np.add.at(d, (y, x), s)
    return d.cumsum(0).cumsum(1)[:gy, :gx].ravel()


def check(b, n, gx, gy):
    rect = to_np_u32(b["rect"]).reshape(-1, 2)[:n]
    area = ((rect[:, 1] & 0xFFFF) - (rect[:, 0] & 0xFFFF)) * ((rect[:, 1] >> 16) - (rect[:, 0] >> 16))
    assert np.array_equal(area, to_np_u32(b["tiles"])[:n])
    assert np.array_equal(counted(rect, gx, gy), to_np_u32(b["tc"]))
    return area


@pytest.mark.parametrize("W,H,n", [(W, H, n) for W, H, ns in GRIDS for n in ns])
def test_projection(W, H, n):
    import torch
    abi = lib_ready()
    cam = synth.look_at_camera(np.array([1.0, -8.0, 3.0]), np.zeros(3), W, H, d_max=30.0)
    g = synth.random_gaussians(n, n, cam, depth=(1.0, 30.0), scale=(0.01, 0.4))
    gx, gy = (W + 15) // 16, (H + 15) // 16
    b = _bufs(torch, n, gx, gy)
    abi.project_bin({k: cuda(v) for k, v in g.items()}, n, 0, cam, b["rec"], b["dk"], b["rect"],
                    b["tiles"], tile_count=b["tc"])
    area = check(b, n, gx, gy)
    if n >= 100_000:
        assert area.max() > 8 and (area == 0).any() and (area == 1).any()


@pytest.mark.parametrize("W,H,M", [(48, 32, 9), (48, 32, 10), (48, 32, 103), (1920, 1080, 13_055),
                                   (1920, 1080, 13_056), (1920, 1080, 33_001), (2048, 1520, 20_000)])
@pytest.mark.parametrize("fill", [1.0, 0.6])     # selected anchors of the capacity
def test_fused(W, H, M, fill):
    import torch
    abi = lib_ready()
    sc, mlp, cams = synth.CONFIGS["cube4k_128"]()
    cam = synth.look_at_camera(cams[0].campos, np.zeros(3), W, H, d_max=30.0)
    idx, w, _ = oracle.lod_select(sc.pos, sc.level, sc.dL, sc.NL, cams[0], False)
    m = max(int(M * fill), 1)
    counts = np.zeros(8, np.uint32)
    counts[0], counts[1] = m, 10 * m
    gx, gy = (W + 15) // 16, (H + 15) // 16
    b = _bufs(torch, M * 10, gx, gy)
    scr = torch.empty(abi.decode_project_scratch_bytes(), dtype=torch.uint8, device="cuda")
    abi.decode_project_bf16(
        cuda(sc.pos), cuda(sc.feat), cuda(sc.offs), cuda(sc.lv), sc.N,
        {k: cuda(a) for k, a in zip(NAMES, mlp.arrays())}, cam, cuda(np.resize(idx, M).astype(np.int32)),
        cuda(np.resize(w, M).astype(np.float32)), M, cuda(counts.view(np.int32)), b["rec"], b["dk"],
        b["rect"], b["tiles"], scr, out={k: b[k] for k in GAUSS}, tile_count=b["tc"])
    check(b, 10 * m, gx, gy)
