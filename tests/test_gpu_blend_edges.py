"""Blending at the edges of its walks: lists around the staged batches (256 records forward, 128
backward), the entries evaluated at a time (4 and 2) and the parked group (8), ragged images,
clamped opacities, and image gradients that are not finite.  Checked against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import cuda, lib_ready

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("needs a GPU")
    lib_ready()
    return t


def _setup(torch, W, H, G, opac, seed, sigma=(0.8, 10.0)):
    from paper_2403_17898_gb300 import abi
    r = synth.random_records(seed, G, W, H, sigma=sigma, opac=opac)
    gx, gy = (W + 15) // 16, (H + 15) // 16
    order = np.argsort(r["depth"], kind="stable")
    lst = np.tile(order, gx * gy).astype(np.int64)
    start = np.arange(gx * gy + 1, dtype=np.int64) * G
    rec = np.zeros((G, 12), np.float32)
    rec[:, 0], rec[:, 1] = r["u"], r["v"]
    rec[:, 2:4], rec[:, 4], rec[:, 5] = r["conic"][:, 0:2], r["conic"][:, 2], r["opac"]
    rec[:, 6:9] = r["colors"]
    rec[:, 11] = -np.log(255.0 * r["opac"].astype(np.float64))
    t = dict(rec=cuda(rec), lst=cuda(lst.astype(np.int32)),
             tr=cuda(np.stack([start[:-1], start[1:]], 1).astype(np.int32)),
             img=torch.zeros(3, H, W, device="cuda"), T=torch.zeros(H, W, device="cuda"),
             nl=torch.zeros(H, W, dtype=torch.int32, device="cuda"),
             drec=torch.zeros(G, 9, device="cuda"))
    bg = (0.05, 0.1, 0.2)
    abi.blend_fwd(t["rec"], t["lst"], t["tr"], W, H, bg, t["img"], t["T"], t["nl"])

    def bwd(dimg):
        t["drec"].zero_()
        abi.blend_bwd(t["rec"], t["lst"], t["tr"], W, H, bg, t["T"], t["nl"], cuda(dimg), t["drec"])
        torch.cuda.synchronize()
        return t["drec"].cpu().numpy()
    uv = np.stack([r["u"], r["v"]], 1)
    return r, order, lst, start, uv, bg, t, bwd


# opacities up to 1 reach the 0.99 clamp (zero derivative); up to 0.95 they do not
@pytest.mark.parametrize("opac", [(0.05, 0.95), (0.9, 1.0)])
@pytest.mark.parametrize("G", [1, 2, 3, 4, 5, 7, 8, 9, 127, 128, 129, 255, 257, 300])
@pytest.mark.parametrize("W,H", [(33, 17), (16, 16)])
def test_blend_list_and_group_edges(torch, W, H, G, opac):
    r, _, lst, start, uv, bg, t, bwd = _setup(torch, W, H, G, opac, 11 + G)
    fr = oracle.blend(W, H, start, lst, uv, r["conic"], r["opac"], r["colors"], bg)
    dimg = np.random.default_rng(5).normal(size=(3, H, W)).astype(np.float32)
    # FP32 and FP64 may decide differently at a threshold; such pixels take no part.  The clamp
    # is a threshold too: alpha near 0.99 at a pixel.
    near = fr["px_margin"] < 1e-3
    y, x = np.mgrid[0:H, 0:W]
    for g in range(G):
        dx, dy = uv[g, 0].astype(np.float64) - x, uv[g, 1].astype(np.float64) - y
        a, b, c = r["conic"][g].astype(np.float64)
        raw = r["opac"][g] * np.exp(-0.5 * (a * dx * dx + c * dy * dy) - b * dx * dy)
        near |= np.abs(raw - 0.99) < 1e-4
    ok = ~near
    assert np.abs(t["img"].cpu().numpy() - fr["img"])[:, ok].max(initial=0) <= 1e-4
    assert np.abs(t["T"].cpu().numpy() - fr["T"])[ok].max(initial=0) <= 1e-5
    assert np.array_equal(t["nl"].cpu().numpy()[ok], fr["last"][ok])
    dimg[:, near] = 0
    d = bwd(dimg)
    ref = oracle.blend_bwd(W, H, start, lst, uv, r["conic"], r["opac"], r["colors"], bg, dimg)
    for got, want in ((d[:, 0:2], ref["duv"]), (d[:, 2:5], ref["dconic"]),
                      (d[:, 5], ref["dopac"]), (d[:, 6:9], ref["dcolors"])):
        assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want) + 1e-6


def test_blend_bwd_nonfinite_gradient_stays_with_its_pixel(torch):
    """A pixel whose image gradient is not finite reaches the Gaussians blended there and no
    others, whoever shares its 8x8 block."""
    W, H, G = 40, 24, 150
    r, order, _, _, uv, _, t, bwd = _setup(torch, W, H, G, (0.05, 0.9), 3, sigma=(0.6, 4.0))
    dimg = np.random.default_rng(5).normal(size=(3, H, W)).astype(np.float32)
    clean = bwd(dimg)
    assert np.isfinite(clean).all()
    nl = t["nl"].cpu().numpy()
    for bad in (np.nan, np.inf):
        py, px = 13, 21
        hurt = dimg.copy()
        hurt[1, py, px] = bad
        d = bwd(hurt)
        dx, dy = uv[:, 0].astype(np.float64) - px, uv[:, 1].astype(np.float64) - py
        a, b, c = r["conic"].astype(np.float64).T
        alpha = r["opac"] * np.exp(-0.5 * (a * dx * dx + c * dy * dy) - b * dx * dy)
        pos = np.empty(G, int)
        pos[order] = np.arange(G)
        blended = (alpha >= 1 / 255) & (pos < nl[py, px])
        sure = np.abs(alpha * 255 - 1) > 1e-3
        assert blended.sum() > 3 and (~blended).sum() > 3
        assert not np.isfinite(d[blended & sure][:, [0, 5, 7]]).any()
        assert np.isfinite(d[blended & sure][:, [6, 8]]).all()
        rest = ~blended & sure
        assert np.allclose(d[rest], clean[rest], rtol=1e-4, atol=1e-6)
