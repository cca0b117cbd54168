"""The work that users of the renderer have it do, as measurable cases.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from a seed, ``run`` is
one pass through the package's public entry points (``render.Renderer`` / ``render.Trainer`` and
the calls of ``abi``), ``exact`` is the same result from plain torch in 64 bits, ``work`` the bytes
and operations that the path cannot do without.  Kinds:

  frame      one view, forward: selection, decoding, projection, tile lists, blending
  select     level-of-detail selection over all anchors
  gaussians  the selected anchors decoded and projected to screen records
  lists      per-tile front-to-back lists of the records
  blend      blending of the lists into an image, keeping what a backward needs
  blend_bwd  image gradient -> record gradients
  params_bwd record gradients -> anchor and decoder gradients (projection + decoder backward)
  loss       L1 + D-SSIM with its image gradient
  train      one optimisation step over a few views

Scenes are street grids and cubes of anchors on nested voxel grids; sizes are those of the
repository's benchmark scenes (4k anchors at 128x128, 500k at 1600x900, 2M and 8M at 1080p).
"""
import math

import numpy as np
import torch

from paper_2403_17898_gb300 import abi
from paper_2403_17898_gb300.proposal import ProposalNet
from paper_2403_17898_gb300.render import Renderer, Trainer

K = 10            # Gaussians per anchor
F = 32            # feature width
H = 32            # decoder hidden width
BG = (0.1, 0.2, 0.3)
TILE_CAP = 4096   # region entries per tile, as the renderer allocates


def listed():
    return [
        # the smallest call: an object-sized scene at thumbnail size, FP32; launches and latency
        dict(name="view_cube4k_128_fp32", kind="frame", scene="cube", anchors=4096, W=128, H=128,
             precision="fp32", gate=False, altitude=12.0),
        # the serving path: a frame of a large city at 1080p, BF16 decoders, learned gate
        dict(name="view_city2M_1080p_bf16_gated", kind="frame", scene="city", anchors=2_000_000,
             W=1920, H=1080, precision="bf16", gate=True, altitude=60.0),
        # level-of-detail selection over the largest anchor set (the training-scale scene)
        dict(name="select_8M", kind="select", anchors=8_000_000, levels=10, infer=True),
        # FP32 decoding + projection of a 1080p view's anchors (reference-precision path)
        dict(name="gaussians_fp32_100k", kind="gaussians", anchors=100_000, total=2_000_000,
             W=1920, H=1080, precision="fp32"),
        # BF16 fused decoding + projection, with the Gaussians kept for a training backward
        dict(name="gaussians_bf16_100k", kind="gaussians", anchors=100_000, total=2_000_000,
             W=1920, H=1080, precision="bf16"),
        # per-tile lists of a 1080p view in regions (the BF16 renderer's form)
        dict(name="lists_regions_1080p", kind="lists", form="regions", gaussians=800_000, W=1920,
             H=1080),
        # blending of a 1080p training view
        dict(name="blend_1080p", kind="blend", gaussians=800_000, W=1920, H=1080),
        # its backward
        dict(name="blend_bwd_1080p", kind="blend_bwd", gaussians=800_000, W=1920, H=1080),
        # projection + decoder backward of a BF16 training view of the large scenes
        dict(name="params_bwd_bf16_100k", kind="params_bwd", anchors=100_000, total=2_000_000,
             W=1920, H=1080, precision="bf16"),
        # the same in FP32 at a ragged street-scene size
        dict(name="params_bwd_fp32_31k", kind="params_bwd", anchors=31_337, total=500_000,
             W=1600, H=900, precision="fp32"),
        # photometric loss of a 1080p view against a target whose moments are kept
        dict(name="loss_1080p", kind="loss", W=1920, H=1080, cached=True),
        # a whole training step: four 1080p views of the city, L1 + D-SSIM, BF16, Adam
        dict(name="train_city2M_4x1080p_bf16", kind="train", scene="city", anchors=2_000_000,
             W=1920, H=1080, precision="bf16", views=4, altitude=60.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _image(rng):
    """An image size of the range, mostly not a multiple of the 16-pixel tile."""
    h = _log(rng, 128, 1080)
    w = min(1920, max(128, int(h * rng.choice([1.0, 4 / 3, 16 / 9]))))
    return w - rng.randrange(0, 12), h - rng.randrange(0, 12)


def draw(rng):
    kind = rng.choice(["frame", "frame", "select", "gaussians", "lists", "blend", "blend_bwd",
                       "params_bwd", "loss", "train"])
    W, Hh = _image(rng)
    share = W * Hh / (1920 * 1080)
    precision = rng.choice(["fp32", "bf16"])
    if kind == "frame":
        n = _log(rng, 4096, 2_000_000)
        return dict(kind=kind, scene="cube" if n < 20_000 else "city", anchors=n, W=W, H=Hh,
                    precision=precision, gate=rng.random() < 0.5,
                    altitude=12.0 if n < 20_000 else round(rng.uniform(40.0, 400.0), 1))
    if kind == "select":
        return dict(kind=kind, anchors=_log(rng, 3000, 8_000_000), levels=rng.randrange(3, 11),
                    infer=rng.random() < 0.5)
    if kind in ("gaussians", "params_bwd"):
        m = _log(rng, 1000, 100_000 if kind == "gaussians" or precision == "bf16" else 60_000)
        return dict(kind=kind, anchors=m, total=m * rng.randrange(3, 20), W=W, H=Hh,
                    precision=precision)
    if kind in ("lists", "blend", "blend_bwd"):
        c = dict(kind=kind, gaussians=10 * max(100, int(80_000 * share * rng.uniform(0.3, 1.0))),
                 W=W, H=Hh)
        if kind == "lists":
            c["form"] = rng.choice(["regions", "packed"])
        return c
    if kind == "loss":
        return dict(kind=kind, W=W, H=Hh, cached=rng.random() < 0.5)
    return dict(kind=kind, scene="city", anchors=_log(rng, 100_000, 1_000_000), W=W, H=Hh,
                precision=precision, views=rng.randrange(1, 5),
                altitude=round(rng.uniform(40.0, 400.0), 1))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

class _Camera:
    pass


class _Scene:
    pass


class _Weights:
    def __init__(self, arrays):
        self._a = arrays

    def arrays(self):
        return self._a


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _u(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo


def _n(g, *shape, sd=1.0, mean=0.0):
    return torch.randn(*shape, generator=g, device="cuda") * sd + mean


def _look_at(eye, target, W, Hh, d_max, fovx=60.0):
    eye, target = np.asarray(eye, np.float64), np.asarray(target, np.float64)
    f = target - eye
    f /= np.linalg.norm(f)
    r = np.cross(f, [0.0, 0.0, 1.0])
    r /= np.linalg.norm(r)
    c = _Camera()
    c.R = np.stack([r, np.cross(f, r), f]).astype(np.float32)
    c.campos = eye.astype(np.float32)
    c.fx = c.fy = float(np.float32((W / 2) / math.tan(math.radians(fovx) / 2)))
    c.cx, c.cy, c.W, c.H = (W - 1) / 2, (Hh - 1) / 2, W, Hh
    c.znear, c.d_max, c.s = 0.2, float(np.float32(d_max)), 1.0
    return c


def _view(altitude, W, Hh, d_max, rnd):
    """A zoom-out pose: 45 degrees down on the scene's centre, azimuth 30 +- 40 degrees."""
    az = math.radians(30.0 + rnd.uniform(-40.0, 40.0))
    return _look_at([-altitude * math.cos(az), -altitude * math.sin(az), altitude], [0, 0, 0], W,
                    Hh, d_max)


def _unique_cells(points, cell, need, g):
    """`need` distinct voxel centres among those of the points, in random order (or None)."""
    v = torch.round(points / cell)
    q = v.to(torch.int64) + (1 << 20)
    key = torch.unique((q[:, 0] << 42) | (q[:, 1] << 21) | q[:, 2])
    if key.numel() < need:
        return None
    key = key[torch.randperm(key.numel(), generator=g, device="cuda")[:need]]
    m = (1 << 21) - 1
    q = torch.stack([key >> 42, (key >> 21) & m, key & m], 1) - (1 << 20)
    return q.to(torch.float32) * cell


def _city_points(n, half, extent, boxes, pitch, g):
    """Surface points of a street grid inside |x|, |y| <= half: ground, roofs and walls."""
    nb = boxes.shape[0]
    xy = _u(g, n, 2, lo=-half, hi=half)
    b = ((xy + extent / 2) / pitch).floor().long().clamp(0, nb - 1)
    corner = b * pitch - extent / 2
    box = boxes[b[:, 0], b[:, 1]]                       # x0, y0, wx, wy, h within the block
    loc = xy - corner
    inside = ((loc >= box[:, :2]) & (loc <= box[:, :2] + box[:, 2:4])).all(1)
    z = torch.where(inside, box[:, 4], torch.zeros_like(box[:, 4]))
    wall = _u(g, n) < 0.45
    face = (_u(g, n) * 4).long()
    t = _u(g, n)
    wx = torch.where(face < 2, box[:, 0] + t * box[:, 2],
                     box[:, 0] + (face == 2).float() * box[:, 2])
    wy = torch.where(face >= 2, box[:, 1] + t * box[:, 3],
                     box[:, 1] + (face == 0).float() * box[:, 3])
    p = torch.stack([xy[:, 0], xy[:, 1], z], 1)
    pw = torch.stack([corner[:, 0] + wx, corner[:, 1] + wy, _u(g, n) * box[:, 4]], 1)
    p = torch.where(wall[:, None], pw, p)
    return p[(p[:, :2].abs() <= half).all(1)]


def _anchors(kind, n, g):
    """(pos, level, cell per level, NL, d_max) of an anchor set: nested voxel grids on a city's
    surfaces, finer near the centre, or filling a 10 m cube."""
    if kind == "cube":
        NL, d_max = 3, 30.0
        cells = [10.0 / 2 ** (L + 3) for L in range(NL)]
        weights = [4.0 ** L for L in range(NL)]
    elif n < 700_000:
        NL, extent, c0 = 6, 600.0, 2.0
        d_max = 1.2 * extent
    elif n < 4_000_000:
        NL, extent, c0 = 8, 2000.0, 4.0
        d_max = 1.75 * extent
    else:
        NL, extent, c0 = 10, 4000.0, 6.0
        d_max = 1.75 * extent
    if kind != "cube":
        cells = [c0 / 2 ** L for L in range(NL)]
        weights = [4.0 ** (0.45 * L) for L in range(NL)]
        pitch = 120.0
        nb = int(math.ceil(extent / pitch))
        wxy = _u(g, nb, nb, 2, lo=10.0, hi=60.0)
        boxes = torch.cat([10.0 + _u(g, nb, nb, 2) * (100.0 - wxy), wxy,
                           _u(g, nb, nb, 1, lo=10.0, hi=60.0)], 2)
        # a plaza at the centre, where the cameras look
        mid = (torch.arange(nb, device="cuda") + 0.5) * pitch - extent / 2
        free = (mid[:, None].square() + mid[None, :].square()).sqrt() < 100.0
        boxes[..., 4] = torch.where(free, torch.zeros_like(boxes[..., 4]), boxes[..., 4])
    counts = [int(n * w / sum(weights)) for w in weights]
    counts[-1] += n - sum(counts)
    pos, level = [], []
    for L in range(NL):
        m, got = int(counts[L] * 1.6) + 4096, None
        while got is None:
            if kind == "cube":
                p = (_u(g, m, 3, lo=-5.0, hi=5.0) / cells[L]).floor() * cells[L]
            else:
                p = _city_points(m, extent / 2 * 2.0 ** (-0.55 * L), extent, boxes, pitch, g)
            got = _unique_cells(p, cells[L], counts[L], g)
            m *= 2
        pos.append(got)
        level.append(torch.full((counts[L],), L, dtype=torch.uint8, device="cuda"))
    perm = torch.randperm(n, generator=g, device="cuda")
    return torch.cat(pos)[perm], torch.cat(level)[perm], torch.tensor(cells, device="cuda"), NL, d_max


def _decoder(g, d_max):
    """Decoder weights at the scale of a trained network's start (uniform, fan-in), biases that
    give opaque enough, coloured, anisotropic Gaussians."""
    bi, bh = 1 / math.sqrt(F + 4), 1 / math.sqrt(H)
    w1 = _u(g, 3, H, F + 4, lo=-bi, hi=bi)
    w1[:, :, F + 3] /= d_max
    cov = _u(g, 7 * K, lo=-bh, hi=bh).reshape(K, 7)
    cov[:, :3] += _u(g, K, 3, lo=-1, hi=1)
    cov[:, 3:] += _n(g, K, 4)
    return dict(w1=w1, b1=_u(g, 3, H, lo=-bi, hi=bi), w2_op=_u(g, K, H, lo=-bh, hi=bh),
                b2_op=_u(g, K, lo=-bh, hi=bh) + 0.5, w2_col=_u(g, 3 * K, H, lo=-bh, hi=bh),
                b2_col=_u(g, 3 * K, lo=-1.5, hi=1.5), w2_cov=_u(g, 7 * K, H, lo=-bh, hi=bh),
                b2_cov=cov.reshape(-1).contiguous())


def _scene(case, g):
    pos, level, cells, NL, d_max = _anchors(case["scene"], case["anchors"], g)
    n = pos.shape[0]
    s = _Scene()
    lv = cells[level.long()][:, None].expand(n, 3)
    for name, t in (("pos", pos), ("level", level), ("dL", (_u(g, n, hi=0.3) * 100).round() / 100),
                    ("feat", _n(g, n, F, sd=0.1)), ("offs", _n(g, n, K, 3, sd=0.5)), ("lv", lv)):
        setattr(s, name, t.contiguous().cpu().numpy())
    s.NL = NL
    w = _decoder(g, d_max)
    return s, _Weights([t.cpu().numpy() for t in w.values()]), d_max


def _proposal(g, rd, cam):
    """A gate network whose output bias keeps about 72 % of the anchors in front of the camera."""
    bi, bh = 1 / math.sqrt(F + 5), 1 / 8
    a = [_u(g, 64, F + 5, lo=-bi, hi=bi), _u(g, 64, lo=-bi, hi=bi), _u(g, 64, 64, lo=-bh, hi=bh),
         _u(g, 64, lo=-bh, hi=bh), _u(g, 1, 64, lo=-bh, hi=bh), torch.zeros(1, device="cuda")]
    R, c = torch.tensor(cam.R, device="cuda"), torch.tensor(cam.campos, device="cuda")
    q = (rd.pos - c) @ R.T
    seen = torch.nonzero((q[:, 2] > 0.2) & (q[:, :2].abs() < 0.6 * q[:, 2:3]).all(1))[:20_000, 0]
    d = q[seen].norm(dim=1, keepdim=True)
    x = torch.cat([rd.feat[seen], rd.level[seen].float()[:, None] / (rd.NL - 1), q[seen] / d,
                   torch.log(d / cam.d_max)], 1)
    h = torch.relu(torch.relu(x @ a[0].T + a[1]) @ a[2].T + a[3])
    logit = (h @ a[4].T)[:, 0]
    p_star = 0.6
    if logit.numel():
        a[5] += math.log(p_star / (1 - p_star)) - torch.quantile(logit, 0.28)
    return ProposalNet(_Weights([t.cpu().numpy() for t in a])).w, p_star


def _capacities(case):
    n, px = case["anchors"], case["W"] * case["H"]
    return dict(sel_cap=max(4096, min(n, 400_000)), pair_cap=max(1 << 18, 3 * px))


def _fit(rd, cams, infer, gate=None):
    """Renders each view once, which sizes the renderer's buffers for them."""
    for _ in range(2):
        for cam in cams:
            rd.render(cam, infer=infer, bg=BG, gate=gate)


def _smooth_image(g, W, Hh):
    """An image with structure at several scales, in [0, 1]."""
    t = torch.zeros(1, 3, Hh, W, device="cuda")
    for cells, amp in ((4, 0.5), (24, 0.3), (120, 0.2)):
        a = _u(g, 1, 3, max(2, cells * Hh // 1080 + 2), max(2, cells * W // 1080 + 2))
        t += amp * torch.nn.functional.interpolate(a, (Hh, W), mode="bilinear")
    return (t[0] * 0.95 + 0.05 * _u(g, 3, Hh, W)).contiguous()


def _selected(case, g):
    """A view's selection: camera, anchors seen by it with cells as the level rule gives them at
    their distance, their index list, weights and counters."""
    m, n, W, Hh = case["anchors"], case["total"], case["W"], case["H"]
    d_max = 3500.0
    cam = _look_at([-80.0, -50.0, 90.0], [0.0, 0.0, 0.0], W, Hh, d_max)
    z = torch.exp(_u(g, m, lo=math.log(15.0), hi=math.log(1500.0)))
    tan = torch.tensor([W / (2 * cam.fx), Hh / (2 * cam.fy)], device="cuda")
    xy = _u(g, m, 2, lo=-1.3, hi=1.3) * tan * z[:, None]
    seen = torch.cat([xy, z[:, None]], 1) @ torch.tensor(cam.R, device="cuda") + torch.tensor(
        cam.campos, device="cuda")
    coarser = (torch.log(_u(g, m, lo=1e-4)) / math.log(0.28)).floor().clamp(0, 6)
    cell = 4.0 / d_max * z * _u(g, m, lo=1.0, hi=2.0) * 2.0 ** coarser
    idx = torch.randperm(n, generator=g, device="cuda")[:m].sort().values
    a = dict(pos=_n(g, n, 3, sd=300.0), feat=_n(g, n, F, sd=0.1), offs=_n(g, n, K, 3, sd=0.5),
             lv=torch.ones(n, 3, device="cuda"))
    a["pos"][idx] = seen
    a["lv"][idx] = cell[:, None].expand(m, 3)
    w = torch.where(_u(g, m) < 0.15, _u(g, m, lo=0.01), torch.ones(m, device="cuda"))
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    counts[0], counts[1] = m, m * K
    return cam, a, idx.to(torch.int32), w, counts, _decoder(g, d_max)


def _screen(case, g):
    """Screen records of a view (u, v, conic, opacity, colour, depth, radius, skip bound), tile
    rectangles, tile counts and depth keys; the ten Gaussians of an anchor lie together.  Some
    are culled (transparent or outside the image), as in any view."""
    G, W, Hh = case["gaussians"], case["W"], case["H"]
    m = G // K
    size = torch.tensor([W, Hh], device="cuda", dtype=torch.float32)
    centre = torch.where((_u(g, m) < 0.75)[:, None], _u(g, m, 2, lo=-0.15, hi=1.15) * size,
                         (0.5 + 0.17 * _n(g, m, 2)) * size)
    base = _u(g, m, lo=1.2, hi=2.4) * 2.0 ** (torch.log(_u(g, m, lo=1e-4)) / math.log(0.2)).floor()
    rep = lambda t: t.repeat_interleave(K, 0)  # noqa: E731
    base = rep(base)
    uv = rep(centre) + _n(g, G, 2) * base[:, None]
    s1 = base * _u(g, G, lo=0.6, hi=1.4)
    s2 = s1 * _u(g, G, lo=0.25, hi=1.0)
    th = _u(g, G, hi=math.pi)
    c, s = torch.cos(th), torch.sin(th)
    a = c * c * s1 * s1 + s * s * s2 * s2 + 0.3
    b = c * s * (s1 * s1 - s2 * s2)
    d = s * s * s1 * s1 + c * c * s2 * s2 + 0.3
    det = a * d - b * b
    mid = 0.5 * (a + d)
    radius = 3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1)))
    opac = torch.tanh(_n(g, G, sd=0.35, mean=0.5))
    depth = rep(torch.exp(_u(g, m, lo=math.log(5.0), hi=math.log(800.0)))) * _u(g, G, lo=0.99,
                                                                              hi=1.01)
    lo = torch.floor(torch.ceil(uv - radius[:, None]) / 16).clamp_min(0)
    hi = torch.minimum(torch.floor(torch.floor(uv + radius[:, None]) / 16) + 1,
                       torch.ceil(size / 16))
    seen = (opac > 0.002) & (lo < hi).all(1)
    lo, hi = (torch.where(seen[:, None], t, torch.zeros_like(t)).to(torch.int32) for t in (lo, hi))
    rec = torch.stack([uv[:, 0], uv[:, 1], d / det, -b / det, a / det, opac, _u(g, G), _u(g, G),
                       _u(g, G), depth, radius, -torch.log(255 * opac.clamp_min(1e-6))], 1)
    rec = torch.where(seen[:, None], rec, torch.zeros_like(rec)).contiguous()
    tiles = (hi - lo).prod(1).to(torch.int32)
    rect = torch.stack([lo[:, 0] | (lo[:, 1] << 16), hi[:, 0] | (hi[:, 1] << 16)], 1).contiguous()
    key = torch.where(seen, depth.view(torch.int32), torch.full_like(tiles, -1))
    return rec, rect, tiles, key, lo, hi


def _lists(case, screen):
    """Packed per-tile lists, nearest first, and each tile's range, in plain torch."""
    _, _, tiles, key, lo, hi = screen
    gx, gy = (case["W"] + 15) // 16, (case["H"] + 15) // 16
    per = tiles.long()
    g = torch.repeat_interleave(torch.arange(per.numel(), device="cuda"), per)
    i = torch.arange(g.numel(), device="cuda") - (per.cumsum(0) - per)[g]
    w = (hi[:, 0] - lo[:, 0]).long()[g]
    t = (lo[g, 1].long() + i // w) * gx + lo[g, 0].long() + i % w
    order = torch.sort((t << 32) | (key[g].long() & 0xFFFFFFFF), stable=True).indices
    count = torch.bincount(t, minlength=gx * gy)
    end = count.cumsum(0)
    return g[order].to(torch.int32), torch.stack([end - count, end], 1).to(torch.int32).contiguous()


def prepare(case, seed):
    g = _gen(seed)
    rnd = np.random.default_rng(seed)
    kind, W, Hh = case["kind"], case.get("W"), case.get("H")
    st = dict(case=case)
    empty = lambda *s, dtype=torch.float32: torch.zeros(*s, dtype=dtype, device="cuda")  # noqa: E731
    if kind == "frame":
        scene, mlp, d_max = _scene(case, g)
        cam = _view(case["altitude"], W, Hh, d_max, rnd)
        rd = Renderer(scene, mlp, W, Hh, precision=case["precision"], **_capacities(case))
        gate = _proposal(g, rd, cam) if case["gate"] else None
        _fit(rd, [cam], True, gate)
        st.update(rd=rd, cam=cam, gate=gate)
    elif kind == "train":
        scene, mlp, d_max = _scene(case, g)
        cams = [_view(case["altitude"] * 2.0 ** (0.5 * i), W, Hh, d_max, rnd)
                for i in range(case["views"])]
        # late in a run: a small step size and second moments that have settled
        tr = Trainer(scene, mlp, W, Hh, lr=1e-5, ssim_lambda=0.2, precision=case["precision"],
                     **_capacities(case))
        _fit(tr, cams, False)
        for t in tr.adam_v.values():
            t.copy_(_u(g, *t.shape, lo=1e-7, hi=4e-7).square())
        tr.step_count = 1000
        st.update(tr=tr, cams=cams, targets=[_smooth_image(g, W, Hh) for _ in cams])
    elif kind == "select":
        pos, level, _, _, d_max = _anchors("city" if case["anchors"] >= 20_000 else "cube",
                                           case["anchors"], g)
        n = pos.shape[0]
        st.update(pos=pos, level=level.clamp_max(case["levels"] - 1), n=n,
                  dL=((_u(g, n, hi=0.3) * 100).round() / 100), idx=empty(n, dtype=torch.int32),
                  w=empty(n), counts=empty(8, dtype=torch.int32),
                  scratch=empty(abi.lod_select_scratch_bytes(n), dtype=torch.uint8),
                  cam=abi.camera(_view(80.0 if n >= 20_000 else 12.0, 1920, 1080, d_max, rnd)))
    elif kind == "gaussians":
        cam, a, idx, w, counts, mlp = _selected(case, g)
        G, gx, gy = case["anchors"] * K, (W + 15) // 16, (Hh + 15) // 16
        out = dict(means=empty(G, 3), scales=empty(G, 3), quats=empty(G, 4), opac=empty(G),
                   colors=empty(G, 3))
        st.update(cam=abi.camera(cam), cam_py=cam, a=a, idx=idx, w=w, counts=counts, mlp=mlp,
                  mlp_s=abi.mlp_struct(mlp), out=out, out_s=abi.gaussians_struct(out),
                  rec=empty(G, 12), key=empty(G, dtype=torch.int32),
                  rect=empty(G, 2, dtype=torch.int32), tiles=empty(G, dtype=torch.int32),
                  tile_count=empty(gx * gy, dtype=torch.int32),
                  scratch=empty(abi.decode_project_scratch_bytes(), dtype=torch.uint8))
    elif kind == "lists":
        screen = _screen(case, g)
        G, nt = case["gaussians"], ((W + 15) // 16) * ((Hh + 15) // 16)
        st.update(rect=screen[1], tiles=screen[2], key=screen[3], nt=nt, G=G,
                  counts=empty(8, dtype=torch.int32), ranges=empty(nt, 2, dtype=torch.int32))
        if case["form"] == "regions":
            pk, pg = (empty(nt * TILE_CAP, dtype=torch.int32) for _ in range(2))
            st.update(pair_key=pk, pairs=pg, bins=abi.tile_bins(pk, pg, TILE_CAP),
                      scratch=empty(abi.sort_bins_scratch_bytes(nt), dtype=torch.uint8))
        else:
            P = int(screen[2].sum())
            st.update(P=P, pairs=empty(P, dtype=torch.int32),
                      scratch=empty(abi.sort_scratch_bytes(G, P, nt), dtype=torch.uint8))
    elif kind in ("blend", "blend_bwd"):
        screen = _screen(case, g)
        pairs, ranges = _lists(case, screen)
        st.update(rec=screen[0], pairs=pairs, ranges=ranges, img=empty(3, Hh, W), T=empty(Hh, W),
                  n_last=empty(Hh, W, dtype=torch.int32))
        if kind == "blend_bwd":
            _blend(st)
            n = 3 * W * Hh
            st.update(drec=empty(case["gaussians"], 9),
                      dimg=(torch.sign(_n(g, 3, Hh, W)) * 0.8 + _n(g, 3, Hh, W, sd=0.2)) / n)
    elif kind == "params_bwd":
        cam, a, idx, w, counts, mlp = _selected(case, g)
        m = case["anchors"]
        gs = _decode64(cam, a, idx, w, mlp, torch.float32)
        rec, rect = _project64(cam, gs)
        drec = _n(g, m * K, 9) * torch.tensor([3e-8, 3e-8, 3e-6, 3e-6, 3e-6, 1e-6, 1e-6, 1e-6,
                                               1e-6], device="cuda")
        drec = torch.where((rect[:, 0] != rect[:, 1])[:, None], drec, torch.zeros_like(drec))
        gs = {k: v.contiguous() for k, v in gs.items()}
        grads = dict(feat=torch.zeros_like(a["feat"]), offs=torch.zeros_like(a["offs"]),
                     lv=torch.zeros_like(a["lv"]))
        dmlp = {k: torch.zeros_like(v) for k, v in mlp.items()}
        st.update(cam=abi.camera(cam), cam_py=cam, a=a, idx=idx, w=w, counts=counts, mlp=mlp,
                  mlp_s=abi.mlp_struct(mlp), g=gs, g_s=abi.gaussians_struct(gs),
                  rect=rect.contiguous(), drec=drec.contiguous(), grads=grads, dmlp=dmlp,
                  dmlp_s=abi.mlp_struct(dmlp), dmeans=empty(m * K, 3), dscales=empty(m * K, 3),
                  dquats=empty(m * K, 4),
                  scratch=empty(abi.decode_bwd_scratch_bytes(m), dtype=torch.uint8))
    elif kind == "loss":
        img, target = _smooth_image(g, W, Hh), _smooth_image(g, W, Hh)
        img = (0.7 * target + 0.3 * img).contiguous()      # a render on its way to its target
        st.update(img=img, target=target, dimg=empty(3, Hh, W), loss=empty(1), stats=None,
                  scratch=empty(abi.loss_l1_ssim_scratch_bytes(3, Hh, W), dtype=torch.uint8))
        if case["cached"]:
            st["stats"] = empty(2, 3, Hh, W)
            abi.ssim_target_stats(target, st["stats"])
    return st


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------

def _blend(st):
    c = st["case"]
    abi.blend_fwd(st["rec"], st["pairs"], st["ranges"], c["W"], c["H"], BG, st["img"], st["T"],
                  st["n_last"])
    return st["img"], st["T"], st["n_last"]


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "frame":
        rd = st["rd"]
        rd.render(st["cam"], infer=True, bg=BG, check=False, gate=st["gate"])
        return rd.img, rd.T
    if kind == "train":
        tr = st["tr"]
        tr.train_step(st["cams"], st["targets"], bg=BG)
        out = {"loss": tr.loss, "stamp": tr.stamp}
        for n, t in list(tr._anchor_params().items()) + [("mlp." + k, v) for k, v in tr.mlp.items()]:
            out[n], out["m." + n], out["v." + n] = t, tr.adam_m[n], tr.adam_v[n]
        return out
    if kind == "select":
        st["counts"].zero_()
        abi.lod_select(st["pos"], st["level"], st["dL"], st["n"], c["levels"], K, st["cam"],
                       c["infer"], st["idx"], st["w"], st["n"], st["counts"], st["scratch"])
        return st["idx"], st["w"], st["counts"]
    if kind == "gaussians":
        a, m = st["a"], c["anchors"]
        if c["precision"] == "fp32":
            abi.decode(a["pos"], a["feat"], a["offs"], a["lv"], c["total"], st["mlp_s"], st["cam"],
                       st["idx"], st["w"], m, st["counts"], st["out_s"])
            abi.project_bin(st["out_s"], m * K, 1, st["cam"], st["rec"], st["key"], st["rect"],
                            st["tiles"], st["counts"], tile_count=st["tile_count"])
        else:
            abi.decode_project_bf16(a["pos"], a["feat"], a["offs"], a["lv"], c["total"],
                                    st["mlp_s"], st["cam"], st["idx"], st["w"], m, st["counts"],
                                    st["rec"], st["key"], st["rect"], st["tiles"], st["scratch"],
                                    out=st["out_s"], tile_count=st["tile_count"])
        return dict(st["out"], rec=st["rec"], key=st["key"], rect=st["rect"], tiles=st["tiles"],
                    tile_count=st["tile_count"])
    if kind == "lists":
        st["counts"].zero_()
        gx, gy = (c["W"] + 15) // 16, (c["H"] + 15) // 16
        if c["form"] == "regions":
            abi.sort_bins(st["key"], st["rect"], st["tiles"], st["G"], st["G"], gx, gy, st["bins"],
                          st["ranges"], st["counts"], st["scratch"])
        else:
            abi.sort(st["key"], st["rect"], st["tiles"], st["G"], st["G"], gx, gy, st["pairs"],
                     st["ranges"], st["P"], st["counts"], st["scratch"])
        return st["pairs"], st["ranges"], st["counts"]
    if kind == "blend":
        return _blend(st)
    if kind == "blend_bwd":
        st["drec"].zero_()
        abi.blend_bwd(st["rec"], st["pairs"], st["ranges"], c["W"], c["H"], BG, st["T"],
                      st["n_last"], st["dimg"], st["drec"])
        return st["drec"]
    if kind == "params_bwd":
        a, m, gr = st["a"], c["anchors"], st["grads"]
        abi.project_bwd(st["g_s"], m * K, 1, st["cam"], st["rect"], st["drec"], st["dmeans"],
                        st["dscales"], st["dquats"], st["counts"])
        abi.decode_bwd(a["pos"], a["feat"], a["offs"], a["lv"], c["total"], st["mlp_s"], st["cam"],
                       st["idx"], st["w"], m, st["counts"], st["dmeans"], st["dscales"],
                       st["dquats"], st["drec"], gr["feat"], gr["offs"], gr["lv"], st["dmlp_s"],
                       st["scratch"], bf16=c["precision"] == "bf16")
        return dict(gr, **st["dmlp"])
    st["loss"].zero_()
    abi.loss_l1_ssim(st["img"], st["target"], 0.2, st["dimg"], st["loss"], st["scratch"],
                     target_stats=st["stats"])
    return st["dimg"], st["loss"]


# ---------------------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------------------

def _decode64(cam, a, idx, w, mlp, dtype=torch.float64, leaves=None):
    """Neural Gaussians of the selected anchors (means relative to the camera)."""
    j = idx.long()
    p = leaves or {**{n: a[n][j].to(dtype) for n in ("feat", "offs", "lv")},
                   **{n: t.to(dtype) for n, t in mlp.items()}}
    dv = a["pos"][j].to(dtype) - torch.tensor(cam.campos, device="cuda").to(dtype)
    d = dv.norm(dim=1, keepdim=True)
    z = torch.cat([p["feat"], dv / d, d], 1)
    hid = [torch.relu(z @ p["w1"][i].T + p["b1"][i]) for i in range(3)]
    m = j.numel()
    op = torch.tanh(hid[0] @ p["w2_op"].T + p["b2_op"]) * w.to(dtype)[:, None]
    col = torch.sigmoid(hid[1] @ p["w2_col"].T + p["b2_col"])
    cov = (hid[2] @ p["w2_cov"].T + p["b2_cov"]).reshape(m, K, 7)
    lv = p["lv"][:, None, :]
    q = cov[..., 3:]
    return dict(means=(dv[:, None, :] + p["offs"] * lv).reshape(m * K, 3),
                scales=(lv * torch.sigmoid(cov[..., :3])).reshape(m * K, 3),
                quats=(q / q.norm(dim=2, keepdim=True)).reshape(m * K, 4),
                opac=op.reshape(m * K), colors=col.reshape(m * K, 3))


def _project64(cam, gs):
    """Screen records of Gaussians (zeros where culled) and their packed tile rectangles."""
    dt = gs["means"].dtype
    R = torch.tensor(cam.R, device="cuda").to(dt)
    p = gs["means"] @ R.T
    front = (p[:, 2] > cam.znear) & (gs["opac"] > 0)
    p = torch.where(front[:, None], p, torch.ones_like(p))
    z = p[:, 2]
    w, x, y, k = gs["quats"].unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                      2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                      2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)],
                     1).reshape(-1, 3, 3)
    M = Rq * gs["scales"][:, None, :]
    limx, limy = 1.3 * cam.W / (2 * cam.fx), 1.3 * cam.H / (2 * cam.fy)
    tx, ty = (p[:, 0] / z).clamp(-limx, limx) * z, (p[:, 1] / z).clamp(-limy, limy) * z
    o = torch.zeros_like(z)
    J = torch.stack([cam.fx / z, o, -cam.fx * tx / z ** 2, o, cam.fy / z, -cam.fy * ty / z ** 2],
                    1).reshape(-1, 2, 3)
    TM = (J @ R) @ M
    C = TM @ TM.transpose(1, 2)
    ca, cb, cc = C[:, 0, 0] + 0.3, C[:, 0, 1], C[:, 1, 1] + 0.3
    det = ca * cc - cb * cb
    mid = 0.5 * (ca + cc)
    r = 3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1)))
    u, v = cam.fx * p[:, 0] / z + cam.cx, cam.fy * p[:, 1] / z + cam.cy
    gx, gy = (cam.W + 15) // 16, (cam.H + 15) // 16
    with torch.no_grad():
        lo = [torch.floor(torch.ceil(t - r) / 16).clamp_min(0) for t in (u, v)]
        hi = [torch.floor(torch.floor(t + r) / 16 + 1).clamp_max(n) for t, n in ((u, gx), (v, gy))]
        seen = front & (det > 0) & (lo[0] < hi[0]) & (lo[1] < hi[1])
        rect = torch.stack([torch.where(seen, a.clamp(0, 65535) + b.clamp(0, 65535) * 65536, o)
                            for a, b in ((lo[0], lo[1]), (hi[0], hi[1]))], 1)
        rect = rect.to(torch.int64).to(torch.int32)
    op = torch.where(seen, gs["opac"], torch.ones_like(o))
    col = gs["colors"]
    rec = torch.stack([u, v, cc / det, -cb / det, ca / det, op, col[:, 0], col[:, 1], col[:, 2], z,
                       r, -torch.log(255 * op)], 1)
    return torch.where(seen[:, None], rec, torch.zeros_like(rec)), rect


def _blend64(st, dimg=None):
    """Image and transmittance of the lists, one list position of every tile at a time; with an
    image gradient, the record gradients."""
    c = st["case"]
    W, Hh = c["W"], c["H"]
    gx = (W + 15) // 16
    rec = st["rec"].double()
    rng = st["ranges"].long()
    n = rng[:, 1] - rng[:, 0]
    order = torch.argsort(n, descending=True)
    start = rng[order, 0]
    lens = n[order]
    q = torch.arange(256, device="cuda")
    px = ((order % gx) * 16)[:, None] + q % 16
    py = ((order // gx) * 16)[:, None] + q // 16
    out_of = (px >= W) | (py >= Hh)
    px, py = px.double(), py.double()
    nt = len(order)

    def step(i, A, T, done):
        """alpha of list entry i for A tiles' pixels, and which of them it is blended into."""
        r = rec[st["pairs"][start[:A] + i].long()]
        dx, dy = r[:, 0:1] - px[:A], r[:, 1:2] - py[:A]
        power = -0.5 * (r[:, 2:3] * dx * dx + r[:, 4:5] * dy * dy) - r[:, 3:4] * dx * dy
        G = torch.exp(power)
        raw = r[:, 5:6] * G
        al = raw.clamp_max(0.99)
        ok = ~done[:A] & (power <= 0) & (power >= r[:, 11:12])
        sat = ok & (T[:A] * (1 - al) < 1e-4)
        done[:A] |= sat
        return r, dx, dy, G, raw, al, ok & ~sat

    def fresh():
        return torch.ones(nt, 256, dtype=torch.float64, device="cuda"), out_of.clone()

    T, done = fresh()
    C = torch.zeros(3, nt, 256, dtype=torch.float64, device="cuda")
    for i, A in enumerate(_past(lens)):
        r, _, _, _, _, al, ok = step(i, A, T, done)
        w = torch.where(ok, al * T[:A], torch.zeros_like(al))
        for ch in range(3):
            C[ch, :A] += w * r[:, 6 + ch:7 + ch]
        T[:A] -= w
    for ch in range(3):
        C[ch] += T * BG[ch]
    at = (py * W + px).long()[~out_of]
    if dimg is None:
        img = torch.empty(3, Hh * W, dtype=torch.float64, device="cuda")
        Tf = torch.empty(Hh * W, dtype=torch.float64, device="cuda")
        img[:, at] = C[:, ~out_of]
        Tf[at] = T[~out_of]
        return img.reshape(3, Hh, W), Tf.reshape(Hh, W)
    d = torch.zeros(3, nt, 256, dtype=torch.float64, device="cuda")
    d[:, ~out_of] = dimg.double().reshape(3, -1)[:, at]
    total = (C * d).sum(0)                                   # what lies behind, times T
    drec = torch.zeros(rec.shape[0], 9, dtype=torch.float64, device="cuda")
    T, done = fresh()
    acc = torch.zeros_like(T)
    for i, A in enumerate(_past(lens)):
        r, dx, dy, G, raw, al, ok = step(i, A, T, done)
        w = torch.where(ok, al * T[:A], torch.zeros_like(al))
        cd = sum(r[:, 6 + ch:7 + ch] * d[ch, :A] for ch in range(3))
        acc[:A] += w * cd
        da = torch.where(ok & (raw < 0.99), T[:A] * cd - (total[:A] - acc[:A]) / (1 - al),
                         torch.zeros_like(al))
        T[:A] -= w
        dp = da * al
        s = [(-dp * (r[:, 2:3] * dx + r[:, 3:4] * dy)), (-dp * (r[:, 4:5] * dy + r[:, 3:4] * dx)),
             -0.5 * dp * dx * dx, -dp * dx * dy, -0.5 * dp * dy * dy, da * G,
             w * d[0, :A], w * d[1, :A], w * d[2, :A]]
        drec.index_add_(0, st["pairs"][start[:A] + i].long(),
                        torch.stack([t.sum(1) for t in s], 1))
    return drec


def _past(lens):
    """Number of tiles (longest list first) that have a list entry i, for i = 0, 1, ..."""
    host = lens.tolist()
    n = len(host)
    for i in range(host[0]):
        while host[n - 1] <= i:
            n -= 1
        yield n


def _window():
    x = torch.arange(11, dtype=torch.float64, device="cuda") - 5
    w = torch.exp(-x * x / (2 * 1.5 ** 2))
    return w / w.sum()


def _loss64(img, target, lam):
    w = _window()

    def blur(t):
        t = torch.nn.functional.pad(t, (5, 5, 5, 5))
        t = sum(w[i] * t[:, i:t.shape[1] - 10 + i] for i in range(11))
        return sum(w[i] * t[:, :, i:t.shape[2] - 10 + i] for i in range(11))

    x = img.double().requires_grad_(True)
    y = target.double()
    mx, my = blur(x), blur(y)
    vx, vy, vxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    S = ((2 * mx * my + 1e-4) * (2 * vxy + 9e-4)) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
    loss = (1 - lam) * (x - y).abs().mean() + lam * (1 - S.mean())
    loss.backward()
    return x.grad, loss.detach().reshape(1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("frame", "train", "lists", "select"):
        return None          # whole calls; lists and selections are whole numbers
    st = prepare(case, seed)
    if kind == "gaussians":
        gs = _decode64(st["cam_py"], st["a"], st["idx"], st["w"], st["mlp"])
        rec, _ = _project64(st["cam_py"], gs)
        return dict(gs, rec=rec, key=None, rect=None, tiles=None, tile_count=None)
    if kind == "blend":
        img, T = _blend64(st)
        return img, T, None
    if kind == "blend_bwd":
        return _blend64(st, st["dimg"])
    if kind == "loss":
        return _loss64(st["img"], st["target"], 0.2)
    j = st["idx"].long()
    leaves = {**{n: st["a"][n][j].double() for n in ("feat", "offs", "lv")},
              **{n: t.double() for n, t in st["mlp"].items()}}
    for t in leaves.values():
        t.requires_grad_(True)
    gs = _decode64(st["cam_py"], st["a"], st["idx"], st["w"], st["mlp"], leaves=leaves)
    rec, _ = _project64(st["cam_py"], gs)
    # the visible set is the one that was projected, whatever 64 bits say at its edge
    seen = (st["rect"][:, 0] != st["rect"][:, 1])[:, None] & (rec[:, 10:11] > 0)
    torch.where(seen, rec[:, :9] * st["drec"].double(), torch.zeros_like(rec[:, :9])).sum().backward()
    out = {}
    for n in ("feat", "offs", "lv"):
        out[n] = torch.zeros_like(st["a"][n], dtype=torch.float64)
        out[n][j] = leaves[n].grad
    return dict(out, **{n: leaves[n].grad for n in st["mlp"]})


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    px = case.get("W", 0) * case.get("H", 0)
    flop_anchor = 2 * (96 * 36 + 110 * 32)                  # decoder layers of one anchor
    if kind == "select":
        n = case["anchors"]
        return {"bytes": 17 * n + 8 * n // 30, "flops": 30 * n}
    if kind == "gaussians":
        m = case["anchors"]
        return {"bytes": m * (8 + 12 + 128 + 120 + 12) + m * K * (56 + 64), "flops": m * (flop_anchor + K * 250)}
    if kind == "params_bwd":
        m = case["anchors"]
        per = 8 + 12 + 128 + 120 + 12 + 2 * (128 + 120 + 12)    # inputs, gradients read and written
        return {"bytes": m * (per + K * (56 + 36 + 8)), "flops": m * (3 * flop_anchor + K * 600)}
    if kind in ("lists", "blend", "blend_bwd"):
        G = case["gaussians"]
        pairs = 2.6 * G                                     # of these screen distributions
        if kind == "lists":
            return {"bytes": 16 * G + 4 * pairs, "flops": 20 * pairs}
        seen = 0.65 * G * 48 + 4 * pairs
        if kind == "blend":
            return {"bytes": seen + px * 20, "flops": 16 * 110 * pairs}
        return {"bytes": seen + px * 20 + 0.65 * G * 36 + 36 * G, "flops": 40 * 110 * pairs}
    if kind == "loss":
        planes = 2 + 1 + (2 if case["cached"] else 0)
        moments = 3 if case["cached"] else 5
        return {"bytes": 12 * px * planes, "flops": 3 * px * (44 * (moments + 3) + 60)}
    # whole calls: each anchor's selection data once, the selected anchors, Gaussians and pixels
    n = case["anchors"]
    m = min(n, 0.05 * n + 2000)
    fwd_b = 17 * n + m * 280 + m * K * (48 + 16) + px * 16
    fwd_f = 30 * n + m * (flop_anchor + K * 250) + 16 * 60 * px
    if kind == "frame":
        return {"bytes": fwd_b, "flops": fwd_f}
    v = case["views"]
    return {"bytes": v * (fwd_b + m * (540 + K * 92) + px * 60) + m * 65 * 28,
            "flops": v * (fwd_f + m * 3 * flop_anchor + 40 * 60 * px + 3 * px * 320)}
