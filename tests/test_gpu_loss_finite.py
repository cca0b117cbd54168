"""L1 + D-SSIM where the numerator factor A2 = 2 cov(x, y) + C2 of the SSIM map vanishes: S is 0 there
and its partial derivatives are finite (dS/d(cov) = 2 A1 / (B1 B2)).  FP32 meets A2 = 0 exactly wherever
the covariance passes -C2 / 2, now and then."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda, lib_ready

pytestmark = pytest.mark.gpu

C1, C2 = 0.01 ** 2, 0.03 ** 2


def run(abi, x, y, lam, stats=None):
    import torch
    dimg = torch.full(x.shape, 7.0, device="cuda")
    loss = torch.zeros(1, device="cuda")
    scr = torch.empty(abi.loss_l1_ssim_scratch_bytes(*x.shape), dtype=torch.uint8, device="cuda")
    abi.loss_l1_ssim(cuda(x), cuda(y), lam, dimg, loss, scr, target_stats=stats)
    return loss.item(), dimg.cpu().numpy()


def test_gradient_where_a2_is_zero():
    """Image 1, target 0, so that cov = -mx my; target moments given such that A2 walks through 0 by
    single FP32 steps.  Only D-SSIM (lambda 1).  Tolerance: B2 = 0.25 + (a cancellation of a few
    1e-7), A2 and my exact to a few FP32 roundings: relative errors of 1e-6 to 1e-5."""
    abi = lib_ready()
    shape = (1, 64, 96)
    x, y = np.ones(shape, np.float32), np.zeros(shape, np.float32)
    half = np.float32(0.5) * np.float32(0.03 * 0.03)
    step = np.arange(-48, 48, dtype=np.int32)
    my = np.broadcast_to((half.view(np.int32) + step).view(np.float32), shape).copy()
    eyy = (my * my + np.float32(0.25)).astype(np.float32)
    _, got = run(abi, x, y, 1.0, cuda(np.stack([my, eyy])))
    win = oracle.gaussian_window()
    d = [a.astype(np.float64) for a in (x, y, my, eyy)]
    mx, exx = oracle._blur(d[0], win), oracle._blur(d[0] ** 2, win)
    A1, A2 = 2 * mx * d[2] + C1, C2 - 2 * mx * d[2]
    B1, B2 = mx * mx + d[2] ** 2 + C1, exx - mx * mx + d[3] - d[2] ** 2 + C2
    q = 1 / (B1 * B2)
    S = A1 * A2 * q
    g1 = 2 * d[2] * (A2 - A1) * q + 2 * S * mx * (1 / B2 - 1 / B1)
    want = -(oracle._blur(g1, win) + 2 * d[0] * oracle._blur(-S / B2, win)
             + d[1] * oracle._blur(2 * A1 * q, win)) / S.size
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)


@pytest.mark.parametrize("cached", [False, True])
def test_halves_that_exclude_each_other(cached):
    """Image 1 in the left half, target t in the right one: x y = 0, so cov = -mx my; t goes through
    96 consecutive floats (one per plane) about the value that makes the covariance -C2 / 2 on a
    column next to the border.  Tolerances as in the other oracle tests of the loss: the moments'
    FP32 cancellation, a few 1e-7 of 1 against C2 = 9e-4."""
    import torch
    abi = lib_ready()
    C, H, W = 96, 24, 48
    x = np.zeros((C, H, W), np.float32)
    x[..., :W // 2] = 1.0
    mask = np.zeros((1, H, W))
    mask[..., W // 2:] = 1.0
    win = oracle.gaussian_window()
    p = oracle._blur(x[:1].astype(np.float64), win)[0, H // 2, W // 2 + 1]
    q = oracle._blur(mask, win)[0, H // 2, W // 2 + 1]
    t = np.float32(0.5 * C2 / (p * q)).view(np.int32) + np.arange(-C // 2, C // 2, dtype=np.int32)
    y = (t.view(np.float32)[:, None, None] * mask).astype(np.float32)
    stats = None
    if cached:
        stats = torch.empty(2, C, H, W, device="cuda")
        abi.ssim_target_stats(cuda(y), stats)
    loss, got = run(abi, x, y, 0.2, stats)
    L_ref, want = oracle.photometric_loss(x, y, 0.2)
    assert np.isfinite(got).all()
    assert abs(loss - L_ref) <= 1e-4
    assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want)
