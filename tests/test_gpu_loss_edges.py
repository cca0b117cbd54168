"""L1 + D-SSIM at the edges of its column strips (64 columns, two per lane) and row pairs: odd and
tiny images, several channels, images past one strip, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda, lib_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cached", [False, True])
@pytest.mark.parametrize("shape", [(1, 6, 6), (2, 7, 8), (2, 9, 63), (3, 8, 64), (3, 17, 65),
                                   (3, 54, 129), (1, 109, 131), (5, 33, 7)])
def test_l1_ssim_strip_edges(shape, cached):
    import torch
    abi = lib_ready()
    rng = np.random.default_rng(sum(shape))
    x = rng.uniform(size=shape).astype(np.float32)
    y = np.clip(x + rng.normal(0, 0.15, size=shape), 0, 1).astype(np.float32)
    L_ref, g_ref = oracle.photometric_loss(x, y, 0.2)
    dimg = torch.full(shape, 7.0, device="cuda")
    loss = torch.zeros(1, device="cuda")
    scr = torch.empty(abi.loss_l1_ssim_scratch_bytes(*shape), dtype=torch.uint8, device="cuda")
    stats = None
    if cached:
        stats = torch.empty((2,) + shape, device="cuda")
        abi.ssim_target_stats(cuda(y), stats)
    abi.loss_l1_ssim(cuda(x), cuda(y), 0.2, dimg, loss, scr, target_stats=stats)
    torch.cuda.synchronize()
    # the moments' FP32 cancellation (a few 1e-7 of 1 against C2 = 9e-4) bounds both
    assert abs(loss.item() - L_ref) <= 1e-4
    assert np.linalg.norm(dimg.cpu().numpy() - g_ref) <= 1e-3 * np.linalg.norm(g_ref)


def test_l1_ssim_unaligned_planes():
    """Planes that start 4 bytes off an 8-byte boundary take the scalar accesses."""
    import torch
    abi = lib_ready()
    shape = (3, 20, 70)
    n = int(np.prod(shape))
    rng = np.random.default_rng(1)
    x = rng.uniform(size=shape).astype(np.float32)
    y = rng.uniform(size=shape).astype(np.float32)

    def off(a):
        t = torch.empty(n + 1, device="cuda")[1:]
        t.copy_(cuda(a).reshape(-1))
        return t.reshape(shape)
    out = []
    for place in (cuda, off):
        dimg = place(np.zeros(shape, np.float32))
        scr = torch.empty(abi.loss_l1_ssim_scratch_bytes(*shape), dtype=torch.uint8, device="cuda")
        abi.loss_l1_ssim(place(x), place(y), 0.2, dimg, None, scr)
        out.append(dimg.cpu().numpy())
    assert np.array_equal(out[0], out[1])
