"""L1 + D-SSIM by 32 x 32 tiles (all but large images) and by column strips: odd sizes, tile, strip and halo
edges, both sides of the line between them, against the FP64 oracle; and the time by tiles."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda, lib_ready

pytestmark = pytest.mark.gpu

LINE = 2_600_000       # values C H W from which strips are taken


@pytest.mark.parametrize("cached", [False, True])
@pytest.mark.parametrize("shape", [(1, 6, 6), (1, 1, 100_000), (2, 31, 33), (1, 32, 64), (3, 159, 213), (2, 33, 1601),
                                   (5, 161, 131), (1, 11, 236_363), (1, 1600, 1624), (1, 1600, 1625),
                                   (40, 250, 281), (3, 967, 967), (4, 1, 700_001), (2, 90_001, 17), (1, 2_100_001, 1)])
def test_l1_ssim_tiles_and_strips(shape, cached):
    import torch
    abi = lib_ready()
    rng = np.random.default_rng(shape[1] + shape[2])
    assert shape != (1, 1600, 1625) or np.prod(shape) == LINE
    x = rng.uniform(size=shape).astype(np.float32)
    y = np.clip(x + rng.normal(0, 0.15, size=shape), 0, 1).astype(np.float32)
    L_ref, g_ref = oracle.photometric_loss(x, y, 0.2)
    n = x.size
    buf = torch.full((n + 2,), 7.0, device="cuda")           # nothing outside the gradient is written
    dimg = buf[1:1 + n].reshape(shape)
    loss = torch.full((1,), 2.0, device="cuda")              # the loss is added to what is there
    scr = torch.empty(abi.loss_l1_ssim_scratch_bytes(*shape), dtype=torch.uint8, device="cuda")
    stats = None
    if cached:
        stats = torch.empty((2,) + shape, device="cuda")
        abi.ssim_target_stats(cuda(y), stats)
    abi.loss_l1_ssim(cuda(x), cuda(y), 0.2, dimg, loss, scr, target_stats=stats)
    # the moments' FP32 cancellation (a few 1e-7 of 1 against C2 = 9e-4) bounds both
    assert abs(loss.item() - 2.0 - L_ref) <= 1e-4
    assert np.linalg.norm(dimg.cpu().numpy() - g_ref) <= 1e-3 * np.linalg.norm(g_ref)
    assert buf[0].item() == 7.0 and buf[-1].item() == 7.0


def test_time_of_a_small_image():
    """480 x 270 takes a quarter of the time of 1600 x 900, for 0.09 of its pixels (18.4 us by tiles of 75 by
    strips; by strips of four rows, whose halo triples the work, it took 26.8, 0.36 of it)."""
    import torch
    abi = lib_ready()
    best = {}
    for W, H in [(480, 270), (1600, 900)] * 8:
        x, y = torch.rand(3, H, W, device="cuda"), torch.rand(3, H, W, device="cuda")
        d, loss = torch.empty_like(x), torch.zeros(1, device="cuda")
        scr = torch.empty(abi.loss_l1_ssim_scratch_bytes(3, H, W), dtype=torch.uint8, device="cuda")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        abi.loss_l1_ssim(x, y, 0.2, d, loss, scr)
        torch.cuda._sleep(2_000_000)
        a.record()
        for _ in range(20):
            abi.loss_l1_ssim(x, y, 0.2, d, loss, scr)
        b.record()
        torch.cuda.synchronize()
        best[W] = min(best.get(W, np.inf), a.elapsed_time(b))
    assert best[480] <= 0.3 * best[1600]
