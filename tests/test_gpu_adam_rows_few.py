"""Adam over touched rows where a warp's window of rows changes with their number (4, 32 or 64
for rows of up to 8, 128), at the edges of the windows, against the formula in FP64; and its time on few rows."""
import numpy as np
import pytest

from gpu_helpers import lib_ready

pytestmark = pytest.mark.gpu

FEW, WIN = 32768, 152 * 128      # rows from which windows of 32 (64) are taken; one window of 128 per SM
MANY, MANY_SHORT = 24 * WIN, 16 * WIN      # rows from which windows of 128 are taken


@pytest.mark.parametrize("row_len", [1, 8, 9, 33])
@pytest.mark.parametrize("rows,share", [(3, 1.0), (5, 1.0), (FEW - 1, 1.0), (FEW, 0.3), (FEW + 63, 1.0),
                                        (FEW + 65, 0.02), (MANY_SHORT - 1, 0.05), (MANY_SHORT + 129, 0.05),
                                        (MANY - 1, 0.05), (MANY, 0.05), (MANY + 127, 0.05), (MANY + 129, 0.0)])
def test_adam_rows_by_number_of_rows(rows, share, row_len):
    import torch
    abi = lib_ready()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + row_len)
    rnd = lambda: torch.randn(rows, row_len, generator=gen, device="cuda")  # noqa: E731
    a = [rnd(), rnd(), rnd(), rnd().square()]
    hit = torch.rand(rows, generator=gen, device="cuda") < share
    hit[-1] = share > 0
    stamp = torch.where(hit, 7, 5).to(torch.int32)
    p, g, m, v = (t.clone() for t in a)
    abi.adam_rows(p, g, m, v, stamp, 7, 1e-2, 0.9, 0.999, 1e-15, 5, True)
    h = hit[:, None]
    P, G, M, V = (t.double() for t in a)
    M2, V2 = 0.9 * M + 0.1 * G, 0.999 * V + 0.001 * G * G
    P2 = P - 1e-2 * (M2 / (1 - 0.9 ** 5)) / (torch.sqrt(V2 / (1 - 0.999 ** 5)) + 1e-15)
    # beta1, beta2 are FP32 (1 - 0.999 to 2e-5 relative); the quotient a few ulp
    step = (P2 - P).abs()
    assert (m.double() - torch.where(h, M2, M)).abs().le(1e-5 * M2.abs() + 1e-6).all()
    assert (v.double() - torch.where(h, V2, V)).abs().le(1e-4 * V2 + 1e-6).all()
    assert (p.double() - torch.where(h, P2, P)).abs().le(
        1e-5 * P2.abs() + 2e-5 * step.max().clamp_min(1.0)).all()
    for got, was in ((p, a[0]), (g, a[1]), (m, a[2]), (v, a[3])):
        assert torch.equal(got[~hit], was[~hit])
    assert not g[hit].any()


def test_few_rows_do_not_wait_for_one_another():
    """4096 rows of 32, all touched (a small scene's step): as many warps as groups of four rows, so
    the call takes a few round trips to memory.  It took 45 us in windows of 128 rows, 14.5 with a warp
    walking 32 rows one by one, and takes 4.5; the bound leaves a factor of two."""
    import torch
    abi = lib_ready()
    p, g, m, v = (torch.zeros(4096, 32, device="cuda") for _ in range(4))
    stamp = torch.ones(4096, dtype=torch.int32, device="cuda")
    best = np.inf
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(2_000_000)
        a.record()
        for _ in range(20):
            abi.adam_rows(p, g, m, v, stamp, 1, 1e-3, 0.9, 0.999, 1e-15, 5, True)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / 20)
    assert best < 10.0
