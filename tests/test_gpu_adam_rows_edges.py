"""Adam over touched rows at the edges of a warp's 128-row window, for short and long rows, and the
clearing of a view's record gradients."""
import numpy as np
import pytest

from gpu_helpers import cuda, lib_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("row_len", [1, 3, 30, 32, 33, 200])
@pytest.mark.parametrize("rows,share", [(1, 1.0), (31, 0.5), (128, 1.0), (129, 0.1), (5000, 0.03),
                                        (5000, 0.0), (257, 1.0)])
def test_adam_rows_windows(rows, share, row_len):
    import torch
    abi = lib_ready()
    rng = np.random.default_rng(rows + row_len)
    a = [rng.normal(size=(rows, row_len)).astype(np.float32) for _ in range(4)]
    a[3] = a[3] ** 2
    hit = rng.uniform(size=rows) < share
    stamp = np.where(hit, 7, rng.integers(0, 6, size=rows)).astype(np.int32)
    p, g, m, v = (cuda(x) for x in a)
    abi.adam_rows(p, g, m, v, cuda(stamp), 7, 1e-2, 0.9, 0.999, 1e-15, 5, True)
    torch.cuda.synchronize()
    P, G, M, V = (x.astype(np.float64) for x in a)
    M2 = np.where(hit[:, None], 0.9 * M + 0.1 * G, M)
    V2 = np.where(hit[:, None], 0.999 * V + 0.001 * G * G, V)
    step = 1e-2 * (M2 / (1 - 0.9 ** 5)) / (np.sqrt(V2 / (1 - 0.999 ** 5)) + 1e-15)
    P2 = np.where(hit[:, None], P - step, P)
    # beta1, beta2 are FP32 (1 - 0.999 to 2e-5 relative); the quotient a few ulp
    np.testing.assert_allclose(m.cpu().numpy(), M2, rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(v.cpu().numpy(), V2, rtol=1e-4, atol=1e-6)
    np.testing.assert_allclose(p.cpu().numpy(), P2, rtol=1e-5, atol=2e-5 * max(1.0, np.abs(step).max()))
    assert np.array_equal(g.cpu().numpy()[~hit], a[1][~hit]) and not g.cpu().numpy()[hit].any()
    assert np.array_equal(p.cpu().numpy()[~hit], a[0][~hit])


@pytest.mark.parametrize("n,cap,off", [(0, 10, 0), (1, 10, 0), (7, 10, 0), (10, 10, 0), (99, 10, 0),
                                       (1000, 4000, 1)])
def test_clear_records(n, cap, off):
    import torch
    abi = lib_ready()
    buf = torch.ones(cap * 9 + 16, device="cuda")
    drec = buf[off:off + cap * 9].reshape(cap, 9)
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    counts[1] = n
    abi.clear_records(drec, counts)
    torch.cuda.synchronize()
    got = buf.cpu().numpy()
    k = 9 * min(n, cap)
    assert not got[off:off + k].any() and (got[:off] == 1).all() and (got[off + k:] == 1).all()
