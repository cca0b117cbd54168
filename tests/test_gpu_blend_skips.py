"""Blend backward: an entry that a pixel skips leaves that pixel's walk as it is.  The walk multiplies the
transmittance by the reciprocal of 1 - alpha with alpha = 0 there, which has to be exactly 1."""
import numpy as np
import pytest

from gpu_helpers import cuda, lib_ready

pytestmark = pytest.mark.gpu

W = H = 16
BG = (0.1, 0.2, 0.3)


def record(u, v, sigma, o, color, depth):
    a = 1.0 / sigma ** 2
    return [u, v, a, 0.0, a, o, *color, depth, 3 * sigma, -np.log(255.0 * o)]


def gradients(abi, torch, recs, dimg):
    rec = cuda(np.asarray(recs, np.float32))
    lst = torch.arange(len(recs), dtype=torch.int32, device="cuda")
    rng = torch.tensor([[0, len(recs)]], dtype=torch.int32, device="cuda")
    img, T = torch.zeros(3, H, W, device="cuda"), torch.zeros(H, W, device="cuda")
    nl = torch.zeros(H, W, dtype=torch.int32, device="cuda")
    abi.blend_fwd(rec, lst, rng, W, H, BG, img, T, nl)
    drec = torch.zeros(len(recs), 9, device="cuda")
    abi.blend_bwd(rec, lst, rng, W, H, BG, T, nl, cuda(dimg), drec)
    return drec.cpu().numpy(), T.cpu().numpy()


@pytest.mark.parametrize("careful", [False, True])
@pytest.mark.parametrize("n", [1, 9, 600])
def test_skipped_entries_change_nothing(n, careful):
    """One pixel carries the image gradient.  n entries between the two that it blends are blended by its
    neighbour alone: the gradients of those two must have the bits that they have without the n (the
    other pixels add zeros).  careful: an opacity that reaches the clamp."""
    import torch
    abi = lib_ready()
    x, y = 5, 3
    front = record(6.3, 4.1, 5.0, 0.995 if careful else 0.6, (0.9, 0.2, 0.4), 1.0)
    back = record(3.2, 2.7, 7.0, 0.5, (0.1, 0.8, 0.3), 900.0)
    mid = [record(x + 1.0, float(y), 0.2, 0.01, (0.5, 0.5, 0.5), 2.0 + i) for i in range(n)]
    dimg = np.zeros((3, H, W), np.float32)
    dimg[:, y, x] = (0.7, -1.3, 0.4)
    want, T0 = gradients(abi, torch, [front, back], dimg)
    got, T1 = gradients(abi, torch, [front] + mid + [back], dimg)
    assert T1[y, x] == T0[y, x] and T1[y, x + 1] < T0[y, x + 1]
    assert want.all(axis=None) or careful
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[-1], want[1])
    assert not got[1:-1].any()
