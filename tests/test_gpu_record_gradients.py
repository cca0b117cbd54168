"""Renderer.drec after a backward: the view's record gradients, and zero in every row past its Gaussians,
also when the view before had more."""
import numpy as np
import pytest

import synth
from gpu_helpers import lib_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_rows_past_the_view_are_zero(precision):
    import torch
    lib_ready()
    from paper_2403_17898_gb300.render import Trainer
    sc, mlp, cams = synth.CONFIGS["cube4k_128"]()
    far = synth.look_at_camera(np.array([0.0, -60.0, 20.0]), np.zeros(3), 128, 128, d_max=30.0)
    tr = Trainer(sc, mlp, 128, 128, precision=precision)
    dimg = torch.full((3, 128, 128), 1e-3, device="cuda")
    seen, counts = [], []
    for cam in (cams[0], far, cams[0], far):
        c = tr.render(cam, infer=False)
        counts.append(c.n_gaussians)
        tr.backward(cam, dimg, tr.grads, tr._dmlp_struct,
                    on_drec=lambda st: seen.append(tr.drec.clone()))
    assert 0 < counts[1] < counts[0] <= tr.g_cap
    for n, d in zip(counts, seen):
        assert d[:n].any() and not d[n:].any()
    # the same view gives the same gradients whatever came before (float atomics: order of sums)
    for a, b in ((0, 2), (1, 3)):
        assert (seen[a] - seen[b]).norm() <= 1e-4 * seen[a].norm()


@pytest.mark.parametrize("cap,off", [(1, 0), (1000, 0), (1000, 1), (200_000, 0)])
def test_renewed_rows(cap, off):
    """ogs_renew_records: the rows of the frame before go to zero, nothing else is touched, and the next
    call clears this frame's."""
    import torch
    abi = lib_ready()
    buf = torch.zeros(cap * 9 + 16, device="cuda")
    drec = buf[off:off + cap * 9].reshape(cap, 9)
    counts = torch.zeros(8, dtype=torch.int32, device="cuda")
    held = torch.zeros(2, dtype=torch.int32, device="cuda")
    before = 0
    for n in (cap, cap // 2, 0, 1, cap // 3, cap + 5, cap):
        counts[1] = n
        buf.fill_(2.0)
        abi.renew_records(drec, counts, held)
        want = torch.full_like(buf, 2.0)
        want[off:off + 9 * min(before, cap)] = 0
        assert torch.equal(buf, want)
        assert held.tolist() == [n, 0]
        before = n
