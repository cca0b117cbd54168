"""Training towards targets that are made for one step and freed: the D-SSIM moments kept per target must
not serve another tensor that took the same memory."""
import pytest

import synth
from gpu_helpers import lib_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("views", [1, 2])
def test_freed_target(views):
    import torch
    abi = lib_ready()
    from paper_2403_17898_gb300.render import Trainer
    sc, mlp, cams = synth.CONFIGS["cube4k_128"]()
    tr = Trainer(sc, mlp, 128, 128, ssim_lambda=0.2)
    cam = cams[0]
    tr.render(cam, infer=False)
    img = tr.img.clone()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(2)
    targets = [torch.rand(3, 128, 128, generator=gen, device="cuda") * s for s in (1.0, 0.4, 0.7)]
    scr = torch.empty(abi.loss_l1_ssim_scratch_bytes(3, 128, 128), dtype=torch.uint8, device="cuda")
    places = set()
    for y in targets:
        want, d = torch.zeros(1, device="cuda"), torch.empty_like(img)
        abi.loss_l1_ssim(img, y, 0.2, d, want, scr)
        t = y.clone()
        places.add(t.data_ptr())
        tr.train_step([cam] * views, [t] * views, update=False)
        # a sum of 5e4 values in FP32 parts, with moments given or not
        assert abs(tr.loss.item() - views * want.item()) <= 1e-6 * views
        del t
    assert len(places) < len(targets)                # some memory was taken again


def test_kept_target_is_looked_up_once():
    import torch
    lib_ready()
    from paper_2403_17898_gb300.render import Trainer
    sc, mlp, cams = synth.CONFIGS["cube4k_128"]()
    tr = Trainer(sc, mlp, 128, 128, ssim_lambda=0.2)
    batch = torch.rand(2, 3, 128, 128, device="cuda")
    st = torch.cuda.current_stream()
    first = [tr._target_stats(batch[i], st) for i in range(2)]       # views of a tensor that lives
    assert all(tr._target_stats(batch[i], st) is first[i] for i in range(2))
    batch.mul_(0.5)
    assert tr._target_stats(batch[0], st) is not first[0]
