"""Requests whose kernels start while the one before them ends (programmatic
launches): images of different content through one slot, one after another
without a pause, each bit for bit as alone; the EPF ones also as the
no-allocation entry point (plain launches) gives them."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xs,ys", [(1, 1), (48, 40), (131, 77), (1024, 520)])
@pytest.mark.parametrize("epf", [0, 1])
@pytest.mark.parametrize("dc", [0, 1, 2])     # none; F.2; F.2 and Annex H
def test_back_to_back(gpu_lib, xs, ys, epf, dc):
    import torch
    imgs = [synth.make_image(xs, ys, 3, coef_scale=2.0, acmul=0.5, dc='smooth'),
            synth.make_image(xs, ys, 4), synth.make_image(xs, ys, 5, dc='smooth')]
    p = binding.filter_defaults(epf=epf, gab=1, dc_smooth=dc > 0, lf_predict=dc > 1)
    dev = [binding.to_device(i, torch) for i in imgs]
    new = lambda: torch.full((ys, xs, 3), 7, dtype=torch.float32, device="cuda")
    with binding.Context(device=0) as ctx:
        want = [binding.decode(ctx, i, p, binding.OUT_F32_LINEAR) for i in imgs]
        outs = [new() for _ in range(24)]
        torch.cuda.synchronize()
        for k, o in enumerate(outs):
            ctx.poll(ctx.submit(dev[k % 3], p, o, binding.OUT_F32_LINEAR, True))
    for k, o in enumerate(outs):
        assert np.array_equal(o.cpu().numpy().view(np.uint32), want[k % 3].view(np.uint32))
    if epf and not dc:
        for d, w in zip(dev, want):
            o = new()
            torch.cuda.synchronize()
            binding.run_noalloc(d, p, o, binding.OUT_F32_LINEAR)
            torch.cuda.synchronize()
            assert np.array_equal(o.cpu().numpy().view(np.uint32), w.view(np.uint32))
