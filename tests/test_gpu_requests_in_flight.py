"""Requests of several kinds and sizes in flight together, each bit for bit as
alone: on one stream, where a request's first kernels follow the last of the
one before without a pause, and on the slots' own streams, where they overlap
(kernels of one request start while the one before them in it ends)."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu

KINDS = [dict(epf=1, gab=1, dc_smooth=1, lf_predict=1), dict(gab=1), dict(epf=1, gab=1),
         dict(dc_smooth=1), dict(), dict(epf=1, dc_smooth=1), dict(epf=1, gab=1, qco=1)]
SIZES = [(1024, 520), (48, 40), (131, 77), (601, 403), (1, 1)]


@pytest.mark.parametrize("own_streams", [False, True])
def test_as_alone(gpu_lib, own_streams):
    import torch
    works = []
    with binding.Context(device=0) as ctx:
        for i, (kw, (xs, ys)) in enumerate([(k, s) for k in KINDS for s in SIZES]):
            img = synth.make_image(xs, ys, 40 + i, coef_scale=2.0, acmul=0.5, dc="smooth")
            p = binding.filter_defaults(**kw)
            want = binding.decode(ctx, img, p, binding.OUT_F32_LINEAR)
            works.append((binding.to_device(img, torch), p, want))
    rng = np.random.default_rng(3)
    stream = None if own_streams else torch.cuda.Stream()
    with binding.Context(device=0, max_slots=8,
                         stream=None if own_streams else stream.cuda_stream) as ctx:
        for _ in range(12):
            picks = rng.integers(len(works), size=8)
            outs = [torch.full(works[k][2].shape, 7, dtype=torch.float32, device="cuda") for k in picks]
            torch.cuda.synchronize()
            tickets = [ctx.submit(works[k][0], works[k][1], o, binding.OUT_F32_LINEAR, True)
                       for k, o in zip(picks, outs)]
            for t in tickets:
                ctx.poll(t)
            for k, o in zip(picks, outs):
                assert np.array_equal(o.cpu().numpy().view(np.uint32), works[k][2].view(np.uint32))
