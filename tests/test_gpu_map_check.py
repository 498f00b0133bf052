"""The transform kernel's check of device maps (C.5.4) refuses exactly the
maps that the host check of host inputs refuses: varblock maps with single
bytes changed, at sizes whose last cells are partial."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def _status(ctx, img, params, torch, device):
    out = torch.empty((img['ysize'], img['xsize'], 3), dtype=torch.uint8, device="cuda")
    host = np.empty((img['ysize'], img['xsize'], 3), np.uint8)
    try:
        if device:
            t = ctx.submit(binding.to_device(img, torch), params, out, binding.OUT_U8_SRGB, True)
        else:
            t = ctx.submit(img, params, host, binding.OUT_U8_SRGB, False, out_on_device=False)
        ctx.poll(t)
        return binding.JXLR_OK
    except binding.JxlrError as e:
        return e.status


@pytest.mark.parametrize("xs,ys", [(8, 8), (40, 24), (72, 104)])
def test_same_maps_refused(gpu_lib, xs, ys):
    import torch
    rng = np.random.default_rng(xs)
    img = synth.make_image(xs, ys, 5)
    p = binding.filter_defaults(gab=1)
    refused = 0
    with binding.Context(device=0) as ctx:
        assert _status(ctx, img, p, torch, True) == binding.JXLR_OK
        for _ in range(60):
            bad = dict(img, vmap=img['vmap'].copy())
            for _ in range(rng.integers(1, 3)):
                by, bx = rng.integers(bad['vmap'].shape[0]), rng.integers(bad['vmap'].shape[1])
                bad['vmap'][by, bx] = rng.choice([0, 1, 4, 5, 6, 7, 8, 9, 10, 11, 14, 15, 200, 255])
            want = _status(ctx, bad, p, torch, False)
            assert _status(ctx, bad, p, torch, True) == want, bad['vmap']
            refused += want != binding.JXLR_OK
        assert refused > 20
        assert _status(ctx, img, p, torch, True) == binding.JXLR_OK
