"""Device maps whose varblocks overlap so that a cell has the most transform
items that any map gives it (768 of rows, or of columns, against 384 in a
tiling): the request is refused and the ones after it are unharmed."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("codes", [(8, 6), (9, 7)])     # 1x4 and 1x2 blocks; 4x1 and 2x1
@pytest.mark.parametrize("opts", [dict(), dict(epf=1, gab=1), dict(epf=1, qco=1)])
def test_refused_without_harm(gpu_lib, codes, opts):
    import torch
    img = synth.make_image(128, 96, 3)
    p = binding.filter_defaults(**opts)
    i = np.indices(img['vmap'].shape)[0 if codes[0] == 8 else 1] % 4
    bad = dict(img, vmap=np.where(i == 0, codes[0], np.where(i == 2, codes[1], 0)).astype(np.uint8))
    out = torch.empty((96, 128, 3), dtype=torch.float32, device="cuda")
    with binding.Context(device=0) as ctx:
        want = binding.decode(ctx, img, p, binding.OUT_F32_LINEAR)
        for _ in range(3):
            with pytest.raises(binding.JxlrError) as e:
                ctx.poll(ctx.submit(binding.to_device(bad, torch), p, out, binding.OUT_F32_LINEAR, True))
            assert e.value.status == binding.JXLR_EINVAL
        got = binding.decode(ctx, img, p, binding.OUT_F32_LINEAR)
    assert np.array_equal(want.view(np.uint32), got.view(np.uint32))
