"""Scratch of a JPEG1 request: sample planes only for the components that go
through one (subsampled, or with the M.6.3 side channel).  Under a cap of
exactly that the request runs, with the same result; one byte less refuses it."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def up(v):
    return (v + 255) // 256 * 256


@pytest.mark.parametrize("sampling", ["grey", "444", "420"])
@pytest.mark.parametrize("gab", [(), (0,), (1,)])
@pytest.mark.parametrize("cond", [None, (40.0, 0.5)])
@pytest.mark.parametrize("host", [False, True])
def test_cap(gpu_lib, sampling, gab, cond, host):
    import torch
    st = synth.make_jpeg(203, 141, 9, sampling=sampling, gab=True, cond=cond)
    hmax = max(c['h_samp'] for c in st['components'])
    need = up(32)
    for i, c in enumerate(st['components']):
        if i not in gab:
            c['gab'] = None
        n = c['coeffs'].shape[0] * c['coeffs'].shape[1]
        planes = 2 if i in gab else 0 if c['h_samp'] == hmax else 1
        need += planes * up(256 * n) + (up(128 * n) if host else 0)
        need += 4 * up(4 * n) + 2 * up(n) if cond else 0
    need += up(3 * 203 * 141) if host else 0
    src = st if host else binding.jpeg_to_device(st, torch)

    def run(cap):
        out = (np.zeros((141, 203, 3), np.uint8) if host else
               torch.zeros((141, 203, 3), dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        with binding.Context(device=0, hbm_cap_bytes=cap) as ctx:
            ctx.poll(ctx.submit_jpeg(src, out, binding.OUT_U8_SRGB, not host, not host))
        return out if host else out.cpu().numpy()

    assert np.array_equal(run(0), run(need))
    with pytest.raises(binding.JxlrError) as e:
        run(need - 1)        # (a cap of 0 is none)
    assert e.value.status == binding.JXLR_ENOMEM
