"""J.2 with and without the stored plane of guide bytes gives the same bits:
a request whose scratch does not fit under the HBM cap with the plane runs
without it, and is accepted wherever the filter's own scratch fits."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def _need(bw, bh):
    """Scratch of a device-resident EPF + Gaborish request without the plane:
    status words, XYB, sigma, J.2 output, block list, each 256-byte aligned."""
    up = lambda v: (v + 255) // 256 * 256
    return (up(8 * 4) + 2 * up(12 * 64 * bw * bh) + up(2 * bw * bh) + up(4 * bw * bh))


@pytest.mark.parametrize("xs,ys", [(1, 1), (8, 8), (13, 9), (31, 70), (200, 133), (641, 335)])
@pytest.mark.parametrize("dc", ["noise", "smooth"])
def test_plane_or_not(gpu_lib, xs, ys, dc):
    kw = dict(coef_scale=2.0, acmul=0.5) if dc == "smooth" else {}
    img = synth.make_image(xs, ys, 77 + xs, dc=dc, **kw)
    p = binding.filter_defaults(epf=1, gab=1)
    need = _need((xs + 7) // 8, (ys + 7) // 8)
    with binding.Context(device=0) as ctx:
        want = binding.decode(ctx, img, p, binding.OUT_F32_LINEAR)
    with binding.Context(device=0, hbm_cap_bytes=need) as ctx:
        got = binding.decode(ctx, img, p, binding.OUT_F32_LINEAR)
    assert np.array_equal(want.view(np.uint32), got.view(np.uint32))
    with binding.Context(device=0, hbm_cap_bytes=need - 256) as ctx:
        with pytest.raises(binding.JxlrError) as e:
            binding.decode(ctx, img, p, binding.OUT_F32_LINEAR)
        assert e.value.status == binding.JXLR_ENOMEM
