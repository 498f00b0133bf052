"""Row kernel of the JPEG1 path at its edges: images narrower than a block,
ragged widths, subsampling along one axis only, a luma component that is
the subsampled one, output rows whose stride or start allows no wide stores.
Bounds as in test_gpu_jpeg1 (binary32 samples of magnitude <= ~2 against the
FP64 oracle: 1e-5; bytes within 1)."""
import numpy as np
import pytest

from oracle import jpeg1 as J
from paper_1908_03565_gb300 import synth
from test_gpu_parity import B  # noqa: F401

pytestmark = pytest.mark.gpu


def _stream(xs, ys, samp, seed, gab=()):
    """Components with the sampling factors samp on grids that just cover the image."""
    hmax, vmax = max(h for h, _ in samp), max(v for _, v in samp)
    comps = []
    for i, (h, v) in enumerate(samp):
        w = 8 * -(-xs // (8 * (hmax // h)))
        t = 8 * -(-ys // (8 * (vmax // v)))
        c = synth.make_jpeg(w, t, seed + i, sampling='grey', gab=i in gab, ac_scale=3.0)
        c = dict(c['components'][0], h_samp=h, v_samp=v)
        comps.append(c)
    return {'xsize': xs, 'ysize': ys, 'components': comps}


@pytest.mark.parametrize("xs,ys", [(1, 1), (7, 9), (8, 8), (17, 5), (129, 23), (258, 16)])
@pytest.mark.parametrize("samp", [((2, 2), (1, 1), (1, 1)), ((2, 1), (1, 1), (1, 1)),
                                  ((1, 2), (1, 1), (1, 1)), ((1, 1), (2, 2), (2, 1)),
                                  ((1, 1), (1, 1), (1, 1)), ((1, 1),)])
def test_rows(B, xs, ys, samp):  # noqa: F811
    import torch
    st = _stream(xs, ys, samp, 31 * xs + ys)
    want = J.rasterize(st)
    ds = B.jpeg_to_device(st, torch)
    with B.Context(device=0) as ctx:
        for dtype, tdt, size in ((0, torch.float32, 4), (1, torch.float16, 2), (2, torch.uint8, 1)):
            for pad, lead in ((0, 0), (5, 0), (3, 1)):      # elements behind a row, before the first
                out = torch.full((ys * (3 * xs + pad) + lead,), 7, dtype=tdt, device="cuda")
                view = out[lead:]
                ctx.poll(ctx.submit_jpeg(ds, view, dtype, out_stride=size * (3 * xs + pad)))
                rows = view.cpu().numpy()[:ys * (3 * xs + pad)].reshape(ys, 3 * xs + pad)
                assert np.all(rows[:, 3 * xs:] == 7) and np.all(out[:lead].cpu().numpy() == 7)
                got = rows[:, :3 * xs].reshape(ys, xs, 3).astype(np.float64)
                if dtype == 2:
                    assert np.abs(got - J.to_u8(want)).max() <= 1
                else:
                    ulp = np.spacing(np.abs(want / 255.0).astype(np.float16)).astype(np.float64)
                    assert np.all(np.abs(got - want / 255.0) <= 1e-5 + (0.5 * ulp if dtype else 0))
