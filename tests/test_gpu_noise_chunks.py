"""K.5.2 channels at the numbers of groups where the generator's chunks change
length (on 152 SMs 8 rows up to 101 groups, 16 up to 202, then 32), against the
sequential oracle: thin images whole, of wide ones the first, an inner and the
last (ragged) group.  Zero XYB and a constant LUT of 1, so that the output is
the channels' alone; binary32 rounding as in test_gpu_noise."""
import numpy as np
import pytest

from oracle import noise as N
from test_gpu_noise import _staged
from test_gpu_parity import B, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def group(gx, gy, xs, ys):
    x0, y0 = 256 * gx, 256 * gy
    w, h = min(256, xs - x0), min(256, ys - y0)
    a = [0.22 * N.laplacian(c) for c in N.random_channels(x0, y0, w, h)]
    nr, ng = (0.01 * a[c] + 0.99 * a[2] for c in (0, 1))
    return np.s_[:, y0:y0 + h, x0:x0 + w], np.stack([nr - ng, nr + ng, 0.935669 * (nr + ng)])


@pytest.mark.parametrize("xs,ys", [
    (17, 256 * 101), (17, 256 * 101 + 1), (3, 256 * 202), (5, 256 * 202 + 40),   # 101, 102, 202, 203
    (2601, 2567), (3845, 3333)])                                                  # 121, 224
def test_chunks(B, ctx, xs, ys):  # noqa: F811
    lp = B.filter_defaults(noise=1, noise_lut=[1.0] * 16)
    got = _staged(B, ctx, np.zeros((3, ys, xs), np.float32), lp)
    nx, ny = -(-xs // 256), -(-ys // 256)
    for gx, gy in ([(0, gy) for gy in range(ny)] if nx == 1 else
                   [(0, 0), (nx // 2, ny // 2), (nx - 1, ny - 1)]):
        at, want = group(gx, gy, xs, ys)
        np.testing.assert_allclose(got[at], want, atol=2e-6, rtol=0)
    assert np.abs(got).max() > 0.1
