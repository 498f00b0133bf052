"""Device maps whose varblocks cross on blocks coded as covered (every block is
covered, some twice) are refused like any other map that is not a tiling
(C.5.4), by each form of the transform kernel."""
import itertools

import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu

# blocks a varblock is wide and high, per DctSelect code
WIDE = [1, 1, 1, 1, 2, 4, 1, 2, 1, 4, 2, 4, 1, 1, 1]
HIGH = [1, 1, 1, 1, 2, 4, 2, 1, 4, 1, 4, 2, 1, 1, 1]


def tiles(m):
    """C.5.4: every block covered by exactly one aligned varblock, inside."""
    bh, bw = m.shape
    count = np.zeros((bh, bw), int)
    for y, x in zip(*np.nonzero(m != 255)):
        c = m[y, x]
        if c >= 15 or x % WIDE[c] or y % HIGH[c] or x + WIDE[c] > bw or y + HIGH[c] > bh:
            return False
        count[y:y + HIGH[c], x:x + WIDE[c]] += 1
    return bool((count == 1).all())


def crossing(rng, bw, bh):
    """Aligned varblocks at random places whose first block is still free, their
    footprints crossing at times; what none of them reaches is DCT8."""
    m = np.full((bh, bw), 255, np.uint8)
    reached = np.zeros((bh, bw), bool)
    for _ in range(3 * bw * bh):
        c = rng.integers(15)
        x, y = rng.integers(bw) // WIDE[c] * WIDE[c], rng.integers(bh) // HIGH[c] * HIGH[c]
        foot = np.s_[y:y + HIGH[c], x:x + WIDE[c]]
        if x + WIDE[c] > bw or y + HIGH[c] > bh or reached[y, x] or (m[foot] != 255).any():
            continue
        m[y, x] = c
        reached[foot] = True
    m[~reached] = 0
    return m


def maps(bw, bh):
    if (bw, bh) == (2, 2):
        yield from (np.array(t, np.uint8).reshape(2, 2)
                    for t in itertools.product((0, 4, 6, 7, 255), repeat=4))
        return
    rng = np.random.default_rng(bw)
    for _ in range(80):
        yield crossing(rng, bw, bh)


@pytest.fixture(params=["grid", "persistent", "tensor cores"])
def ctx(gpu_lib, request, monkeypatch):
    if request.param == "persistent":
        monkeypatch.setenv("JXLR_RECON_VARIANT", "persistent")
    precision = binding.PREC_TC_F16X3 if request.param == "tensor cores" else binding.PREC_FP32
    with binding.Context(device=0, precision=precision) as c:
        yield c


@pytest.mark.parametrize("bw,bh", [(2, 2), (4, 4), (6, 7)])
def test_refused(ctx, bw, bh):
    import torch
    img = synth.make_image(8 * bw, 8 * bh, 5)
    dev = binding.to_device(img, torch)
    out = torch.empty((8 * bh, 8 * bw, 3), dtype=torch.uint8, device="cuda")
    p = binding.filter_defaults()
    seen = {True: 0, False: 0}
    ms = list(maps(bw, bh))
    vmaps = [torch.from_numpy(m).cuda() for m in ms]
    torch.cuda.synchronize()
    for m, vmap in zip(ms, vmaps):
        want = tiles(m)
        seen[want] += 1
        t = ctx.submit(dict(dev, vmap=vmap), p, out, binding.OUT_U8_SRGB, True)
        try:
            ctx.poll(t)
            assert want, m
        except binding.JxlrError as e:
            assert e.status == binding.JXLR_EINVAL and not want, m
    assert min(seen.values()) >= 2
