"""Requests in flight together under an HBM cap: the guide bytes that J.2 can
use cost none of them its place.  What the context admits is what the
filters' own scratch, computed here, allows; it holds that and, as far as the cap
leaves room, guide bytes."""
import numpy as np
import pytest

from paper_1908_03565_gb300 import binding, synth

pytestmark = pytest.mark.gpu

MiB = 1 << 20


def up(v, a=256):
    return (v + a - 1) // a * a


def need(xs, ys, kind):
    """Scratch of a device-resident request: status words; XYB (but for caller
    XYB); with the EPF sigma, J.2 output and block list."""
    n = ((xs + 7) // 8) * ((ys + 7) // 8)
    return (up(32) + (up(768 * n) if kind != "xyb" else 0) +
            (up(2 * n) + up(768 * n) + up(4 * n) if kind != "gab" else 0))


class Slots:
    """The arenas of a context: a request takes the smallest idle one that holds
    it, else the largest, grown to whole MiB; idle ones are given up first."""

    def __init__(self, n, cap):
        self.arena, self.busy, self.cap = [0] * n, [False] * n, cap

    def take(self, size):
        if size > self.cap:
            return binding.JXLR_ENOMEM, None
        idle = [i for i, b in enumerate(self.busy) if not b]
        if not idle:
            return binding.JXLR_EBUSY, None
        fit = [i for i in idle if self.arena[i] >= size]
        s = min(fit, key=lambda i: self.arena[i]) if fit else max(idle, key=lambda i: self.arena[i])
        if self.arena[s] < size:
            if sum(self.arena) - self.arena[s] + size > self.cap:
                for i in idle:
                    if i != s:
                        self.arena[i] = 0
                if sum(self.arena) - self.arena[s] + size > self.cap:
                    return binding.JXLR_EBUSY, None
            self.arena[s] = up(size, MiB)
        self.busy[s] = True
        return binding.JXLR_OK, s


class Work:
    """An image and its result in a context without a cap."""

    def __init__(self, torch, ctx, xs, ys, kind):
        self.kind, self.size, self.need = kind, (xs, ys), need(xs, ys, kind)
        img = synth.make_image(xs, ys, 3 + xs, coef_scale=2.0, acmul=0.5, dc="smooth")
        self.img = binding.to_device(img, torch)
        self.p = binding.filter_defaults(epf=kind != "gab", gab=1)
        if kind == "xyb":
            x = binding.decode(ctx, img, binding.filter_defaults(), binding.OUT_F32_XYB)
            self.xyb = torch.from_numpy(np.ascontiguousarray(x.transpose(2, 0, 1))).cuda()
        self.torch = torch
        torch.cuda.synchronize()
        out, t = self.submit(ctx)
        ctx.poll(t)
        self.want = out.cpu()

    def submit(self, ctx):
        xs, ys = self.size
        out = self.torch.zeros((ys, xs, 3), dtype=self.torch.float32, device="cuda")
        self.torch.cuda.synchronize()
        if self.kind == "xyb":
            return out, ctx.submit_xyb(self.xyb, xs, ys, self.img["vmap"], self.img["acmul"],
                                       self.img["sharpness"], self.p, out,
                                       binding.OUT_F32_LINEAR)
        return out, ctx.submit(self.img, self.p, out, binding.OUT_F32_LINEAR, True)

    def right(self, out):
        return self.torch.equal(out.cpu().view(self.torch.int32), self.want.view(self.torch.int32))


@pytest.mark.parametrize("kind", ["epf", "xyb"])
@pytest.mark.parametrize("extra", [-256, 0, 2 * MiB, 5 * MiB])
def test_two_at_once(gpu_lib, kind, extra):
    """Two equal requests fit from the first one's arena and the second one's
    need on; with the guide bytes of both they would want 3 MiB more each."""
    import torch
    with binding.Context(device=0) as ctx:
        w = Work(torch, ctx, 1024, 1024, kind)
    with binding.Context(device=0, max_slots=2, hbm_cap_bytes=up(w.need, MiB) + w.need + extra) as ctx:
        got = [w.submit(ctx)]
        assert ctx.device_bytes() == up(w.need, MiB) + 3 * MiB     # with its guide bytes
        if extra < 0:
            with pytest.raises(binding.JxlrError) as e:
                w.submit(ctx)
            assert e.value.status == binding.JXLR_EBUSY
        else:
            got.append(w.submit(ctx))
            # the first one's stay where the second one's scratch leaves room
            assert ctx.device_bytes() == 2 * up(w.need, MiB) + (3 * MiB if extra == 5 * MiB else 0)
        for out, t in got:
            ctx.poll(t)
            assert w.right(out)


def test_any_order(gpu_lib):
    import torch
    rng = np.random.default_rng(8)
    with binding.Context(device=0) as ctx:
        works = [Work(torch, ctx, xs, ys, kind)
                 for xs, ys in [(131, 77), (520, 392), (768, 512), (1024, 1024)]
                 for kind in ("gab", "epf", "xyb")]
    model = Slots(4, 37 * MiB)
    flight, refused, kept = [], 0, 0
    with binding.Context(device=0, max_slots=4, hbm_cap_bytes=model.cap) as ctx:
        for _ in range(240):
            if flight and rng.random() < 0.4:
                w, s, out, t = flight.pop(rng.integers(len(flight)))
                ctx.poll(t)
                model.busy[s] = False
                assert w.right(out)
                continue
            w = works[rng.integers(len(works))]
            want, s = model.take(w.need)
            try:
                out, t = w.submit(ctx)
                assert want == binding.JXLR_OK
                flight.append((w, s, out, t))
            except binding.JxlrError as e:
                assert e.status == want
                refused += not all(model.busy)
            assert 0 <= ctx.device_bytes() - sum(model.arena) <= max(0, model.cap - sum(model.arena)) + MiB
            kept += ctx.device_bytes() > sum(model.arena)
        for w, s, out, t in flight:
            ctx.poll(t)
            assert w.right(out)
    assert refused > 5    # refusals by the cap, not for want of a slot
    assert kept > 5       # times with guide bytes beside the scratch
