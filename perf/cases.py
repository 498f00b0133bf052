"""The work that users of this library give it, as measurable cases.

A case is a dict of plain values.  ``listed()`` gives the standing ones,
``draw(rng)`` another one of the same ranges, ``prepare(case, seed)`` what a
program holds before the call (inputs on the device or, for the host case, in
pinned host memory; the context; for batches the captured batch), ``run(state)``
one call as a program makes it, ``work(case)`` the bytes and operations the call
cannot do without, and ``exact(case, seed)`` the call's floating results in 64
bits by plain torch.

Two kinds of image content:

* ``bench``: the statistics of the benchmark and the parity tests: a random
  tiling of 12 varblock shapes, Laplace(0, 64 / (1 + u + v)) coefficients, a
  log-uniform quant field, random chroma-from-luma factors.  About 40% of the
  blocks reach the edge-preserving filter, few of its weights survive.
* ``photo``: the same tiling over a slowly varying bright field with small
  coefficients (scale 2, AcMul around 0.5, none beyond DC in 8x32 and 32x8), as
  photographic content has: most blocks reach the filter and most of its
  weights count.
"""
import functools
import math

import numpy as np
import torch

from paper_1908_03565_gb300 import binding

DTYPES = {"u8": (binding.OUT_U8_SRGB, torch.uint8), "f16": (binding.OUT_F16_LINEAR, torch.float16),
          "f32": (binding.OUT_F32_LINEAR, torch.float32)}
NOISE_LUT = tuple((40 + 12 * i) / 1024 for i in range(16))
# width and height in blocks of the DctSelect codes the tilings use
SHAPE8 = {0: (1, 1), 1: (1, 1), 2: (1, 1), 3: (1, 1), 4: (2, 2), 5: (4, 4), 6: (1, 2), 7: (2, 1),
          8: (1, 4), 9: (4, 1), 10: (2, 4), 11: (4, 2)}


def _image(name, width, height, content, out, kind="image", epf=True, gab=True, dct8=False,
           dc_smooth=False, lf_predict=False, qco=False, noise=False):
    return {"name": name, "kind": kind, "width": width, "height": height, "content": content,
            "out": out, "epf": epf, "gab": gab, "dct8": dct8, "dc_smooth": dc_smooth,
            "lf_predict": lf_predict, "qco": qco, "noise": noise}


def listed():
    return [
        # an icon: the smallest requests a server sees, nothing but latency
        _image("icon_u8", 48, 40, "bench", "u8"),
        # one 256x256 group of plain DCT8 without filters, f32 out
        _image("group_f32", 256, 256, "bench", "f32", epf=False, gab=False, dct8=True),
        # one video-sized frame for display, inputs on the device
        _image("hd_u8", 1920, 1088, "bench", "u8"),
        # the same size decoded from host memory back to host memory, as a
        # program does whose entropy decoder runs on the CPU
        _image("hd_host_f32", 1920, 1088, "photo", "f32", kind="host"),
        # a photograph with every step that the format has on by default:
        # DC smoothing, AC prediction, edge-preserving filter, Gaborish
        _image("photo_u8", 3001, 2003, "photo", "u8", dc_smooth=True, lf_predict=True),
        # the benchmark's headline image
        _image("full_f32", 4096, 4096, "bench", "f32"),
        # the transform alone to half floats, as a training pipeline asks for
        _image("plain_f16", 4096, 4096, "photo", "f16", epf=False, gab=False),
        # the optional steps: quantization constraint and noise synthesis
        _image("options_u8", 2047, 1535, "photo", "u8", qco=True, noise=True),
        # the largest side that serving takes
        _image("large_u8", 8192, 8192, "bench", "u8"),
        # a caller without an allocator, on its own stream
        _image("fixed_u8", 1280, 720, "photo", "u8", kind="fixed"),
        # many uneven images in one graph replay, half u8 and half f16
        {"name": "batch_mixed", "kind": "batch", "images": 48, "low": 64, "high": 2048,
         "sizes": 7, "content": "photo"},
        # a JPEG1 stream of the usual subsampling
        {"name": "jpeg420_u8", "kind": "jpeg", "width": 4096, "height": 4096, "sampling": "420",
         "out": "u8"},
    ]


def draw(rng):
    def side(low, high):
        return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))

    kind = rng.choices(["image", "host", "fixed", "batch", "jpeg"], [6, 1, 1, 1, 2])[0]
    if kind == "batch":
        return {"kind": "batch", "images": rng.randint(8, 48), "low": 64,
                "high": side(256, 2048), "sizes": rng.randint(1, 10 ** 6),
                "content": rng.choice(["bench", "photo"])}
    if kind == "jpeg":
        return {"kind": "jpeg", "width": side(48, 6000), "height": side(48, 6000),
                "sampling": rng.choice(["420", "420", "444", "grey"]),
                "out": rng.choice(["u8", "u8", "f32"])}
    out = rng.choice(["u8", "u8", "f32", "f16"])
    # the benchmark's samples leave the range of half floats
    content = "photo" if out == "f16" else rng.choice(["bench", "photo"])
    top = {"image": 8192 if content == "bench" else 4096, "host": 2600, "fixed": 2300}[kind]
    case = _image(None, side(32, top), side(32, top), content, out, kind=kind)
    del case["name"]
    if rng.random() < 0.25:
        case["epf"] = False
        case["gab"] = rng.random() < 0.5
    elif out == "u8" and content == "photo" and kind != "fixed":
        for step in ("dc_smooth", "lf_predict", "qco", "noise"):
            case[step] = rng.random() < 0.3
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _tiling(bw, bh, gen, dct8):
    """The DctSelect map (0xFF on covered blocks) and the block-wise width and
    height, in blocks, of the varblock that owns each block."""
    dev = gen.device
    one = torch.ones((bh, bw), dtype=torch.int64, device=dev)
    if dct8:
        return torch.zeros((bh, bw), dtype=torch.uint8, device=dev), one, one.clone()
    cw, ch = -(-bw // 4), -(-bh // 4)
    by, bx = torch.meshgrid(torch.arange(bh, device=dev), torch.arange(bw, device=dev), indexing="ij")

    def uniform(step):
        r = torch.rand((ch * 4 // step, cw * 4 // step), generator=gen, device=dev)
        return r.repeat_interleave(step, 0).repeat_interleave(step, 1)[:bh, :bw]

    def fits(step):
        return ((bx // step + 1) * step <= bw) & ((by // step + 1) * step <= bh)

    r8, r16, o16, r32, o32 = uniform(1), uniform(2), uniform(2), uniform(4), uniform(4)
    v = torch.zeros((bh, bw), dtype=torch.int64, device=dev)
    w8, h8 = one.clone(), one.clone()

    def put(mask, code):
        w, h = SHAPE8[code]
        at = (bx % w == 0) & (by % h == 0)
        v[mask] = torch.where(at, code, 255)[mask]
        w8[mask], h8[mask] = w, h

    put(r8 >= 2 / 3, 3)
    put(r8 >= 5 / 6, 2)
    put(r8 >= 11 / 12, 1)
    f16, f32 = fits(2), fits(4)
    put(f16 & (r16 < 0.1875), 4)
    put(f16 & (r16 >= 0.1875) & (r16 < 0.25) & (o16 < 0.5), 6)
    put(f16 & (r16 >= 0.1875) & (r16 < 0.25) & (o16 >= 0.5), 7)
    put(f32 & (r32 < 0.10), 5)
    for low, codes in ((0.10, (10, 11)), (0.15, (8, 9))):
        put(f32 & (r32 >= low) & (r32 < low + 0.05) & (o32 < 0.5), codes[0])
        put(f32 & (r32 >= low) & (r32 < low + 0.05) & (o32 >= 0.5), codes[1])
    return v.to(torch.uint8), w8, h8


def _spread(t):
    """Block-wise values to samples."""
    return t.repeat_interleave(8, 0).repeat_interleave(8, 1)


def _make_image(xs, ys, content, seed, dct8=False):
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    dev = gen.device
    bw, bh = -(-xs // 8), -(-ys // 8)
    vmap, w8, h8 = _tiling(bw, bh, gen, dct8)
    bx = torch.arange(bw, device=dev)[None, :]
    by = torch.arange(bh, device=dev)[:, None]
    ox, oy = bx - bx % w8, by - by % h8
    u = torch.arange(8 * bw, device=dev)[None, :] - 8 * _spread(ox)
    v = torch.arange(8 * bh, device=dev)[:, None] - 8 * _spread(oy)
    photo = content == "photo"
    scale = (2.0 if photo else 64.0) / (1.0 + u + v).to(torch.float32)
    if photo:                          # the 8x32 matrices reach far past any photograph's range
        scale = torch.where(_spread(w8 + h8) == 5, 0.0, scale)
    llf = (u < _spread(w8)) & (v < _spread(h8))
    cx, cy = _spread(ox) + u, _spread(oy) + v        # the DC sample of an LLF slot
    coeffs = torch.empty((3, 8 * bh, 8 * bw), dtype=torch.int16, device=dev)
    phase = torch.rand((3, 2), generator=gen, device=dev) * (2 * math.pi)
    for c in range(3):
        r = torch.rand(u.shape, generator=gen, device=dev) - 0.5
        lap = -torch.sign(r) * torch.log1p(-2.0 * r.abs().clamp(max=0.4999999)) * scale
        if photo:
            level, swing = ((0.0, 30.0), (250.0, 120.0), (250.0, 120.0))[c]
            field = level + swing * (torch.sin(2 * math.pi / 48.0 * cx + phase[c, 0])
                                     * torch.cos(2 * math.pi / 48.0 * cy + phase[c, 1]))
            noise = torch.randn(u.shape, generator=gen, device=dev)
            lap = torch.where(llf, field + 0.7 * noise, lap)
        coeffs[c] = lap.round().clamp(-32768, 32767).to(torch.int16)
    low, high = (0.35, 0.7) if photo else (0.5, 4.0)
    field = torch.exp(torch.rand((bh, bw), generator=gen, device=dev) * math.log(high / low)) * low
    acmul = torch.ones((bh, bw), device=dev) if dct8 else field[oy, ox].contiguous()
    cfl = torch.rand((-(-bh // 8), -(-bw // 8), 2), generator=gen, device=dev) - 0.5
    if dct8:
        cfl.zero_()
    elif photo:
        cfl *= 0.2
    sharp = torch.randint(0, 8, (bh, bw), generator=gen, device=dev, dtype=torch.uint8)
    return {"xsize": xs, "ysize": ys, "coeffs": coeffs, "vmap": vmap, "acmul": acmul.to(torch.float32),
            "cfl": cfl.contiguous(), "sharpness": sharp}


def _make_jpeg(xs, ys, sampling, seed):
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    dev = gen.device
    samp = {"420": [(2, 2), (1, 1), (1, 1)], "444": [(1, 1)] * 3, "grey": [(1, 1)]}[sampling]
    top = samp[0][0]
    mx, my = -(-xs // (8 * top)), -(-ys // (8 * top))
    uu, vv = torch.arange(64, device=dev) // 8, torch.arange(64, device=dev) % 8
    comps = []
    for i, (h, v) in enumerate(samp):
        bw, bh = mx * h, my * v
        quant = ((3, 4)[i > 0] + (2, 3)[i > 0] * (uu + vv)).cpu().numpy().astype(np.uint16)
        r = torch.rand((bh, bw, 64), generator=gen, device=dev) - 0.5
        q = -torch.sign(r) * torch.log1p(-2.0 * r.abs().clamp(max=0.4999999)) * (6.0 / (1.0 + uu + vv))
        ph = torch.rand(2, generator=gen, device=dev) * (2 * math.pi)
        by, bx = torch.meshgrid(torch.arange(bh, device=dev), torch.arange(bw, device=dev), indexing="ij")
        q[:, :, 0] = 200.0 * torch.sin(2 * math.pi / 40.0 * bx + ph[0]) * torch.cos(
            2 * math.pi / 40.0 * by + ph[1]) + 2.0 * torch.randn((bh, bw), generator=gen, device=dev)
        comps.append({"coeffs": q.round().clamp(-32768, 32767).to(torch.int16), "quant": quant,
                      "h_samp": h, "v_samp": v})
    return {"xsize": xs, "ysize": ys, "components": comps}


def _sizes(case):
    """Sides of a batch's images: multiples of 8, log-uniform."""
    rng = np.random.default_rng(case["sizes"])
    s = np.exp(rng.uniform(math.log(case["low"]), math.log(case["high"]), size=(case["images"], 2)))
    return [(max(8, 8 * int(round(w / 8))), max(8, 8 * int(round(h / 8)))) for w, h in s]


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _context():
    """A program keeps one context for all of its images."""
    return binding.Context(device=0)


def _params(case):
    p = binding.filter_defaults(epf=int(case["epf"]), gab=int(case["gab"]),
                                dc_smooth=int(case["dc_smooth"]),
                                lf_predict=int(case["lf_predict"]), qco=int(case["qco"]),
                                noise=int(case["noise"]))
    if case["noise"]:
        for i, x in enumerate(NOISE_LUT):
            p.noise_lut[i] = x
    return p


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "ctx": None if kind == "fixed" else _context()}
    if kind == "batch":
        jobs = []
        for i, (w, h) in enumerate(_sizes(case)):
            code, tdt = DTYPES[("u8", "f16")[i % 2]]
            img = _make_image(w, h, case["content"], seed * 1009 + i)
            out = torch.empty((h, w, 3), dtype=tdt, device="cuda")
            jobs.append((img, binding.filter_defaults(epf=1, gab=1), out, code))
        torch.cuda.synchronize()       # the batch runs on its own stream when it is made
        state["out"] = [j[2] for j in jobs]
        state["batch"] = state["ctx"].batch(jobs)
        return state
    state["dtype"], tdt = DTYPES[case["out"]]
    shape = (case["height"], case["width"], 3)
    if kind == "jpeg":
        state["stream"] = _make_jpeg(case["width"], case["height"], case["sampling"], seed)
        state["out"] = torch.empty(shape, dtype=tdt, device="cuda")
        return state
    img = _make_image(case["width"], case["height"], case["content"], seed, case["dct8"])
    state["params"] = _params(case)
    if kind == "host":
        img = {k: t.cpu().pin_memory().numpy() if isinstance(t, torch.Tensor) else t
               for k, t in img.items()}
        state["out"] = torch.empty(shape, dtype=tdt, pin_memory=True).numpy()
    else:
        state["out"] = torch.empty(shape, dtype=tdt, device="cuda")
    state["img"] = img
    return state


def run(state):
    kind, ctx, out = state["kind"], state["ctx"], state["out"]
    if kind == "batch":
        state["batch"].launch(torch.cuda.current_stream().cuda_stream)
    elif kind == "fixed":
        binding.run_noalloc(state["img"], state["params"], out, state["dtype"],
                            stream=torch.cuda.current_stream().cuda_stream)
    elif kind == "jpeg":
        ctx.poll(ctx.submit_jpeg(state["stream"], out, state["dtype"]))
    else:
        device = kind == "image"
        ctx.poll(ctx.submit(state["img"], state["params"], out, state["dtype"], on_device=device,
                            out_on_device=device))
    return out


def _image_work(width, height, content, out, epf=True, gab=True, lf=False, qco=False, noise=False):
    padded = (-(-width // 8) * 8) * (-(-height // 8) * 8)
    pixels = width * height
    # coefficients, map + quant field + sharpness per block, factors per tile, output
    nbytes = padded * (6 + (5 + epf) / 64 + 8 / 4096) + pixels * 3 * {"u8": 1, "f16": 2, "f32": 4}[out]
    # per pixel: dequantisation 21, transforms 54, colour 20; Gaborish 27;
    # the filter 456 on the blocks that reach it, its guide 17
    flops = pixels * (95 + 27 * gab + epf * (17 + 456 * (0.6 if content == "photo" else 0.4)))
    flops += pixels * (3 * lf + 108 * qco + 40 * noise)
    return nbytes, flops


def work(case):
    if case["kind"] == "batch":
        parts = [_image_work(w, h, case["content"], ("u8", "f16")[i % 2])
                 for i, (w, h) in enumerate(_sizes(case))]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if case["kind"] == "jpeg":
        pixels = case["width"] * case["height"]
        samples = pixels * {"420": 1.5, "444": 3, "grey": 1}[case["sampling"]]
        return {"bytes": 2 * samples + pixels * 3 * {"u8": 1, "f32": 4}[case["out"]],
                "flops": 11 * samples + 14 * pixels}
    nbytes, flops = _image_work(case["width"], case["height"], case["content"], case["out"],
                                case["epf"], case["gab"], case["dc_smooth"] or case["lf_predict"],
                                case["qco"], case["noise"])
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# 64-bit results (floating outputs; bytes have to be equal and need none)
# ---------------------------------------------------------------------------
# C.6.1.1: distance bands per channel of the DCT shapes by (short, long) side,
# with eccentricity bands for 8 x 32
BANDS = {
    (8, 8): ((5.0, 0.0, -0.4, -0.4, -0.4, -2.0), (1.1, 0.0, -0.3, -0.3, -0.3, -0.3),
             (1.0, -3.0, 0.0, 0.0, -1.0, -2.0)),
    (4, 4): ((32.0, -0.4, 0.0, 0.0), (6.0, 0.0, 0.0, 0.0), (4.0, -5.0, -1.0, -1.0)),
    (16, 16): ((3.1965020925735868, -1.8000777393353804, -0.39424529824571225,
                -0.33909377445710343, -0.6350101832695744, -0.90177264050827612,
                -1.5162099239887414),
               (0.77917081615440487, -0.57424582104194355, -0.90745813428471001,
                -0.64925837484843441, -0.35865440981033403, -0.21322389111877305,
                -0.27615025315725483),
               (0.22259376988644336, -3.0531423165804414, -0.2, -0.30687130033378396,
                -0.42708730624733904, -1.4856834539296244, -5.9209142884401604)),
    (32, 32): ((0.47968775359573942, -1.025, -0.98, -0.9012, -0.4, -0.48819395464, -0.421064,
                -0.27),
               (0.22295421389982905, -0.8041958212306401, -0.7633036457487539,
                -0.55660379990111464, -0.49785304658857626, -0.43699592683512467,
                -0.40180866526242109, -0.27321683125358037),
               (0.11607457694128877, -3.060733579805728, -2.0413270132490346,
                -2.0235650159727417, -0.5495389509954993, -0.4, -0.4, -0.3)),
    (8, 16): ((5.0, -0.7, -0.7, -0.2, -0.2, -0.2, -0.5), (1.0, -0.5, -0.5, -0.5, -0.2, -0.2, -0.2),
              (0.35, -1.4, -0.2, -0.5, -0.5, -1.5, -3.6)),
    (8, 32): ((0.90897201669289496, -2.523575079652864, 1.5606102630460328, -0.6828050717528521,
               -14.770016895841904, -31.365240527393656, 0.565929254166433, 26.789646874558219),
              (0.3603042187746216, -0.11724474917749789, -0.85426302204085935, -0.5404181207241352,
               -0.45637619443533173, -0.82707923060149569, -1.09760551067614, -54.16057009483842),
              (0.25176400522276937, -10.060949304689093, -4.5316627381323995, -5.4569229849460807,
               -10.549754675878864, 1.7512906265092971, -1.6854706115725824, 3.3092762331901451)),
    (16, 32): ((1.1280371559733287, -0.98868, -0.658, -0.42026, -0.22712, -0.2206, -0.226, -0.2),
               (0.38961075971152237, -0.62525308982767058, -0.83770786552491361,
                -0.79014862079498627, -0.2692727459704829, -0.38272769465388551,
                -0.2292422253091453, -0.20719098826199578),
               (0.098, -2.41, -0.23, -0.2, -0.4, -0.8, -0.4, -0.5)),
}
ECCENTRICITY = {(8, 32): ((-0.40751133465833289, 2.2055690721475925, -1.4434547377534228,
                           2.0590289434445102),
                          (0.12452072219659419, 0.065578935001406033, -0.14598888885596958,
                           0.12114139909222557),
                          (0.0586589025020419, -2.2654958780302183, -4.6996221931893647,
                           1.8254498073137184))}
IDENTITY_WEIGHTS = ((221.50801256717435, 7087.151589594002, 4466.9924939259863),
                    (29.535505378287006, 1454.6663024982124, 1368.041230099175),
                    (9.2887405354132238, 23.982311358829531, 11.201853748207084))
DCT2_WEIGHTS = ((3840.0, 2560.0, 1280.0, 640.0, 480.0, 300.0),
                (960.0, 640.0, 320.0, 180.0, 140.0, 120.0),
                (640.0, 320.0, 128.0, 64.0, 32.0, 16.0))
DCT4_DIVISORS = ((1.0, 1.0), (0.7, 0.7), (1.0, 1.0))
ONE_BIAS = (0.05465007330715401, 0.07005449891748593, 0.049935103337343655)
M_DC = tuple(x / (64.0 * math.sqrt(2.0)) for x in (0.02, 0.2, 0.2))
EPF_SCALE = (899.676941, 111.965157, 45.275791)
GAB_W = (0.115169525, 0.061248592)
OPSIN = ((2542.56835937500000, -2326.53173828125000, 44.17734527587891),
         (-698.04852294921875, 1012.71777343750000, -76.22974395751953),
         (-827.36480712890625, 709.83502197265625, 451.38488769531250))
OPSIN_BIAS = (-0.00100549, -0.00100549, -0.00094081)


def _bands(first, rest):
    out = [first]
    for x in rest:
        out.append(out[-1] * (x + 1.0 if x > 0 else 1.0 / (1.0 - x)))
    return out


def _between(pos, top, bands):
    at = pos * (len(bands) - 1) / top
    i = int(math.floor(at))
    if i >= len(bands) - 1:
        return bands[-1]
    return bands[i] * (bands[i + 1] / bands[i]) ** (at - i)


def _band_weights(w, h, c):
    key = (min(w, h), max(w, h))
    dist = _bands(BANDS[key][c][0], BANDS[key][c][1:])
    ecc = _bands(1.0, ECCENTRICITY[key][c]) if key in ECCENTRICITY else [1.0, 1.0]
    out = np.zeros((h, w))
    for y in range(h):
        for x in range(w):
            d = math.hypot(x / w, y / h)
            e = abs(x / w - y / h) / d if d > 0 else 0.0
            out[y, x] = _between(d, math.sqrt(2.0), dist) * _between(e, 1.0, ecc)
    return out


def _axis_scale(n, k):
    """The factor of frequency k that a dimension of n samples gives the
    numerators of C.6.1 (I of I.2.6.1)."""
    i8 = math.sqrt(2.0 / n) * (math.sqrt(0.5) if k == 0 else 1.0) * math.cos(k * math.pi / (2 * n))
    return i8 if n == 8 else 1.0 / (n * i8)


@functools.lru_cache(maxsize=None)
def _matrices(code):
    """C.6.1 dequantisation matrices of a code, (3, h, w)."""
    w, h = (8 * s for s in SHAPE8[code])
    out = np.ones((3, h, w))
    for c in range(3):
        if code == 1:
            wt = np.full((8, 8), IDENTITY_WEIGHTS[c][0])
            wt[0, 1] = wt[1, 0] = IDENTITY_WEIGHTS[c][1]
            wt[1, 1] = IDENTITY_WEIGHTS[c][2]
            out[c] = 1.0 / wt
        elif code == 2:
            wt, p = np.ones((8, 8)), DCT2_WEIGHTS[c]
            for k, s in enumerate((1, 2, 4)):
                wt[:s, s:2 * s] = wt[s:2 * s, :s] = p[2 * k]
                wt[s:2 * s, s:2 * s] = p[2 * k + 1]
            out[c] = 1.0 / wt
        elif code == 3:
            wt = np.kron(_band_weights(4, 4, c), np.ones((2, 2)))
            wt[0, 1] /= DCT4_DIVISORS[c][0]
            wt[1, 0] /= DCT4_DIVISORS[c][0]
            wt[1, 1] /= DCT4_DIVISORS[c][1]
            n4 = np.array([_axis_scale(4, k // 2) for k in range(8)])
            out[c] = np.outer(n4, n4) / 64.0 / wt
        else:
            nx = np.array([_axis_scale(w, k) for k in range(w)])
            ny = np.array([_axis_scale(h, k) for k in range(h)])
            out[c] = np.outer(ny, nx) / (w * h) / _band_weights(w, h, c)
    return out


def _idct(n):
    """The draft's inverse transform of n points: samples from frequencies."""
    k, t = np.arange(n)[None, :], np.arange(n)[:, None]
    scale = 1.0 / np.cos(k * math.pi / 16.0) if n == 8 else 2.0 * np.cos(k * math.pi / (2.0 * n))
    return np.where(k == 0, 1.0, scale) * np.cos((2 * t + 1) * k * math.pi / (2.0 * n))


def _corner(b, s):
    """One 2x2 Hadamard level on the top-left s x s of b (..., 8, 8)."""
    h, out = s // 2, b.copy()
    p, q, r, t = b[..., :h, :h], b[..., :h, h:s], b[..., h:s, :h], b[..., h:s, h:s]
    out[..., 0:s:2, 0:s:2], out[..., 0:s:2, 1:s:2] = p + q + r + t, p + q - r - t
    out[..., 1:s:2, 0:s:2], out[..., 1:s:2, 1:s:2] = p - q + r - t, p - q - r + t
    return out


@functools.lru_cache(maxsize=None)
def _operator(code):
    """The 64 x 64 operator (samples from coefficients) of codes 1, 2, 3."""
    b = np.eye(64).reshape(64, 8, 8)
    if code == 2:
        return _corner(_corner(_corner(b, 2), 4), 8).reshape(64, 64).T.copy()
    dc, out = _corner(b, 2), np.zeros((64, 8, 8))
    for y in range(2):
        for x in range(2):
            q = b[:, y::2, x::2].copy()
            if code == 3:
                q[:, 0, 0] = dc[:, y, x]
                s = _idct(4) @ q @ _idct(4).T
            else:
                q[:, 0, 0] = 0.0
                mid = (dc[:, y, x] - q.sum((1, 2)) / 16.0)[:, None, None]
                q[:, 0, 0] = q[:, 1, 1]
                q[:, 1, 1] = 0.0
                s = q + mid
            out[:, 4 * y:4 * y + 4, 4 * x:4 * x + 4] = s
    return out.reshape(64, 64).T.copy()


@functools.lru_cache(maxsize=None)
def _llf_from_dc(w8, h8):
    """I.2.7: the inverse of the 8x8 means of the LLF-only reconstruction."""
    means = np.zeros((w8 * h8, w8 * h8))
    for j in range(w8 * h8):
        col = _idct(8 * h8)[:, j // w8].reshape(h8, 8).mean(1)
        row = _idct(8 * w8)[:, j % w8].reshape(w8, 8).mean(1)
        means[:, j] = np.outer(col, row).reshape(-1)
    return np.linalg.inv(means)


def _f64(a, like):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=like.device)


def _exact_xyb(img):
    co, vmap = img["coeffs"], img["vmap"]
    out = torch.zeros(co.shape, dtype=torch.float64, device=co.device)
    for code, (w8, h8) in SHAPE8.items():
        by, bx = torch.nonzero(vmap == code, as_tuple=True)
        if not len(by):
            continue
        w, h = 8 * w8, 8 * h8
        rows = (8 * by)[:, None, None] + torch.arange(h, device=co.device)[None, :, None]
        cols = (8 * bx)[:, None, None] + torch.arange(w, device=co.device)[None, None, :]
        q = co[:, rows, cols].to(torch.float64)                       # 3, n, h, w
        one = 1.0 - _f64(ONE_BIAS, co)[:, None, None, None]
        b = torch.where(q.abs() <= 1, q * one, q - 0.145 / torch.where(q == 0, 1.0, q))
        b = b * img["acmul"][by, bx].to(torch.float64)[:, None, None]
        b = b * _f64(_matrices(code), co)[:, None]
        k = img["cfl"][by // 8, bx // 8].to(torch.float64)            # n, 2
        b[0] += k[:, 0, None, None] * b[1]
        b[2] += k[:, 1, None, None] * b[1]
        dc = q[:, :, :h8, :w8].reshape(3, -1, w8 * h8) * _f64(M_DC, co)[:, None, None]
        b[:, :, :h8, :w8] = (dc @ _f64(_llf_from_dc(w8, h8), co).T).reshape(3, -1, h8, w8)
        if code in (1, 2, 3):
            s = (b.reshape(3, -1, 64) @ _f64(_operator(code), co).T).reshape(b.shape)
        else:
            s = _f64(_idct(h), co) @ b @ _f64(_idct(w), co).T
        out[:, rows, cols] = s
    return out


def _weight_bits(sad, mul4):
    return (((min(sad, 507) << 6) * mul4 >> 18) + (127 << 7)) << 16


@functools.lru_cache(maxsize=None)
def _mul_table():
    """4 * mul of J.2.4 for sigma 0 .. 672: for every fourth sigma the first
    mul whose weight at sad = sigma / 4 is above 0.5, linear between."""
    tab, mul, half = [0] * 673, -32768, 0x3F000000
    for s in range(16, 673, 4):
        while mul < 0 and _weight_bits(s >> 2, 4 * mul) <= half:
            mul += 1
        tab[s] = 4 * mul
    for s in range(16, 672, 4):
        for i in range(1, 4):
            tab[s + i] = tab[s] + i * ((tab[s + 4] - tab[s]) // 4)
    return tab


def _mirrored(t, pad):
    """t (..., h, w) with pad samples mirrored on each side (6.5)."""
    for d in (-1, -2):
        n = t.shape[d]
        i = torch.arange(-pad, n + pad, device=t.device)
        i = i % (2 * n)
        t = t.index_select(d, torch.where(i >= n, 2 * n - 1 - i, i))
    return t


def _exact_epf(xyb, img):
    ys, xs = xyb.shape[1:]
    bh, bw = -(-ys // 8), -(-xs // 8)
    scaled = xyb.clone()
    scaled[0] += 0.03
    scaled *= _f64(EPF_SCALE, xyb)[:, None, None]
    # range of each block over its in-image samples, then of its varblock
    grow = (0, 8 * bw - xs, 0, 8 * bh - ys)
    hi = torch.nn.functional.pad(scaled, grow, value=-math.inf)
    lo = torch.nn.functional.pad(scaled, grow, value=math.inf)
    r = (hi.reshape(3, bh, 8, bw, 8).amax((2, 4)) - lo.reshape(3, bh, 8, bw, 8).amin((2, 4))).amax(0)
    rng = r.clone()
    for code, (w8, h8) in SHAPE8.items():
        by, bx = torch.nonzero(img["vmap"] == code, as_tuple=True)
        if len(by) and w8 * h8 > 1:
            rows = by[:, None, None] + torch.arange(h8, device=r.device)[None, :, None]
            cols = bx[:, None, None] + torch.arange(w8, device=r.device)[None, None, :]
            rng[rows, cols] = r[rows, cols].amax((1, 2), keepdim=True).expand(-1, h8, w8)
    sigma = rng.clamp(max=70.0) * 12.6 * (img["sharpness"].to(torch.float64) / 7.0)
    sigma = torch.minimum(sigma, 20.0 / img["acmul"].to(torch.float64)).clamp(max=170.0).floor().long()
    on = _spread(sigma >= 16)[:ys, :xs]
    mul4 = torch.tensor(_mul_table(), device=xyb.device)[sigma.clamp(16, 672)]
    mul4 = _spread(mul4)[:ys, :xs]
    guide = _mirrored(scaled.clamp(0.0, 255.0).to(torch.int16), 8)
    samples = _mirrored(xyb, 8)
    num, den = torch.zeros_like(xyb), torch.zeros_like(xyb[0])
    near = guide[:, 4:-4, 4:-4]                                       # 4 samples around the image
    for dy in range(-3, 4):
        for dx in range(-3, 5):
            far = guide[:, 4 + dy:guide.shape[1] - 4 + dy, 4 + dx:guide.shape[2] - 4 + dx]
            d = (near - far).abs().sum(0, dtype=torch.int32)
            d = d[3:3 + ys] + d[4:4 + ys] + d[5:5 + ys]
            sad = d[:, 3:3 + xs] + d[:, 4:4 + xs] + d[:, 5:5 + xs] + d[:, 6:6 + xs]
            bits = (((sad.clamp(max=507).long() << 6) * mul4 >> 18) + (127 << 7)) << 16
            wt = bits.to(torch.int32).view(torch.float32)
            wt = torch.where(wt < np.float32(0.3).item(), 0.0, wt).to(torch.float64)
            den += wt
            num += wt * samples[:, 8 + dy:8 + dy + ys, 8 + dx:8 + dx + xs]
    return torch.where(on, num / den, xyb)


def _exact_image(img, epf, gab):
    """Linear RGB divided by 255, (ys, xs, 3)."""
    xyb = _exact_xyb(img)[:, :img["ysize"], :img["xsize"]].contiguous()
    if epf:
        xyb = _exact_epf(xyb, img)
    if gab:
        ys, xs = xyb.shape[1:]
        p, (w1, w2) = _mirrored(xyb, 1), GAB_W
        out = torch.zeros_like(xyb)
        for dy in range(3):
            for dx in range(3):
                wt = (1.0, w1, w2)[abs(dy - 1) + abs(dx - 1)] / (1.0 + 4 * w1 + 4 * w2)
                out += wt * p[:, dy:dy + ys, dx:dx + xs]
        xyb = out
    mix = torch.stack([xyb[1] + xyb[0], xyb[1] - xyb[0], xyb[2]]) ** 3
    mix += _f64(OPSIN_BIAS, xyb)[:, None, None]
    return torch.einsum("rk,khw->hwr", _f64(OPSIN, xyb), mix) / 255.0


def _exact_jpeg(stream):
    """M.6 without side channels: samples / 255, (ys, xs, 3)."""
    planes, comps = [], stream["components"]
    basis = np.cos((2 * np.arange(8)[:, None] + 1) * np.arange(8)[None, :] * math.pi / 16.0) / 2.0
    basis[:, 0] *= math.sqrt(0.5)
    for c in comps:
        q = c["coeffs"]
        b = q.to(torch.float64) * _f64(c["quant"].astype(np.float64), q)
        m = _f64(basis, q)
        s = m @ b.reshape(*q.shape[:2], 8, 8) @ m.T
        p = s.permute(0, 2, 1, 3).reshape(8 * q.shape[0], 8 * q.shape[1])
        if c["h_samp"] != comps[0]["h_samp"]:
            for d in (1, 0):
                n = p.shape[d]
                i = torch.arange(n, device=p.device)
                prev = p.index_select(d, (i - 1).abs())
                after = p.index_select(d, torch.where(i == n - 1, max(n - 2, 0), i + 1))
                pair = torch.stack([0.75 * p + 0.25 * prev, 0.75 * p + 0.25 * after], d + 1)
                p = pair.reshape([2 * n if k == d else p.shape[k] for k in (0, 1)])
        planes.append(p[:stream["ysize"], :stream["xsize"]])
    y = planes[0] + 128.0
    if len(planes) == 1:
        return torch.stack([y, y, y], -1) / 255.0
    cb, cr = planes[1:]
    return torch.stack([y + 1.402 * cr, y - 0.34414 * cb - 0.71414 * cr, y + 1.772 * cb], -1) / 255.0


def _as_half(t):
    """Values past the largest half float become infinite, as in the output."""
    return torch.where(t.abs() >= 65520.0, torch.sign(t) * math.inf, t)


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for i, (w, h) in enumerate(_sizes(case)):
            img = _make_image(w, h, case["content"], seed * 1009 + i) if i % 2 else None
            out.append(_as_half(_exact_image(img, True, True)) if i % 2 else None)
        return out
    if case["out"] == "u8":
        return None                    # bytes: equal or wrong
    if case["kind"] == "jpeg":
        return _exact_jpeg(_make_jpeg(case["width"], case["height"], case["sampling"], seed))
    img = _make_image(case["width"], case["height"], case["content"], seed, case["dct8"])
    rgb = _exact_image(img, case["epf"], case["gab"])
    return _as_half(rgb) if case["out"] == "f16" else rgb
