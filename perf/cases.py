"""Workloads of the wavelet codec through its public entry points (package paper_2405_12631_gb300).

A case is a dict of plain values; its "kind" selects the call:

  decode   streams of one size -> images (Codec.decode_batch and its device / page-locked forms)
  ragged   streams of different sizes -> images, in one call (Codec.decode_ragged)
  gop      one GOP container -> frames (Codec.decode_gop_into)
  serve    a burst of requests of mixed sizes through a Server, submitted and collected
  encode   images of one size -> streams (Codec.encode_batch)

The contexts and models are kept between states, as a program that decodes many streams keeps
them: one context per precision class and model. Weights are seeded random-init ones (the
architecture's stand-in for a trained model, always the same); images and with them the
streams come from the seed.
"""
import functools
import math
import random

import numpy as np
import torch

import paper_2405_12631_gb300 as pw

DEV = "cuda"


# ---- cases -------------------------------------------------------------------
def listed():
    return [
        # The smallest call: one gray image in the plain FP32 class; launches and the coder's
        # serial chains are all there is.
        dict(name="gray256_fp32", kind="decode", prec="fp32", C=32, levels=4, ll=0, count=1,
             h=256, w=256, ch=1, bits=8, lossless=False, q=8.0, where="host"),
        # One photo (768x512 RGB) for a viewer: latency of a single image in the fastest class.
        dict(name="photo_fp8", kind="decode", prec="fp8", C=64, levels=4, ll=0, count=1,
             h=512, w=768, ch=3, bits=8, lossless=False, q=8.0, where="host"),
        # The throughput workload: 24 photos per call, streams and images in device memory.
        dict(name="batch24_fp8", kind="decode", prec="fp8", C=64, levels=4, ll=0, count=24,
             h=512, w=768, ch=3, bits=8, lossless=False, q=16.0, where="device"),
        # The same batch in the BF16 class from and to page-locked host memory.
        dict(name="batch24_bf16_pinned", kind="decode", prec="bf16", C=64, levels=4, ll=0,
             count=24, h=512, w=768, ch=3, bits=8, lossless=False, q=4.0, where="pinned"),
        # An archive scan of odd size: one large gray image, latency at full width.
        dict(name="scan_odd_bf16", kind="decode", prec="bf16", C=64, levels=4, ll=0, count=1,
             h=1365, w=2047, ch=1, bits=8, lossless=False, q=8.0, where="host"),
        # A thumbnail sheet of a mixed album: RGB images of similar, odd sizes in one call.
        dict(name="album_ragged_fp8", kind="ragged", prec="fp8", C=64, levels=4, ll=0, count=12,
             h=700, w=960, ch=3, bits=8, lossless=False, q=8.0, mix=3),
        # Medical / scientific archive: 12-bit lossless 4K RGB, five levels (the largest call).
        dict(name="lossless4k_fp8", kind="decode", prec="fp8", C=64, levels=5, ll=0, count=2,
             h=2160, w=3840, ch=3, bits=12, lossless=True, q=1.0, where="pinned"),
        # Portable streams: the integer-network class with the autoregressive LL model.
        dict(name="portable_int8_arll", kind="decode", prec="int8", C=32, levels=4, ll=1,
             count=1, h=384, w=512, ch=1, bits=8, lossless=False, q=8.0, where="host"),
        # Video playback: one 8-frame GOP of 1920x1080 RGB with motion compensation.
        dict(name="gop1080p_bf16", kind="gop", prec="bf16", C=64, levels=4, ll=0, count=8,
             h=1080, w=1920, ch=3, bits=8, lossless=False, q=8.0),
        # A decode service: a burst of requests of mixed sizes, gray and RGB.
        dict(name="serve_burst_fp8", kind="serve", prec="fp8", C=64, levels=4, ll=0, count=16,
             h=2048, w=2048, ch=3, bits=8, lossless=False, q=8.0, mix=7),
        # Ingest: a batch of photos encoded from host memory to streams.
        dict(name="encode_batch_fp8", kind="encode", prec="fp8", C=64, levels=4, ll=0, count=12,
             h=512, w=768, ch=3, bits=8, lossless=False, q=8.0),
        # Ingest of one small gray image in the plain class, lossless.
        dict(name="encode_gray_lossless", kind="encode", prec="fp32", C=32, levels=4, ll=0,
             count=1, h=250, w=333, ch=1, bits=8, lossless=True, q=1.0),
    ]


def draw(rng):
    """One more case: kinds, classes and sizes spread over the ranges above."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["decode", "decode", "decode", "ragged", "gop", "serve", "encode"])
    prec = rng.choice(["fp8", "fp8", "bf16", "fp32", "int8"] if kind in ("decode", "encode")
                      else ["fp8", "bf16"])
    slow = prec in ("fp32", "int8")       # the SIMT classes: small calls
    case = dict(kind=kind, prec=prec, C=rng.choice([32, 64]), levels=4, ll=0,
                count=1, h=log(48, 640 if slow else 2048), w=log(48, 640 if slow else 2048),
                ch=rng.choice([1, 3]), bits=8, lossless=False, q=rng.choice([4.0, 8.0, 16.0, 32.0]))
    if kind in ("decode", "encode"):
        case["ll"] = rng.choice([0, 0, 0, 1]) if case["h"] * case["w"] < 400000 else 0
        if rng.random() < 0.2:
            case.update(lossless=True, q=1.0, bits=rng.choice([8, 12]))
        room = (400_000 if slow else 12_000_000) // (case["h"] * case["w"] * case["ch"])
        case["count"] = max(1, min(24, log(1, max(1, room))))
        if kind == "decode":
            case["where"] = rng.choice(["host", "device", "pinned"])
    elif kind == "ragged":
        case.update(h=log(96, 1024), w=log(96, 1024), mix=rng.randrange(1000))
        case["count"] = max(2, min(24, log(2, max(2, 9_000_000 // (case["h"] * case["w"] * case["ch"])))))
    elif kind == "gop":
        case.update(count=rng.choice([2, 4, 8]), h=log(128, 1080), w=log(128, 1920))
    else:
        case.update(h=2048, w=2048, ch=3, count=log(4, 16), mix=rng.randrange(1000))
        while sum(h * w * c for h, w, c, _ in _sizes(case)) > 40_000_000:
            case["count"] -= 1
    return case


def _sizes(case):
    """(h, w, channels, q) of every image of a call."""
    n = case["count"]
    if case["kind"] == "ragged":
        r = random.Random(case["mix"])
        return [(max(16, int(case["h"] * r.uniform(0.86, 1.0))),
                 max(16, int(case["w"] * r.uniform(0.86, 1.0))), case["ch"], case["q"])
                for _ in range(n)]
    if case["kind"] == "serve":
        r = random.Random(case["mix"])

        def side(top):
            return max(16, int(math.exp(r.uniform(math.log(top / 8), math.log(top)))) // 16 * 16)
        return [(side(case["h"]), side(case["w"]), r.choice([1, 3]), r.choice([4.0, 8.0, 16.0, 32.0]))
                for _ in range(n)]
    return [(case["h"], case["w"], case["ch"], case["q"])] * n


# ---- images --------------------------------------------------------------------
def _texture(gen, h, w, std):
    """1/f texture."""
    f = torch.sqrt(torch.fft.fftfreq(h, device=DEV)[:, None] ** 2
                   + torch.fft.rfftfreq(w, device=DEV)[None, :] ** 2)
    f[0, 0] = 1.0
    s = torch.fft.rfft2(torch.randn(h, w, generator=gen, device=DEV)) / f
    s[0, 0] = 0.0
    t = torch.fft.irfft2(s, s=(h, w))
    return t * (std / t.std().clamp_min(1e-9))


def _natural(gen, rng, h, w, ch, top=255.0):
    """Float image [h, w, ch]: gradients, rectangles, 1/f texture."""
    yy = torch.linspace(0, 1, h, device=DEV)[:, None]
    xx = torch.linspace(0, 1, w, device=DEV)[None, :]
    img = torch.empty(h, w, ch, device=DEV)
    for c in range(ch):
        a, lo, hi = rng.uniform(0, 2 * math.pi), rng.uniform(0, top), rng.uniform(0, top)
        t = math.cos(a) * xx + math.sin(a) * yy
        img[:, :, c] = lo + (hi - lo) * (t - t.min()) / (t.max() - t.min()).clamp_min(1e-9)
    for _ in range(rng.randint(6, 20)):
        y, x = rng.randrange(h), rng.randrange(w)
        img[y:y + rng.randint(h // 16 + 1, h // 3 + 1), x:x + rng.randint(w // 16 + 1, w // 3 + 1)] = \
            torch.tensor([rng.uniform(0, top) for _ in range(ch)], device=DEV)
    return img + _texture(gen, h, w, top * 12.0 / 255.0)[:, :, None]


def _finish(img, bits):
    a = img.round().clamp(0, (1 << bits) - 1).cpu().numpy().astype(np.uint8 if bits <= 8 else np.uint16)
    return np.ascontiguousarray(a[:, :, 0] if a.shape[2] == 1 else a)


def _image(seed, k, h, w, ch, bits):
    rng = random.Random(seed * 1009 + k)
    gen = torch.Generator(device=DEV).manual_seed(rng.randrange(1 << 31))
    if bits <= 8:
        return _finish(_natural(gen, rng, h, w, ch), bits)
    # smooth blobs and noise on a mid-grey background
    top = (1 << bits) - 1
    yy, xx = torch.arange(h, device=DEV).float(), torch.arange(w, device=DEV).float()
    n = rng.randint(20, 60)
    s = torch.tensor([rng.uniform(20, 400) for _ in range(n)], device=DEV)
    cy = torch.tensor([rng.uniform(0, h) for _ in range(n)], device=DEV)
    cx = torch.tensor([rng.uniform(0, w) for _ in range(n)], device=DEV)
    gy = torch.exp(-0.5 * ((yy[:, None] - cy) / s) ** 2)
    gx = torch.exp(-0.5 * ((xx[:, None] - cx) / s) ** 2)
    amp = torch.tensor([[rng.uniform(-0.25, 0.5) * top for _ in range(n)] for _ in range(ch)], device=DEV)
    img = torch.stack([(gy * a) @ gx.T for a in amp], dim=2) + top / 4.0
    return _finish(img + 15.0 * torch.randn(h, w, ch, generator=gen, device=DEV), bits)


def _frames(seed, n, h, w, ch):
    """A panned canvas with moving sprites."""
    rng = random.Random(seed * 1009 + 5)
    gen = torch.Generator(device=DEV).manual_seed(rng.randrange(1 << 31))
    pad = 4 * n + 8
    base = _natural(gen, rng, h + 2 * pad, w + 2 * pad, ch)
    spr = [(rng.randrange(h), rng.randrange(w), rng.randint(h // 20 + 2, h // 6 + 2),
            rng.randint(w // 20 + 2, w // 6 + 2), rng.randint(-6, 6), rng.randint(-6, 6),
            torch.tensor([rng.uniform(0, 255) for _ in range(ch)], device=DEV)) for _ in range(4)]
    oy = ox = pad
    out = []
    for f in range(n):
        fr = base[oy:oy + h, ox:ox + w].clone()
        for y, x, hh, ww, vy, vx, col in spr:
            y0, x0 = y + f * vy, x + f * vx
            fr[max(y0, 0):max(y0 + hh, 0), max(x0, 0):max(x0 + ww, 0)] = col
        out.append(_finish(fr, 8))
        oy += rng.randint(-4, 4)
        ox += rng.randint(-4, 4)
    return np.stack(out)


# ---- contexts and models ---------------------------------------------------------
@functools.lru_cache(maxsize=2)
def _codec(prec, C, levels, ll):
    codec = pw.Codec(0, prec)
    return codec, codec.init_random_model(levels, C, 16, ll, seed=0)


@functools.lru_cache(maxsize=1)
def _gop_models(prec, C, levels, ll):
    codec, low = _codec(prec, C, levels, ll)
    return codec, low, codec.init_random_model(levels, C, 16, ll, seed=1)


@functools.lru_cache(maxsize=1)
def _server(prec, C, levels, ll):
    codec, model = _codec(prec, C, levels, ll)
    return pw.Server(codec, model, hbm_budget=100 << 30, lanes=8, max_batch=8)


def _pinned(data):
    return torch.frombuffer(bytearray(data), dtype=torch.uint8).pin_memory()


# ---- prepare and run ---------------------------------------------------------------
def prepare(case, seed):
    kind, key = case["kind"], (case["prec"], case["C"], case["levels"], case["ll"])
    codec, model = _codec(*key)
    st = dict(kind=kind, codec=codec, model=model, case=case)
    if kind == "gop":
        codec, low, high = _gop_models(*key)
        frames = _frames(seed, case["count"], case["h"], case["w"], case["ch"])
        st.update(codec=codec, low=low, high=high, shape=frames.shape[1:],
                  stream=codec.encode_gop(low, high, frames, q=case["q"]),
                  out=torch.empty(frames.shape, dtype=torch.uint8).pin_memory())
        return st
    sizes = _sizes(case)
    imgs = [_image(seed, k, h, w, ch, case["bits"]) for k, (h, w, ch, _) in enumerate(sizes)]
    if kind == "encode":
        # the archive buffer that the streams are written to (with their lengths), one row each
        room = max(im.nbytes for im in imgs) * 2 + 65536
        st.update(imgs=imgs, out=np.zeros((len(imgs), room), dtype=np.uint8))
        return st
    opts = dict(lossless=case["lossless"], bitdepth=case["bits"])
    if kind == "decode":
        streams = codec.encode_batch(model, imgs, q=case["q"], **opts)
        st["shape"] = imgs[0].shape
        if case["where"] != "host":
            dtype = torch.uint8 if case["bits"] <= 8 else torch.int16   # 12-bit samples
            out = torch.zeros((len(imgs),) + imgs[0].shape, dtype=dtype)
            if case["where"] == "device":
                st["bufs"] = [_pinned(s).to(DEV) for s in streams]
                st["out"] = out.to(DEV)
            else:
                st["bufs"] = [_pinned(s) for s in streams]
                st["out"] = out.pin_memory()
    else:
        streams = [codec.encode_image(model, im, q=q, **opts)
                   for im, (_, _, _, q) in zip(imgs, sizes)]
        if kind == "serve":
            st["server"] = _server(*key)
    st["streams"] = streams
    return st


def run(st):
    kind, case, codec, model = st["kind"], st["case"], st["codec"], st["model"]
    if kind == "encode":
        got = codec.encode_batch(model, st["imgs"], q=case["q"], lossless=case["lossless"],
                                 bitdepth=case["bits"])
        for row, s in zip(st["out"], got):
            row[:len(s)] = np.frombuffer(s, dtype=np.uint8)
        return st["out"], np.array([len(s) for s in got])
    if kind == "ragged":
        return codec.decode_ragged(model, st["streams"])
    if kind == "gop":
        codec.decode_gop_into(st["low"], st["high"], st["stream"], case["count"], st["shape"],
                              st["out"].data_ptr())
        return st["out"]
    if kind == "serve":
        server = st["server"]
        tickets = [server.submit(s) for s in st["streams"]]
        return [server.poll(t) for t in tickets]
    if case["where"] == "host":
        got = codec.decode_batch(model, st["streams"])
        return got if got.dtype == np.uint8 else got.view(np.int16)
    ptrs, lens = [b.data_ptr() for b in st["bufs"]], [b.numel() for b in st["bufs"]]
    call = codec.decode_batch_device if case["where"] == "device" else codec.decode_batch_host_ptrs
    call(model, ptrs, lens, st["out"].data_ptr(), st["shape"], case["bits"])
    return st["out"].numpy() if case["where"] == "pinned" else st["out"]


def work(case):
    """Samples in or out and their stream once; the context nets after their linear layers are
    merged, each output computed only where it is used, and the lifting CNNs."""
    C = case["C"]
    n = sum(h * w * ch for h, w, ch, _ in _sizes(case))
    gates = 2 * 9 * (C + 10) * 4 * C
    step1 = 2 * C * C + (2 * 9 * C + 12 * C * C) / 4
    steps = 3 * (2 * (C + 9) * C + 18 * C * C + 18 * C * C / 4)
    lifting = 2 * 5184 * 4 / 3
    temporal = 5184 * 2 * (1 - 1 / case["count"]) if case["kind"] == "gop" else 0
    sample = 1 if case["bits"] <= 8 else 2
    return {"bytes": n * (sample + (sample if case["lossless"] else 0.35)),
            "flops": n * (gates + step1 + steps + lifting + temporal)}


def exact(case, seed):
    """Decoding a lossless stream gives the image back; the other results are whole numbers that
    only the codec itself defines."""
    if case["kind"] == "decode" and case["lossless"]:
        imgs = [_image(seed, k, h, w, ch, case["bits"]) for k, (h, w, ch, _) in enumerate(_sizes(case))]
        got = np.stack(imgs)
        return got if got.dtype == np.uint8 else got.view(np.int16)
    return None
