"""The work a user of this library has it do, as cases to be timed.

A case is a dict of plain values.  Its "kind" names the public entry point:

  view    Stream.decode_viewport: consecutive head poses of one stream, each
          decoded from the next video frame (what a player calls)
  batch   Batch.decode: many viewers' requests over several streams at once
          (what a streaming server calls)
  full    Stream.decode_full of every plane of one frame, as bytes or floats
  encode  wv.encode: a group of frames to stream bytes
  filter  CNN.forward: the learned post-filter on a viewport's luma
  train   CNN.gradients: loss and every parameter gradient of a batch of
          patches (a training step's forward and backward)

Streams carry seeded frames with a natural-image-like spectrum and moving
textured discs, coded with the sizes, wavelets, level counts, inter-frame sets,
block sizes and quantiser steps of the repository's benchmark and tests.
"""
from __future__ import annotations

import math
import struct

import numpy as np
import torch
import torch.nn.functional as F

from paper_2208_10859_gb300 import wv

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _view(name, w, h, **kw):
    d = dict(name=name, kind="view", w=w, h=h, planes=3, levels=5, wavelet=1, tlevels=1, block=256, step=4.0,
             stereo=0, paper=False, host=False, poses=1, out_w=1080, out_h=1080, fov=110.0)
    d.update(kw)
    return d


def listed():
    return [
        # a thumbnail-sized grey frame, coded losslessly, decoded whole: the
        # smallest call, where launches and latency count
        dict(name="full_512_lossless", kind="full", w=512, h=512, planes=1, levels=3, wavelet=0, tlevels=0,
             block=256, step=1.0, as_float=False),
        # a low-resolution preview of a 360-degree video: one small viewport
        _view("view_1k_preview", 1024, 512, levels=3, block=64, out_w=540, out_h=540, fov=90.0),
        # archive quality (lossless 5/3), a frame size that fills no tile or
        # block evenly and a window of odd size
        _view("view_2880_lossless", 2880, 1440, levels=4, wavelet=0, block=128, step=1.0, poses=4, out_w=1001,
              out_h=777, fov=100.0),
        # a headset following an 8k video: the library's main use
        _view("view_8k", 8192, 8192, poses=8, out_w=2160, out_h=2160),
        # stereo video in inter-frame sets of four, one viewport per eye
        _view("view_4k_stereo", 4096, 4096, tlevels=2, block=128, stereo=1, poses=4, out_w=1440, out_h=1440),
        # the byte-record stream format with 32 x 32 blocks, sets of four
        _view("view_4k_records", 4096, 4096, levels=6, tlevels=2, block=32, paper=True, poses=4, out_w=1440,
              out_h=1440),
        # a server's batch: gaze-dependent detail, streams of unequal size,
        # wavelet and level count
        dict(name="batch_24_foveated", kind="batch", n=24, mix="2048/1/4 2048/0/4 4096/1/5 4096/0/5 6144/1/6",
             fovea=True, out=2160, step=4.0),
        # a server's batch at full detail: viewers of the same frames
        dict(name="batch_12_shared", kind="batch", n=12, mix="4096/1/5 2048/0/4", fovea=False, out=1440, step=4.0),
        # every plane of a 4k frame as float samples (processing after the decode)
        dict(name="full_4k_float", kind="full", w=4096, h=4096, planes=3, levels=5, wavelet=1, tlevels=1,
             block=256, step=4.0, as_float=True),
        # coding one inter-frame pair of a 4k video
        dict(name="encode_4k", kind="encode", w=4096, h=4096, planes=3, levels=5, wavelet=1, tlevels=1, block=256,
             step=4.0),
        # the post-filter on a headset's viewport
        dict(name="filter_2160", kind="filter", n=1, h=2160, w=2160),
        # one training step's forward and backward on the trainer's batch
        dict(name="train_16x256", kind="train", n=16, h=256, w=256),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi, levels):
    """A frame side: a multiple of the mask cell, and of 2^levels in the
    half-size chroma planes."""
    m = max(32, 2 << levels)
    return max(m, int(round(_log(rng, lo, hi) / m)) * m)


def draw(rng):
    kind = rng.choice(["view", "view", "view", "batch", "full", "encode", "filter", "train"])
    if kind == "filter":
        return dict(kind=kind, n=rng.choice([1, 1, 2]), h=int(_log(rng, 64, 1440)), w=int(_log(rng, 64, 1440)))
    if kind == "train":
        return dict(kind=kind, n=rng.randint(1, 16), h=int(_log(rng, 32, 256)), w=int(_log(rng, 32, 256)))
    if kind == "batch":
        sizes = {2048: (4, 5), 4096: (5, 6), 6144: (4, 6)}
        mix = []
        for _ in range(rng.randint(1, 4)):
            s = rng.choice([2048, 2048, 4096, 6144])
            mix.append("%d/%d/%d" % (s, rng.randint(0, 1), rng.choice(sizes[s])))
        return dict(kind=kind, n=rng.randint(1, 20), mix=" ".join(mix), fovea=rng.random() < 0.6,
                    out=int(_log(rng, 480, 2160)), step=rng.choice([4.0, 6.0]))
    levels = rng.randint(3, 6)
    wavelet = rng.choice([0, 1, 1])
    if kind == "full":
        w, h = _size(rng, 256, 4096, levels), _size(rng, 256, 4096, levels)
        return dict(kind=kind, w=w, h=h, planes=rng.choice([1, 3]), levels=levels, wavelet=wavelet,
                    tlevels=rng.randint(0, 1), block=rng.choice([64, 128, 256]),
                    step=4.0 if wavelet else 1.0, as_float=rng.random() < 0.5)
    if kind == "encode":
        w, h = _size(rng, 256, 4096, levels), _size(rng, 256, 4096, levels)
        return dict(kind=kind, w=w, h=h, planes=rng.choice([1, 3]), levels=levels, wavelet=wavelet,
                    tlevels=rng.randint(0, 1), block=rng.choice([64, 128, 256]), step=4.0 if wavelet else 1.0)
    paper = rng.random() < 0.2
    if paper:
        wavelet = 1
    w = _size(rng, 512, 8192, levels)
    stereo = int(rng.random() < 0.2)
    if stereo:
        h = max(2, int(round(w / max(64, 2 << levels)))) * max(64, 2 << levels)
    else:
        h = max(1, int(round(w / 2 / max(32, 2 << levels)))) * max(32, 2 << levels)
    c = _view(None, w, h, planes=rng.choice([1, 3, 3, 3]), levels=levels, wavelet=wavelet,
                 tlevels=rng.choice([0, 1, 1, 2]), block=32 if paper else rng.choice([64, 128, 256]),
                 step=rng.choice([4.0, 6.0, 12.0]) if wavelet else 1.0, stereo=stereo, paper=paper,
                 host=rng.random() < 0.1, poses=rng.randint(1, 6), out_w=int(_log(rng, 200, 2160)),
                 out_h=int(_log(rng, 200, 2160)), fov=round(rng.uniform(70.0, 120.0), 1))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _noise(g, h, w, mean, std):
    """Gaussian noise with a 1/f^1.5 amplitude spectrum up to 1/16 cycle per pixel."""
    spec = torch.fft.rfft2(torch.randn((h, w), generator=g, device=DEV))
    f = torch.sqrt(torch.fft.fftfreq(h, device=DEV)[:, None] ** 2 + torch.fft.rfftfreq(w, device=DEV)[None, :] ** 2)
    gain = torch.where((f > 0) & (f <= 1 / 16), f.clamp(min=1e-9) ** -1.5, torch.zeros((), device=DEV))
    x = torch.fft.irfft2(spec * gain, s=(h, w))
    return (x - x.mean()) * (std / x.std().clamp(min=1e-9)) + mean


def _disc(img, cx, cy, r, fn):
    """Paint a disc; longitude wraps."""
    h, w = img.shape
    y0, y1 = max(0, int(cy - r)), min(h, int(cy + r) + 2)
    r = min(r, w / 2 - 2)
    x0, x1 = int(cx - r) - 1, int(cx + r) + 2
    if y1 <= y0:
        return
    dy = torch.arange(y0, y1, device=DEV)[:, None] - cy
    dx = torch.arange(x0, x1, device=DEV)[None, :] - cx
    cols = torch.arange(x0, x1, device=DEV) % w
    img[y0:y1, cols] = torch.where(dx * dx + dy * dy <= r * r, fn(dx, dy), img[y0:y1, cols])


def _frames(w, h, planes, n, seed, grain=0.0):
    """n frames (tuples of uint8 planes, chroma at half size): band-limited
    noise, 50 textured discs moving 2 pixels a frame, optional sensor grain."""
    g = torch.Generator(device=DEV).manual_seed(1000003 * seed + 17)
    rng = np.random.default_rng(seed)
    bg = [_noise(g, h, w, 128.0, 40.0)]
    if planes == 3:
        bg += [_noise(g, h // 2, w // 2, 128.0, 14.0) for _ in range(2)]
    s = w / 8192.0
    discs = [dict(cx=rng.uniform(0, w), cy=rng.uniform(0, h), r=rng.uniform(64, 512) * s, th=rng.uniform(0, 2 * math.pi),
                  k=rng.uniform(1 / 64, 1 / 12), phi=rng.uniform(0, math.pi), amp=rng.uniform(20, 60),
                  v=(rng.uniform(40, 215), rng.uniform(64, 192), rng.uniform(64, 192))) for _ in range(50)]
    out = []
    for t in range(n):
        fr = [p.clone() for p in bg]
        for d in discs:
            cx, cy = (d["cx"] + 2 * t * math.cos(d["th"])) % w, d["cy"] + 2 * t * math.sin(d["th"])
            kx, ky = 2 * math.pi * d["k"] * math.cos(d["phi"]), 2 * math.pi * d["k"] * math.sin(d["phi"])
            _disc(fr[0], cx, cy, d["r"], lambda dx, dy: d["v"][0] + d["amp"] * torch.sin(kx * dx + ky * dy))
            for p in range(1, planes):
                _disc(fr[p], cx / 2, cy / 2, d["r"] / 2, lambda dx, dy: torch.full((), d["v"][p], device=DEV))
        if grain:
            fr = [p + grain * torch.randn(p.shape, generator=g, device=DEV) for p in fr]
        out.append(tuple(p.round().clamp(0, 255).to(torch.uint8) for p in fr))
    return out


def _desc(case, n):
    return dict(width=case["w"], height=case["h"], planes=case["planes"], chroma_420=int(case["planes"] == 3),
                levels=case["levels"], wavelet=case["wavelet"], num_frames=n, tlevels=case["tlevels"],
                block=case["block"], quant=0, step=case["step"], stereo=case.get("stereo", 0))


def _grain(case):
    """Sensor grain (sigma 2): what a camera hands an encoder, and what
    lossless streams carry; the streams of the other cases are of clean frames."""
    return 2.0 if case["kind"] == "encode" or (case["wavelet"] == 0 and case["step"] == 1.0) else 0.0


def _room(case):
    """Bytes of a stream that stores every block of one inter-frame set."""
    n = 0
    for p in range(case["planes"]):
        for k in [case["levels"]] + 3 * list(range(1, case["levels"] + 1)):
            n += math.prod(-(-((case[side] >> (p > 0)) >> k) // case["block"]) for side in "wh")
    return (1 << case["tlevels"]) * n * (4 + 2 * case["block"] ** 2) + 512


def _encode(frames, case):
    d = _desc(case, len(frames))
    # the thresholds of the repository's high-quality record streams
    return wv.encode_paper(frames, d, 0.1, 0.005) if case.get("paper") else wv.encode(frames, d)


# ---- a plain 64-bit coder of the stream format (float whole-plane decodes) ----

_A, _B, _G, _D, _K = -1.586134342059924, -0.052980118572961, 0.882911075530934, 0.443506852043971, 1.230174104914001


def _lift(even, odd, c, to_odd):
    """One CDF 9/7 lifting step along the last axis, whole-sample symmetric."""
    if to_odd:
        return odd + c * (even + torch.cat([even[..., 1:], even[..., -1:]], -1))
    return even + c * (torch.cat([odd[..., :1], odd[..., :-1]], -1) + odd)


def _fwd(x):
    e, o = x[..., 0::2], x[..., 1::2]
    o = _lift(e, o, _A, True)
    e = _lift(e, o, _B, False)
    o = _lift(e, o, _G, True)
    e = _lift(e, o, _D, False)
    return torch.cat([e / _K, o * _K], -1)


def _inv(x):
    n = x.shape[-1] // 2
    e, o = x[..., :n] * _K, x[..., n:] / _K
    e = _lift(e, o, -_D, False)
    o = _lift(e, o, -_G, True)
    e = _lift(e, o, -_B, False)
    o = _lift(e, o, -_A, True)
    return torch.stack([e, o], -1).flatten(-2)


def _codes(case, seed):
    """Dead-zone codes (Mallat layout) of every coefficient frame and plane of
    one inter-frame set of a 9/7 stream."""
    frames = _frames(case["w"], case["h"], case["planes"], 1 << case["tlevels"], seed)
    out = []
    for p in range(case["planes"]):
        c = []
        for f in frames:
            x = f[p].double() - 128.0
            h, w = x.shape
            for lv in range(case["levels"]):
                s = x[:h >> lv, :w >> lv]
                x[:h >> lv, :w >> lv] = _fwd(_fwd(s.t().contiguous()).t().contiguous())
            c.append(x)
        if case["tlevels"] == 1:
            c = [(c[0] + c[1]) / 2, (c[1] - c[0]) / 2]
        out.append([(x.sign() * (x.abs() / case["step"]).floor()).to(torch.int16) for x in c])
    return out


def _pack(case, codes):
    """Stream bytes of the codes: header, block table, stored blocks."""
    B, L, n = case["block"], case["levels"], 1 << case["tlevels"]
    table, payload, slots = [], [], 0
    for t in range(n):
        for p in range(case["planes"]):
            x = codes[p][t]
            h, w = x.shape
            bands = [x[:h >> L, :w >> L]]
            for lv in range(L, 0, -1):
                a, b = h >> lv, w >> lv
                bands += [x[:a, b:2 * b], x[a:2 * a, :b], x[a:2 * a, b:2 * b]]
            for s in bands:
                s = F.pad(s, (0, -s.shape[1] % B, 0, -s.shape[0] % B))
                blk = s.reshape(s.shape[0] // B, B, s.shape[1] // B, B).transpose(1, 2).reshape(-1, B * B)
                keep = (blk != 0).any(1)
                idx = torch.where(keep, torch.cumsum(keep, 0) - 1 + slots, -1)
                slots += int(keep.sum())
                table.append(idx.to(torch.int32).cpu().numpy())
                payload.append(blk[keep].reshape(-1).cpu().numpy())
    table = np.concatenate(table).astype("<i4")
    off = (128 + table.nbytes + 255) // 256 * 256
    d = _desc(case, n)
    head = struct.pack("<4s12IfII3Q", b"WVS1", 1, d["width"], d["height"], d["planes"], d["chroma_420"], d["levels"],
                       d["wavelet"], d["num_frames"], d["tlevels"], d["block"], 0, 0, d["step"], table.size // n, 0,
                       slots, 128, off)
    body = head.ljust(128, b"\0") + table.tobytes()
    return body.ljust(off, b"\0") + np.concatenate(payload).astype("<i2").tobytes()


# ---- the post-filter network ----

def _params(seed):
    """The trainer's initial network (He-normal layers, a small last one)."""
    return wv.cnn_init_params(seed)


def _net64(params, x):
    o, c = 0, x.double()[:, None]
    for k, (co, ci) in enumerate(((32, 1), (32, 32), (32, 32), (32, 32), (1, 32))):
        wt = params[o:o + co * ci * 9].reshape(co, ci, 3, 3)
        b = params[o + co * ci * 9:o + co * ci * 9 + co]
        o += co * ci * 9 + co
        c = F.conv2d(c, wt, b, padding=1)
        if k < 4:
            c = c.clamp(min=0)
    return x.double() + c[:, 0]


def _patches(case, seed):
    """Decoded-like luma in [0, 1] and its original."""
    g = torch.Generator(device=DEV).manual_seed(seed * 7919 + 5)
    n, h, w = case["n"], case["h"], case["w"]
    t = torch.stack([_noise(g, h, w, 0.5, 0.16) for _ in range(n)]).clamp(0, 1)
    x = (t + 0.02 * torch.randn(t.shape, generator=g, device=DEV)).clamp(0, 1)
    return ((x * 255).round() / 255).float().contiguous(), t.float().contiguous()


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _poses(n, seed):
    """A head turning at up to two degrees a frame from a random start (yaw
    anywhere, pitch within 45 degrees)."""
    rng = np.random.default_rng(seed + 77)
    yaw, pitch = rng.uniform(-math.pi, math.pi), rng.uniform(-math.pi / 4, math.pi / 4)
    out = []
    for _ in range(n):
        out.append((float(yaw), float(pitch)))
        yaw += math.radians(rng.uniform(-2, 2))
        pitch = min(max(pitch + math.radians(rng.uniform(-2, 2)), -1.4), 1.4)
    return out


def _rgba(h, w):
    return torch.zeros((h, w, 4), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "view":
        n = max(2, 1 << case["tlevels"])
        s = wv.Stream(_encode(_frames(case["w"], case["h"], case["planes"], n, seed, _grain(case)), case),
                      host_payload=case["host"])
        # stereo: both eyes of every second pose
        eyes = 2 if case["stereo"] else 1
        base = _poses((case["poses"] + eyes - 1) // eyes, seed)
        calls = [(i // eyes % n, *base[i // eyes], math.radians(case["fov"]), _rgba(case["out_h"], case["out_w"]),
                  i % eyes) for i in range(case["poses"])]
        return dict(kind=kind, stream=s, calls=calls)
    if kind == "batch":
        rng = np.random.default_rng(seed + 99)
        streams = []
        for k, m in enumerate(case["mix"].split()):
            size, wavelet, levels = (int(v) for v in m.split("/"))
            c = dict(w=size, h=size, planes=3, levels=levels, wavelet=wavelet, tlevels=1, block=256,
                     step=case["step"])
            streams.append(wv.Stream(_encode(_frames(size, size, 3, 2, seed * 31 + k), c)))
        reqs = []
        for k in range(case["n"]):
            reqs.append(wv.ViewRequest(
                streams[k % len(streams)], int(rng.integers(2)), float(rng.uniform(-math.pi, math.pi)),
                float(rng.uniform(-math.pi / 4, math.pi / 4)), math.radians(float(rng.uniform(90, 120))),
                _rgba(case["out"], case["out"]), case["fovea"], float(rng.uniform(-0.15, 0.15)),
                float(rng.uniform(-0.15, 0.15)), math.radians(20), math.radians(40)))
        return dict(kind=kind, batch=wv.Batch(), reqs=reqs)
    if kind == "full":
        if case["wavelet"] == 1:
            data = _pack(case, _codes(case, seed))
        else:
            data = _encode(_frames(case["w"], case["h"], case["planes"], 1 << case["tlevels"], seed, _grain(case)),
                           case)
        t = torch.float32 if case["as_float"] else torch.uint8
        outs = [torch.zeros((case["h"] >> (p > 0), case["w"] >> (p > 0)), dtype=t, device=DEV)
                for p in range(case["planes"])]
        return dict(kind=kind, stream=wv.Stream(data), outs=outs, frame=case["tlevels"], as_float=case["as_float"])
    if kind == "encode":
        frames = _frames(case["w"], case["h"], case["planes"], 1 << case["tlevels"], seed, _grain(case))
        return dict(kind=kind, case=case, frames=frames, file=np.zeros(_room(case), np.uint8))
    x, t = _patches(case, seed)
    return dict(kind=kind, net=wv.CNN(_params(seed)), x=x, t=t)


def run(state):
    kind = state["kind"]
    if kind == "view":
        s = state["stream"]
        for frame, yaw, pitch, fov, out, eye in state["calls"]:
            s.decode_viewport(frame, yaw, pitch, fov, out, eye)
        return [c[4] for c in state["calls"]]
    if kind == "batch":
        state["batch"].decode(state["reqs"])
        return [r.out for r in state["reqs"]]
    if kind == "full":
        for p, out in enumerate(state["outs"]):
            state["stream"].decode_full(state["frame"], p, out, as_float=state["as_float"])
        return state["outs"]
    if kind == "encode":
        data = _encode(state["frames"], state["case"])
        state["file"][:len(data)] = np.frombuffer(data, np.uint8)
        return len(data), state["file"]
    if kind == "filter":
        return state["net"].forward(state["x"])
    return state["net"].gradients(state["x"], state["t"])


# ---------------------------------------------------------------------------
# what a pass cannot do without, and its values in 64 bits
# ---------------------------------------------------------------------------

def _coverage(fov_deg):
    """Mean share of an equirectangular frame that a viewport of this field of
    view shows, over poses with pitch within 45 degrees (half-degree cells)."""
    cells, n = 0, 24
    t = np.tan(np.radians(fov_deg) / 2) * (np.arange(512) + 0.5 - 256) / 256
    x, y = np.meshgrid(t, -t)
    for k in range(n):
        p = math.pi / 4 * (2 * (k + 0.5) / n - 1)
        dy, dz = y * math.cos(p) + math.sin(p), -y * math.sin(p) + math.cos(p)
        lon = np.degrees(np.arctan2(x, dz)) + 180
        lat = np.degrees(np.arctan2(dy, np.hypot(x, dz))) + 90
        m = np.zeros((180, 360), bool)
        m[np.minimum(lat.astype(int), 179), np.minimum(lon.astype(int), 359)] = True
        cells += m.sum()
    return cells / (n * 180 * 360)


def _stored(wavelet, paper):
    """Share of the coefficients that lies in stored blocks, on these frames
    (all-zero blocks are never read)."""
    return 0.065 if paper else 0.75 if wavelet else 1.0


def _view_work(w, h, planes, levels, wavelet, tlevels, paper, fov, out_px):
    """One viewport: the coefficients of what it shows from every coefficient
    frame (two bytes each) and its pixels.  Arithmetic: the synthesis (both
    axes, all levels) about 24 operations a sample, the projection, filtering
    and colour conversion about 100 a pixel."""
    samples = _coverage(fov) * w * h * (1.5 if planes == 3 else 1.0)
    return (samples * 2 * (1 + tlevels) * _stored(wavelet, paper) + 4 * out_px, 24 * samples + 100 * out_px)


def work(case):
    kind = case["kind"]
    if kind == "view":
        h = case["h"] / (2 if case["stereo"] else 1)
        b, f = _view_work(case["w"], h, case["planes"], case["levels"], case["wavelet"], case["tlevels"],
                          case["paper"], case["fov"], case["out_w"] * case["out_h"])
        return dict(bytes=b * case["poses"], flops=f * case["poses"])
    if kind == "batch":
        # a stream's coefficients are read once, however many of its viewers share them
        px = case["out"] ** 2
        mix = [tuple(int(v) for v in m.split("/")) for m in case["mix"].split()]
        bytes_, flops = 4.0 * px * case["n"], 0.0
        for k, (size, wavelet, levels) in enumerate(mix):
            n = len(range(k, case["n"], len(mix)))
            b, f = _view_work(size, size, 3, levels, wavelet, 1, False, 105.0, px)
            whole = 1.5 * size * size * 4 * _stored(wavelet, False)
            bytes_, flops = bytes_ + min(n * (b - 4 * px), whole), flops + n * f
        return dict(bytes=bytes_, flops=flops)
    if kind in ("filter", "train"):
        # 3 x 3 convolutions 1-32-32-32-32-1 (backward: the gradients of
        # inputs and of weights, each the forward's work)
        px = case["n"] * case["h"] * case["w"]
        mac = 9 * (32 + 3 * 32 * 32 + 32)
        if kind == "filter":
            return dict(bytes=8.0 * px, flops=2.0 * mac * px)
        return dict(bytes=8.0 * px, flops=2.0 * (3 * mac - 9 * 32) * px)
    samples = case["w"] * case["h"] * (1.5 if case["planes"] == 3 else 1.0)
    if kind == "full":
        b = samples * (2 * (1 + case["tlevels"]) * _stored(case["wavelet"], False) + (4 if case["as_float"] else 1))
        return dict(bytes=b, flops=24 * samples)
    n = 1 << case["tlevels"]
    return dict(bytes=n * samples * 3, flops=24 * n * samples)   # 8-bit samples in, 16-bit codes out


def exact(case, seed):
    """64-bit values of what run() returns as floats.  Bytes (pixels of
    viewports, 8-bit planes, stream bytes) are whole numbers, compared as such."""
    kind = case["kind"]
    if kind == "full" and case["wavelet"] == 0:
        # lossless streams give the frame back
        fr = _frames(case["w"], case["h"], case["planes"], 1 << case["tlevels"], seed, _grain(case))[case["tlevels"]]
        return [p.double() if case["as_float"] else p for p in fr]
    if kind == "full" and case["as_float"]:
        outs = []
        for c in _codes(case, seed):
            c = [(q.double() + 0.5 * q.sign().double()) * case["step"] for q in c]
            x = c[0] + c[1] if case["tlevels"] else c[0]
            h, w = x.shape
            for lv in reversed(range(case["levels"])):
                s = x[:h >> lv, :w >> lv]
                x[:h >> lv, :w >> lv] = _inv(_inv(s.contiguous()).t().contiguous()).t()
            outs.append(x + 128.0)
        return outs
    if kind == "filter":
        x, _ = _patches(case, seed)
        with torch.no_grad():
            return _net64(torch.from_numpy(_params(seed)).to(DEV).double(), x)
    if kind == "train":
        x, t = _patches(case, seed)
        p = torch.from_numpy(_params(seed)).to(DEV).double().requires_grad_()
        loss = ((_net64(p, x) - t.double()) ** 2).mean()
        loss.backward()
        return loss.detach(), p.grad
    return None
