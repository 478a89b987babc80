"""The strip fine pass against the square-tile passes (decode mode 2) at the
sizes where strips begin and end: planes narrower than a strip, one column
group past a strip, heights that leave a partial strip of 16, 32 and 64 rows,
every number of coefficient frames, both wavelets and the record format.

Both organisations do the same arithmetic per sample, so 8-bit planes,
viewports and 5/3 floats are equal; 9/7 floats are compared with the bound the
other decodes have."""
import math

import numpy as np
import pytest

import helpers as H

pytestmark = pytest.mark.gpu

# width, height, planes, levels, wavelet, tlevels, block
CASES = [
    (64, 64, 3, 3, 1, 0, 16),        # smallest: chroma of 32 x 32
    (224, 96, 1, 3, 0, 1, 32),       # exactly one strip, a half strip of rows
    (256, 160, 3, 3, 1, 2, 64),      # 32 columns past a strip
    (480, 288, 3, 4, 0, 3, 32),      # four coefficient frames
    (704, 352, 3, 4, 1, 3, 64),
    (1344, 416, 1, 5, 1, 1, 128),    # six strips, grey
    (2048, 1024, 3, 5, 0, 0, 256),   # strips of 16 to 64 rows by plane
]


def _frames(w, h, planes, n, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    out = []
    for _ in range(n):
        fr = []
        for p in range(planes):
            s = 2 if p else 1
            x = torch.rand((1, 1, h // s // 8, w // s // 8), generator=g) * 255
            x = torch.nn.functional.interpolate(x, size=(h // s, w // s), mode="bilinear")[0, 0]
            fr.append((x + 6 * torch.randn(x.shape, generator=g)).round().clamp(0, 255).to(torch.uint8).cuda())
        out.append(tuple(fr))
    return out


def _stream(w, h, planes, levels, wavelet, tlevels, block, seed, paper=False):
    from paper_2208_10859_gb300 import wv
    n = 1 << tlevels
    d = dict(width=w, height=h, planes=planes, chroma_420=int(planes == 3), levels=levels, wavelet=wavelet,
             num_frames=n, tlevels=tlevels, block=block, quant=0, step=3.0, stereo=0)
    fr = _frames(w, h, planes, n, seed)
    return wv.Stream(wv.encode_paper(fr, d, 0.1, 0.005) if paper else wv.encode(fr, d))


def _compare(s, w, h, planes, wavelet, frame):
    import torch
    tol = H.tol_97_levels()
    for p in range(planes):
        pw, ph = (w // 2, h // 2) if p else (w, h)
        got = {}
        for mode in (0, 2):
            s.set_decode_mode(mode)
            u8 = torch.zeros((ph, pw), dtype=torch.uint8, device="cuda")
            # one float past a 16-byte boundary: the scalar stores
            room = torch.zeros(ph * pw + 5, dtype=torch.float32, device="cuda")
            f = room[4:-1].view(ph, pw)
            m = room[1:1 + ph * pw].view(ph, pw)
            s.decode_full(frame, p, u8)
            s.decode_full(frame, p, f, as_float=True)
            f = f.clone()
            s.decode_full(frame, p, m, as_float=True)
            assert torch.equal(f, m) and float(room[0]) == 0.0
            got[mode] = (u8.cpu().numpy(), f.cpu().numpy())
        np.testing.assert_array_equal(got[0][0], got[2][0])
        if wavelet == 0:
            np.testing.assert_array_equal(got[0][1], got[2][1])
        else:
            assert np.abs(got[0][1].astype(np.float64) - got[2][1]).max() <= tol
    for yaw, pitch in ((0.3, 0.2), (3.1, -1.2), (-2.0, 1.4)):
        outs = []
        for mode in (0, 2):
            s.set_decode_mode(mode)
            out = torch.zeros((91, 130, 4), dtype=torch.uint8, device="cuda")
            s.decode_viewport(frame, yaw, pitch, math.radians(95), out)
            outs.append(out.cpu().numpy())
        np.testing.assert_array_equal(outs[0], outs[1])
    assert s.sync_status() == 0


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dx%d-%d-L%d-w%d-t%d" % c[:6])
def test_strips_equal_square_tiles(case):
    w, h, planes, levels, wavelet, tlevels, block = case
    s = _stream(*case, seed=w + h)
    for frame in {0, (1 << tlevels) - 1}:
        _compare(s, w, h, planes, wavelet, frame)


@pytest.mark.parametrize("w,h,planes,levels,tlevels", [(128, 96, 3, 3, 0), (480, 256, 1, 4, 1), (704, 384, 3, 5, 2),
                                                        (256, 192, 3, 4, 3)])
def test_record_strips_equal_square_tiles(w, h, planes, levels, tlevels):
    s = _stream(w, h, planes, levels, 1, tlevels, 32, seed=w, paper=True)
    _compare(s, w, h, planes, 1, (1 << tlevels) - 1)
