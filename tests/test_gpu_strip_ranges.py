"""The strip fine pass in every range of its size rules, against the square-tile
passes (the same arithmetic per sample, so 8-bit results and 5/3 floats are
equal): whole planes cut into 16, 32 and 64 rows, frames whose viewports list
whole 32-row strips and 64-row strips, and batches whose targets sum to 64-row
strips, foveated and not, with several decode classes as branches of the graph."""
import math

import numpy as np
import pytest

import helpers as H

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _strips(w, h):
    """Strips of 64 rows of a 4:2:0 frame (what the rules count)."""
    up = lambda a, b: -(-a // b)
    return up(w, 224) * up(h, 64) + 2 * up(w // 2, 224) * up(h // 2, 64)


def _stream(w, h, levels, wavelet, tlevels, paper, seed, step=3.0):
    from paper_2208_10859_gb300 import wv
    g = torch.Generator(device="cuda").manual_seed(seed)
    frames = []
    for _ in range(1 << tlevels):
        fr = []
        for s in (1, 2, 2):
            x = torch.rand((1, 1, h // s // 8, w // s // 8), generator=g, device="cuda") * 255
            x = torch.nn.functional.interpolate(x, size=(h // s, w // s), mode="bilinear")[0, 0]
            x += 6 * torch.randn(x.shape, generator=g, device="cuda")
            fr.append(x.round().clamp(0, 255).to(torch.uint8))
        frames.append(tuple(fr))
    d = dict(width=w, height=h, planes=3, chroma_420=1, levels=levels, wavelet=wavelet, num_frames=1 << tlevels,
             tlevels=tlevels, block=32, quant=0, step=step, stereo=0)
    return wv.Stream(wv.encode_paper(frames, d, 0.1, 0.005) if paper else wv.encode(frames, d))


# width, height, rows of the luma plane's strips, range of the viewports' strips
# (152 SMs: 16 rows up to 912 of them, 32 up to 912, else 64; viewports: halves
# of 32 rows up to 608 strips of a frame, 32 rows up to 2432, else 64)
SIZES = [(2048, 1024, 16, (0, 608)), (2048, 2048, 32, (0, 608)), (4096, 2080, 64, (609, 2432)),
         (8192, 4128, 64, (2433, 1 << 30))]


@pytest.mark.parametrize("kind", ["9/7", "5/3", "records"])
@pytest.mark.parametrize("w,h,rows,band", SIZES, ids=lambda v: str(v) if isinstance(v, int) else "")
def test_every_range_equals_square_tiles(w, h, rows, band, kind):
    assert band[0] <= _strips(w, h) <= band[1]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        per = lambda r: -(-w // 224) * -(-h // r)
        assert rows == next((r for r in (16, 32) if per(r) <= 6 * sms), 64)
    wavelet = 0 if kind == "5/3" else 1
    s = _stream(w, h, 4, wavelet, 1, kind == "records", seed=w + h)
    for plane in (0, 1, 2):
        pw, ph = (w // 2, h // 2) if plane else (w, h)
        got = {}
        for mode in (0, 2):
            s.set_decode_mode(mode)
            u8 = torch.zeros((ph, pw), dtype=torch.uint8, device="cuda")
            f = torch.zeros((ph, pw), dtype=torch.float32, device="cuda")
            s.decode_full(1, plane, u8)
            s.decode_full(1, plane, f, as_float=True)
            got[mode] = (u8, f)
        assert torch.equal(got[0][0], got[2][0]), plane
        assert float(got[0][0].float().std()) > 5
        if wavelet == 0:
            assert torch.equal(got[0][1], got[2][1])
        else:
            assert float((got[0][1].double() - got[2][1].double()).abs().max()) <= H.tol_97_levels()
    for k, (yaw, pitch) in enumerate(((0.3, 0.2), (3.1, -1.2), (-2.0, 1.4), (1.0, -0.2))):
        outs = []
        for mode in (0, 2):
            s.set_decode_mode(mode)
            out = torch.zeros((203, 330, 4), dtype=torch.uint8, device="cuda")
            s.decode_viewport(k % 2, yaw, pitch, math.radians(95), out)
            outs.append(out)
        assert torch.equal(outs[0], outs[1]), k
    assert s.sync_status() == 0
    s.close()


def test_batches_of_64_row_strips():
    from paper_2208_10859_gb300 import wv
    w, h = 2048, 1024
    streams = [_stream(w, h, 5, 1, 1, False, 1), _stream(w, h, 5, 0, 1, False, 2), _stream(w, h, 4, 1, 0, False, 3),
               _stream(w, h, 3, 0, 0, False, 4)]

    def requests():
        rng = np.random.default_rng(7)
        out = []
        for k in range(16):
            s = streams[k % 4]
            fovea = k % 8 >= 4
            o = torch.zeros((120 + k, 161, 4), dtype=torch.uint8, device="cuda")
            out.append(wv.ViewRequest(s, k % s.desc["num_frames"], float(rng.uniform(-3.1, 3.1)),
                                      float(rng.uniform(-1.3, 1.3)), math.radians(float(rng.uniform(80, 110))), o,
                                      fovea, float(rng.uniform(-0.2, 0.2)), 0.05, 0.25, 0.5))
        return out

    assert 16 * _strips(w, h) > 2432 and 10 * _strips(w, h) < 2432      # together 64 rows, alone finer
    got = {}
    for name, strips, timing, limit in (("square", False, False, None), ("graph", True, False, None),
                                        ("serial", True, True, None), ("waves", True, False, 1 << 24)):
        b = wv.Batch()
        b.set_strips(strips)
        b.set_timing(timing)
        if limit:
            b.set_memory_limit(limit)
        reqs = requests()
        for _ in range(2):          # captured, then replayed
            b.decode(reqs)
        torch.cuda.synchronize()
        assert b.sync_status() == 0
        st = b.stats()
        assert (st["waves"] > 2) == bool(limit) and st["fine_tiles"] > 0
        got[name] = reqs
        b.close()
    for name in ("graph", "serial", "waves"):
        for a, c in zip(got["square"], got[name]):
            assert torch.equal(a.out, c.out), name
    for r in got["graph"]:
        assert float(r.out[..., :3].float().std()) > 5
        if not r.fovea:
            one = torch.zeros_like(r.out)
            r.stream.decode_viewport(r.frame, r.yaw, r.pitch, r.fov, one)
            assert torch.equal(one, r.out)
    for s in streams:
        assert s.sync_status() == 0
        s.close()
