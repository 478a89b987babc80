"""Viewports and whole planes in flight at the same time: a run of calls without
a wait between them (more of them than there are buffer sets, viewports of
different poses and frames, whole planes between them) gives what each call
gives alone, on a frame that takes four sets and on one that takes three; and a
closed stream's internal CUDA streams serve the next one."""
import math

import pytest

pytestmark = pytest.mark.gpu


def _stream(w, h, seed):
    import torch
    from paper_2208_10859_gb300 import wv
    g = torch.Generator(device="cuda").manual_seed(seed)
    frames = []
    for _ in range(2):
        fr = []
        for p in range(3):
            s = 2 if p else 1
            x = torch.rand((1, 1, h // s // 16, w // s // 16), generator=g, device="cuda") * 255
            x = torch.nn.functional.interpolate(x, size=(h // s, w // s), mode="bilinear")[0, 0]
            fr.append(x.round().clamp(0, 255).to(torch.uint8))
        frames.append(tuple(fr))
    d = dict(width=w, height=h, planes=3, chroma_420=1, levels=5, wavelet=1, num_frames=2, tlevels=1, block=128, quant=0,
             step=4.0, stereo=0)
    return wv.Stream(wv.encode(frames, d))


@pytest.mark.parametrize("w,h", [(1024, 512), (8192, 4096)])
def test_calls_in_flight_equal_calls_alone(w, h):
    import torch

    def calls(out, ow, oh):
        for k in range(11):
            yaw, pitch = -3.0 + 0.55 * k, 1.2 * math.sin(1.7 * k)
            if k % 4 == 2:
                p = k % 3
                t = torch.float32 if k % 8 == 2 else torch.uint8
                o = torch.zeros((h >> (p > 0), w >> (p > 0)), dtype=t, device="cuda")
                out.append((o, lambda s, o=o, p=p, k=k, t=t: s.decode_full(k & 1, p, o, as_float=t == torch.float32)))
            else:
                o = torch.zeros((oh, ow, 4), dtype=torch.uint8, device="cuda")
                out.append((o, lambda s, o=o, k=k, yaw=yaw, pitch=pitch:
                            s.decode_viewport(k & 1, yaw, pitch, math.radians(100), o)))
        return out

    s = _stream(w, h, 3)
    alone = calls([], 320, 280)
    for _, c in alone:
        c(s)
        torch.cuda.synchronize()
    assert s.sync_status() == 0
    for rep in range(3):
        t = _stream(w, h, 3) if rep == 2 else s     # a new stream: its sets' first calls, on a closed one's lanes
        flight = calls([], 320, 280)
        for _, c in flight:
            c(t)
        torch.cuda.synchronize()
        assert t.sync_status() == 0
        for (a, _), (b, _) in zip(alone, flight):
            assert torch.equal(a, b)
        if rep == 1:
            s.close()
