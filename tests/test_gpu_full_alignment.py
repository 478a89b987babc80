"""Whole planes into destinations at every address they may have: bytes from any
multiple of 2 (strips store words, so a plane off a word boundary takes the
square tiles), floats from any multiple of 4.  The samples are those of an
aligned destination, nothing outside the plane is written, and addresses the
kernels cannot store to are refused before anything is launched."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# wavelet, levels, quantiser (1: record format), temporal levels
STREAMS = {"9/7": (1, 4, 0, 1), "5/3": (0, 3, 0, 0), "records": (1, 4, 1, 1), "two levels": (0, 2, 0, 0)}


def _stream(name, w=480, h=288):
    from paper_2208_10859_gb300 import wv
    wavelet, levels, quant, tl = STREAMS[name]
    rng = np.random.default_rng(len(name))
    frames = []
    for _ in range(1 << tl):
        fr = []
        for s in (1, 2, 2):
            y, x = np.mgrid[0:h // s, 0:w // s]
            v = 120 + 90 * np.sin(x * s / 37.0) * np.cos(y * s / 23.0) + rng.normal(0, 6, x.shape)
            fr.append(torch.tensor(v.round().clip(0, 255).astype(np.uint8), device="cuda"))
        frames.append(tuple(fr))
    d = dict(width=w, height=h, planes=3, chroma_420=1, levels=levels, wavelet=wavelet, num_frames=1 << tl, tlevels=tl,
             block=32, quant=0, step=2.0, stereo=0)
    return wv.Stream(wv.encode_paper(frames, d, 0.05, 0.005) if quant else wv.encode(frames, d))


@pytest.mark.parametrize("name", STREAMS)
@pytest.mark.parametrize("plane", (0, 2))
def test_unaligned_destinations(name, plane):
    from paper_2208_10859_gb300 import wv
    s = _stream(name)
    h, w = (288, 480) if plane == 0 else (144, 240)
    want = torch.zeros((h, w), dtype=torch.uint8, device="cuda")
    s.decode_full(0, plane, want)
    fwant = torch.zeros((h, w), dtype=torch.float32, device="cuda")
    s.decode_full(0, plane, fwant, as_float=True)
    assert float(want.float().std()) > 10
    for off in (2, 4, 6, 10):
        room = torch.full((h * w + 32,), 77, dtype=torch.uint8, device="cuda")
        s.decode_full(0, plane, room[off:off + h * w])
        assert torch.equal(room[off:off + h * w].view(h, w), want), off
        assert bool((room[:off] == 77).all()) and bool((room[off + h * w:] == 77).all())
    for off in (1, 2, 3):
        room = torch.full((h * w + 8,), -5.0, dtype=torch.float32, device="cuda")
        s.decode_full(0, plane, room[off:off + h * w], as_float=True)
        assert torch.equal(room[off:off + h * w].view(h, w), fwant), off
        assert bool((room[:off] == -5.0).all()) and bool((room[off + h * w:] == -5.0).all())
    room = torch.zeros(4 * h * w + 16, dtype=torch.uint8, device="cuda")
    for off, as_float in ((1, False), (3, False), (1, True), (2, True)):
        with pytest.raises(wv.WVError) as e:
            s.decode_full(0, plane, room[off:], as_float=as_float)
        assert e.value.code == -1
    assert not bool(room.any())
    assert s.sync_status() == 0
    s.close()
