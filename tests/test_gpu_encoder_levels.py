"""The forward transform's column-strip kernel at the sizes where a strip, a
lane or a warp's rows end: 240-column strips, 8-column lanes, warps of 8 to
32 row pairs, subbands down to two samples, and planes that start at an odd
address.  5/3 is integer arithmetic, so the GPU's stream bytes equal the
oracle encoder's."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (width, height, levels): one lane row; below, at and above one and two
# strips; partial lanes at the deep levels (w / 2^l not a multiple of 8);
# one and several warps of rows
SIZES = [(32, 32, 4), (224, 64, 2), (256, 32, 3), (480, 96, 5), (512, 160, 3), (736, 64, 5), (96, 2080, 4),
         (1504, 544, 4)]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("offset", [0, 1])
def test_integer_stream_equals_oracle(size, offset):
    from paper_2208_10859_gb300 import wv
    w, h, levels = size
    rng = np.random.default_rng(w + h)
    frames = [(rng.integers(0, 256, (h, w), dtype=np.uint8),) for _ in range(2)]
    p = O.Params(w, h, 1, 0, levels, O.WAVELET_53, 2, 1, 64, 1.0)
    desc = dict(width=w, height=h, planes=1, chroma_420=0, levels=levels, wavelet=0, num_frames=2, tlevels=1,
                block=64, quant=0, step=1.0)
    dev = []
    for (f,) in frames:
        mem = torch.zeros(w * h + offset, dtype=torch.uint8, device="cuda")
        mem[offset:] = torch.from_numpy(f.ravel()).cuda()
        dev.append((mem[offset:].view(h, w),))
    assert wv.encode(dev, desc) == O.encode(frames, p)
