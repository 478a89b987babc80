"""Device memory of a server's resident streams: the server decodes in batches,
which bring their own planes, so its streams do not hold the scratch of the
third and fourth viewport in flight, a cache budget holds as many streams as
that allows, and the results are those of a stream opened by the caller."""
import math

import pytest

import helpers as H

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _set_floor(p):
    """Bytes that one viewport's planes cannot do without: the reconstruction
    and the float LL_2 planes."""
    px = p.width * p.height * (1.5 if p.chroma_420 else p.planes)
    return int(px + px / 16 * 4)


@pytest.mark.parametrize("name", ("yuv97", "fov97"))
def test_resident_streams_hold_two_sets(name):
    from paper_2208_10859_gb300 import wv
    _, p, data, _ = H.case(name)
    need = wv.query(data)[1]
    one = wv.Stream(data)
    resident = need - 2 * _set_floor(p)     # four sets by default at these sizes
    # room for three such streams, not for three of the caller's size
    sv = wv.Server(slots=1, max_batch=4, cache_bytes=3 * resident)
    assert 3 * resident < 3 * need
    ids = [sv.add_stream(data) for _ in range(3)]
    for rep in range(2):
        for k, i in enumerate(ids):
            got, want = (torch.zeros((48, 64, 4), dtype=torch.uint8, device="cuda") for _ in range(2))
            sv.wait(sv.submit(i, 0, 0.4 * k, 0.1, math.radians(100), got))
            one.decode_viewport(0, 0.4 * k, 0.1, math.radians(100), want)
            torch.cuda.synchronize()
            assert torch.equal(got, want)
    st = sv.stats()
    assert st["uploads"] == 3 and st["evictions"] == 0, st
    assert 0 < st["resident_bytes"] <= 3 * resident
    sv.close()
