"""wv_cnn_forward with the output over the input: the whole network is one
kernel whose thread blocks read pixels around their tiles, so an output that
overlaps the input must not be stored while others still read it.  The results
are those of separate buffers, bit for bit (the network's sums have a fixed
order), for shapes of one and of many tiles, segments and images, for every
kind of overlap, and when captured into a graph."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _net():
    from paper_2208_10859_gb300 import wv
    flat = wv.cnn_init_params(5)
    flat[-(32 * 9 + 1):] *= 8.0     # a residual that no rounding of y hides
    return wv.CNN(flat)


def _run(net, x, y, n, h, w):
    from paper_2208_10859_gb300 import wv
    cs = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert wv._lib().wv_cnn_forward(net.handle, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), n, h, w,
                                    cs) == 0


def _input(n, h, w):
    g = torch.Generator(device="cuda").manual_seed(n * h + w)
    return torch.rand((n, h, w), generator=g, device="cuda")


# one pixel, one tile, the edge of a tile, many tiles, many segments, images
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (1, 20, 100), (1, 9, 121), (2, 64, 300), (1, 700, 1000), (5, 257, 241)])
def test_in_place_equals_separate_buffers(n, h, w):
    net, x = _net(), _input(n, h, w)
    want = net.forward(x)
    assert not torch.equal(want, x)
    for _ in range(3):
        buf = x.clone()
        _run(net, buf, buf, n, h, w)
        assert torch.equal(buf, want)
    # partial overlaps, the output ahead of and behind the input
    k = n * h * w
    for shift in (1, w, w + 7, k - 1):
        for ahead in (True, False):
            room = torch.zeros(2 * k, device="cuda")
            a, b = (0, min(shift, k)) if ahead else (min(shift, k), 0)
            xi, yi = room[a:a + k].view(n, h, w), room[b:b + k].view(n, h, w)
            xi.copy_(x)
            _run(net, xi, yi, n, h, w)
            assert torch.equal(yi, want), (shift, ahead)
    assert net.sync_status() == 0
    net.close()


def test_in_place_captured():
    n, h, w = 1, 300, 500
    net, x = _net(), _input(n, h, w)
    want = net.forward(x)
    buf = x.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _run(net, buf, buf, n, h, w)
    for _ in range(3):
        buf.copy_(x)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, want)
    assert net.sync_status() == 0
    net.close()
