"""The fused network's give-up path: with no polls allowed every role of the
kernel (issuing warps, stages, in the forward pass and behind a filtered
viewport) gives up at its first wait, the call's error word says so, the context
stays usable, and the next call with the default limit gives the same output as
before.  A limit of one round of polls is enough for the real waits."""
import math

import pytest

import helpers as H

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

WV_ERR_TIMEOUT = -6


def test_waits_that_run_out_are_reported():
    from paper_2208_10859_gb300 import wv
    assert wv._lib().wv_strerror(WV_ERR_TIMEOUT) == b"device wait timed out"
    net = wv.CNN(seed=4)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.rand((3, 190, 300), generator=g, device="cuda")
    want = net.forward(x)
    assert net.sync_status() == 0
    s = wv.Stream(H.case("yuv97")[2])
    view = torch.zeros((2, 60, 200, 4), dtype=torch.uint8, device="cuda")
    s.decode_viewport_filtered(0, 0.2, 0.1, math.radians(100), net, view[0])
    assert net.sync_status() == 0
    for _ in range(2):
        net.set_wait_limit(0)
        net.forward(x)
        assert net.sync_status() == WV_ERR_TIMEOUT
        assert net.sync_status() == 0           # read once, cleared
        s.decode_viewport_filtered(0, 0.2, 0.1, math.radians(100), net, view[1])
        assert net.sync_status() == WV_ERR_TIMEOUT
        net.set_wait_limit(1)                   # one round
        assert torch.equal(net.forward(x), want)
        assert net.sync_status() == 0
        net.set_wait_limit(1 << 30)             # the default again
        assert torch.equal(net.forward(x), want)
        s.decode_viewport_filtered(0, 0.2, 0.1, math.radians(100), net, view[1])
        assert net.sync_status() == 0 and torch.equal(view[0], view[1])
    with pytest.raises(wv.WVError):
        net.set_wait_limit(-1)
    assert s.sync_status() == 0
    net.close()


def test_gradients_whose_waits_run_out():
    """The weight-gradient kernel gives up too, and waits for its products in
    flight before it ends; the next call's gradients are those of an untouched
    network (their sums' order varies, so to rounding)."""
    from paper_2208_10859_gb300 import wv
    net = wv.CNN(seed=4)
    g = torch.Generator(device="cuda").manual_seed(2)
    x, t = (torch.rand((4, 130, 300), generator=g, device="cuda") for _ in range(2))
    loss, grads = net.gradients(x, t)
    for _ in range(2):
        net.set_wait_limit(0)
        net.gradients(x, t)
        assert net.sync_status() == WV_ERR_TIMEOUT
        net.set_wait_limit(1 << 20)
        loss2, grads2 = net.gradients(x, t)
        assert net.sync_status() == 0
        assert abs(loss2 - loss) <= 1e-5 * loss
        assert abs(grads2 - grads).max() <= 1e-4 * abs(grads).max()
    net.close()
