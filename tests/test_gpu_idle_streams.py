"""Internal CUDA streams of closed streams: handed to the streams opened next,
never more than 16 of them, and given back to CUDA when the last open stream of
the device is closed (so that nothing of the library outlives its objects, and
a context torn down between two uses leaves no stale handles behind).  In a
child process, where no other test holds a stream open."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SCRIPT = r'''
import math, sys
import torch
sys.path.insert(0, ROOT)
sys.path.insert(0, HERE)
from paper_2208_10859_gb300 import wv
import helpers as H

idle = lambda: wv._lib().wv_debug_idle_streams(0)
data = H.case("yuv97")[2]

def use(s):
    outs = [torch.zeros((48, 64, 4), dtype=torch.uint8, device="cuda") for _ in range(5)]
    for k, o in enumerate(outs):
        s.decode_viewport(0, 0.3 * k, 0.1, math.radians(100), o)
    torch.cuda.synchronize()
    return outs

assert idle() == 0
a, b = wv.Stream(data), wv.Stream(data)
want = use(a)
a.close()
assert 0 < idle() <= 4, idle()          # b is open: a's are kept
got = use(b)                            # and serve b
assert idle() == 0, idle()
assert all(torch.equal(x, y) for x, y in zip(want, got))
many = [wv.Stream(data) for _ in range(6)]
for s in many:
    use(s)
for s in many:
    s.close()
assert idle() == 16, idle()             # 24 came back
b.close()
assert idle() == 0, idle()              # the last one is closed
c = wv.Stream(data)                     # and the next one makes its own
got = use(c)
assert all(torch.equal(x, y) for x, y in zip(want, got)) and c.sync_status() == 0
c.close()
assert idle() == 0
print("idle ok")
'''


def test_idle_streams_are_bounded_and_given_back():
    script = f"ROOT = {ROOT!r}\nHERE = {HERE!r}\n" + SCRIPT
    r = subprocess.run([sys.executable, "-c", script], cwd=HERE, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "idle ok" in r.stdout
