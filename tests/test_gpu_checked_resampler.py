"""The bounds-check build (WV_CHECKED) runs the resampler that viewports and
batches run, with its word loads checked: for every channel layout, at poses over
the seam and both poles and at odd output sizes, its kernels (by name, from the
profiler) are the tap-pair ones, they give the pixels of the general resampler
(which takes the same positions from memory, one byte per tap), and no check
fires.  In a child process, which loads the checked library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SCRIPT = r'''
import math, sys
import numpy as np
import torch
from torch.profiler import ProfilerActivity, profile
sys.path.insert(0, ROOT)
from paper_2208_10859_gb300 import build, wv
assert wv.lib_path() == build.LIB_CHECKED
build.build(checked=True)

def stream(w, h, planes, c420, levels, stereo):
    rng = np.random.default_rng(w + h + planes)
    frame = []
    for p in range(planes):
        s = 2 if p and c420 else 1
        frame.append(torch.tensor(rng.integers(0, 256, (h // s, w // s), dtype=np.uint8), device="cuda"))
    d = dict(width=w, height=h, planes=planes, chroma_420=c420, levels=levels, wavelet=1, num_frames=1, tlevels=0,
             block=32, quant=0, step=1.0, stereo=stereo)
    return wv.Stream(wv.encode([tuple(frame)], d))

names = set()
for w, h, planes, c420, levels, stereo, mode in [
        (64, 64, 1, 0, 3, 0, 0), (256, 160, 3, 1, 3, 0, 0), (256, 160, 3, 1, 3, 0, 2), (320, 160, 3, 0, 3, 0, 0),
        (320, 160, 3, 0, 2, 0, 0), (256, 192, 3, 1, 4, 1, 0)]:
    s = stream(w, h, planes, c420, levels, stereo)
    s.set_decode_mode(mode)
    for ow, oh in ((64, 48), (131, 77)):
        for yaw, pitch in ((0.0, 0.0), (math.pi, 0.3), (0.7, 1.55), (-2.0, -1.5)):
            fov = math.radians(100)
            out = torch.zeros((oh, ow, 4), dtype=torch.uint8, device="cuda")
            want = torch.zeros_like(out)
            batch = torch.zeros_like(out)
            with profile(activities=[ProfilerActivity.CUDA]) as prof:
                s.decode_viewport(0, yaw, pitch, fov, out)
                wv.decode_batch([wv.ViewRequest(s, 0, yaw, pitch, fov, batch)])
                torch.cuda.synchronize()
            names |= {e.key for e in prof.key_averages() if "k_resample" in e.key}
            if not stereo:
                s.resample_at(s.debug_project(yaw, pitch, fov, ow, oh), want)
                torch.cuda.synchronize()
                assert torch.equal(out, want), (w, h, planes, c420, mode, ow, oh, yaw, pitch)
            assert torch.equal(out, batch)
            assert int(out[..., 3].min()) == 255 and float(out[..., :3].float().std()) > 5
    assert s.sync_status() == 0
    s.close()
print(sorted(names))
assert names and not any("general" in n for n in names), names
assert any("k_resample_batch" in n for n in names), names
assert len([n for n in names if "k_resample<" in n]) == 5, names     # every channel layout
print("checked ok")
'''


def test_checked_build_runs_the_resampler_of_the_viewports():
    env = dict(os.environ, WV_CHECKED="1")
    script = f"ROOT = {ROOT!r}\n" + SCRIPT
    r = subprocess.run([sys.executable, "-c", script], env=env, cwd=HERE, capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "checked ok" in r.stdout
