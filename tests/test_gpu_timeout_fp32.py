"""The bounded waits of the FP32 network's convolutions, as test_gpu_timeout.py has them for BF16:
the MMA issuers of the first launch give up after ~1 ms, its other warps after ~2 s, the kernel
ends, and the error goes to the context that made the launch.  Nets whose first convolution takes
tiles of one and of several rows, with the frame left on the device and with one that waits."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

_SCRIPT = r"""
import sys, numpy as np
sys.path.insert(0, {root!r})
import torch
import synth
import paper_2502_11618_gb300 as lnr
s = synth.room_scene(n_points=60_000, seed=0)
W, H, on_device = {W}, {H}, {on_device}
ch = (16, 32, 64)
intr = synth.intrinsics_for(W, H)
view = synth.random_poses(s, 1, seed=2)[0]
def make():
    r = lnr.Renderer(0)
    r.load_cloud(s.xyz, s.rgb, s.scan_id); r.build_grid(0.5); r.set_unet(ch, synth.unet_weights(ch, seed=1), "fp32")
    return r
a, b = make(), make()
def frame(r):
    return r.render(view, intr, W, H, 3, 1.0)
if on_device:
    a.render(view, intr, W, H, 3, 1.0, out=torch.empty((H, W, 3), device="cuda"))
    want = frame(b)                          # another context's frame is its own
try:
    frame(a)
    print("no timeout"); sys.exit(2)
except lnr.LnrError as e:
    assert e.status == -5, e
if not on_device:
    want = frame(b)
assert np.isfinite(want).all() and want.std() > 0
for _ in range(4):                           # eager, then the captured graph
    assert np.array_equal(frame(a), want)
print("recovered")
a.close(), b.close()
"""


@pytest.mark.parametrize("W,H,on_device", [(128, 96, False), (640, 480, True)])
def test_bounded_waits_run_out_and_the_context_recovers(W, H, on_device):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LNR_TEST_STALL_ONCE="1")
    r = subprocess.run([sys.executable, "-c", _SCRIPT.format(root=root, W=W, H=H, on_device=on_device)], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "recovered" in r.stdout
