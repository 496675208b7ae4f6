"""The untuned choice of kernels changes how a network is run, never its results: frames of
the default configuration (tile, parity classes, epilogue warps and accumulator buffers from
the layer's size, level-0 encoder fused) equal those of one fixed configuration (the largest
double-buffered tile, staged stores, every conv apart), bit for bit.  The sizes reach tiles of
one row (few tiles), ragged tile edges, the single-buffered tiles of the wide layers and nets
with batch norm, of 2 and 5 levels."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_SCRIPT = r"""
import sys, numpy as np
sys.path.insert(0, {root!r})
import synth
import paper_2502_11618_gb300 as lnr
s = synth.multiroom_scene(n_points=200_000)
r = lnr.Renderer(0); r.load_cloud(s.xyz, s.rgb, s.scan_id); r.build_grid(0.25)
out = []
for ch, bn, W, H, B, prec in {cases!r}:
    r.set_unet(ch, synth.unet_weights(ch, seed=3, has_bn=bn), "bf16", has_bn=bn)
    intr = synth.intrinsics_for(W, H)
    views = synth.random_poses(s, B + 1, seed=8)
    if prec == "fp8":
        r.calibrate(views[B], intr, W, H, 3, 1.0)
        r.set_precision("fp8")
    out.append(r.render_batch(views[:B], intr, W, H, 3, 1.0).ravel())
np.save(sys.argv[1], np.concatenate(out))
"""
CH4 = (32, 64, 128, 256)
CASES = {
    "small": [(CH4, False, 128, 96, 1, "bf16"), ((16, 32, 64), True, 64, 48, 3, "bf16"), ((32, 64), False, 130, 34, 2, "bf16")],
    "ragged": [(CH4, True, 392, 216, 3, "bf16"), ((16, 32, 64, 128, 256), False, 272, 144, 2, "bf16")],
    "waves": [(CH4, False, 1288, 728, 2, "bf16"), ((16, 32, 64), False, 1288, 728, 1, "bf16")],
    "fp8": [(CH4, False, 264, 136, 1, "fp8"), (CH4, True, 648, 368, 3, "fp8")],
}


@pytest.mark.parametrize("case", list(CASES))
def test_untuned_choice_keeps_every_bit(tmp_path, case):
    got = {}
    for tag, extra in (("default", {}), ("fixed", {"LNR_CONV_TMA_STORE": "2"})):
        env = {k: v for k, v in os.environ.items() if not k.startswith("LNR_CONV")}
        env.update(extra)
        path = str(tmp_path / f"{tag}.npy")
        r = subprocess.run([sys.executable, "-c", _SCRIPT.format(root=ROOT, cases=CASES[case]), path], env=env,
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stdout + r.stderr
        got[tag] = np.load(path)
    assert np.isfinite(got["fixed"]).all()
    assert np.array_equal(got["default"], got["fixed"])
