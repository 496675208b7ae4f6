"""The FP32 network on the tensor cores (three BF16 parts per value) against the network in
64 bits, where its tiles can go wrong: nets of 1 to 5 levels, channel counts that need 16- to
128-channel tiles (48 and 240 in tiles of 16, 256 in two of 128), pooling and concat convs at
each, frames smaller than a tile and ragged in both directions, batches whose tiles differ
from a single view's.

Tolerance: a layer's sums carry relative errors of at most about 3e-7 (9 truncations of a
chunk's accumulator and the FP32 additions of its chunks), 18 layers 1.3e-6 if they all add
up; logits stay below 8, and the sigmoid's slope is at most 1/4: 2 * 1.3e-6 rounded up to
4e-6 on outputs in [0, 1]."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

NETS = [
    ((48,), False, 40, 24, 1),
    ((16,), True, 136, 20, 2),
    ((16, 48), False, 130, 34, 2),
    ((240, 32), False, 66, 18, 1),
    ((16, 32, 64), True, 264, 136, 3),
    ((128, 256), False, 132, 70, 1),
    ((32, 64, 128, 256), False, 392, 216, 1),
    ((16, 16, 32, 128, 256), True, 272, 144, 2),
]


def net64(x, ch, w, bn):
    import torch
    import torch.nn.functional as F
    at = [0]

    def take(*s):
        n = int(np.prod(s))
        at[0] += n
        return torch.from_numpy(w[at[0] - n:at[0]].astype(np.float64)).view(*s)

    convs = [(take(co, ci, 3, 3), take(co)) for name, co, ci, _ in synth.weights.unet_layer_shapes(ch) if name != "head"]
    hw, hb = take(3, ch[0], 1, 1), take(3)
    if bn:
        for i in range(2 * len(ch)):
            g, be, mu, var = (take(ch[i // 2]) for _ in range(4))
            s = g / torch.sqrt(var + 1e-5)
            convs[i] = (convs[i][0] * s[:, None, None, None], (convs[i][1] - mu) * s + be)
    conv = lambda y, i: F.relu(F.conv2d(y, *convs[i], padding=1))  # noqa: E731
    y, skips, L = torch.from_numpy(x.astype(np.float64)).permute(2, 0, 1)[None], [], len(ch)
    for l in range(L):
        y = conv(conv(y, 2 * l), 2 * l + 1)
        if l < L - 1:
            skips.append(y)
            y = F.max_pool2d(y, 2)
    for k, l in enumerate(range(L - 2, -1, -1)):
        y = torch.cat([skips[l], F.interpolate(y, scale_factor=2, mode="nearest")], 1)
        y = conv(conv(y, 2 * L + 2 * k), 2 * L + 2 * k + 1)
    return torch.sigmoid(F.conv2d(y, hw, hb))[0].permute(1, 2, 0).numpy()


@pytest.mark.parametrize("ch,bn,W,H,B", NETS)
def test_fp32_net_against_64_bits(ch, bn, W, H, B):
    import paper_2502_11618_gb300 as lnr
    s = synth.room_scene(n_points=60_000, seed=4)
    r = lnr.Renderer(0)
    r.load_cloud(s.xyz, s.rgb, s.scan_id)
    r.build_grid(0.5)
    w = synth.unet_weights(ch, seed=6, has_bn=bn)
    r.set_unet(ch, w, "fp32", has_bn=bn)
    intr = synth.intrinsics_for(W, H)
    views = synth.random_poses(s, B, seed=12)
    y = r.render_batch(views, intr, W, H, 2, 1.0)
    for v, got in zip(views, y):
        assert np.array_equal(got, r.render(v, intr, W, H, 2, 1.0))
        x = r.render_stage(v, intr, W, H, 2, 1.0, lnr.STAGE_UNET_IN)
        assert np.abs(got - net64(x, ch, w, bn)).max() <= 4e-6
    r.close()
