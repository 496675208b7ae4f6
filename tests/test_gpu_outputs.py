"""Networks with one, two and three outputs: the head's outputs are independent sums, so that a
network with fewer of them gives the same first ones, bit for bit, through every call."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

CH = (16, 32, 64)
W, H, NL, FS = 136, 72, 3, 1.0


def weights(o):
    """The first o outputs of the three-output network."""
    w = synth.unet_weights(CH, seed=1)
    head = len(w) - 3 * CH[0] - 3
    return np.concatenate([w[:head], w[head:head + o * CH[0]], w[-3:][:o]])


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_fewer_outputs_are_the_first_of_three(prec):
    import paper_2502_11618_gb300 as lnr

    s = synth.room_scene(n_points=60_000, seed=0)
    intr = synth.intrinsics_for(W, H)
    views = synth.random_poses(s, 3, seed=2)
    r = lnr.Renderer(0)
    r.load_cloud(s.xyz, s.rgb, s.scan_id)
    r.build_grid(0.5)
    r.set_unet(CH, weights(3), prec)
    want = r.render_batch(views, intr, W, H, NL, FS)
    for o in (1, 2):
        r.set_unet(CH, weights(o), prec, out_ch=o)
        assert np.array_equal(r.render_batch(views, intr, W, H, NL, FS), want[..., :o])
        assert np.array_equal(r.render(views[1], intr, W, H, NL, FS), want[1, ..., :o])
        r.serve_start(max_batch=3, slots=2)
        out = [np.zeros((H, W, o), np.float32) for _ in views]
        tickets = [r.submit_into(v, intr, W, H, NL, FS, b) for v, b in zip(views, out)]
        while tickets:
            tickets = [t for t in tickets if r.poll(t)[1] is None]
        r.serve_stop()
        assert all(np.array_equal(b, f) for b, f in zip(out, want[..., :o]))
    r.close()
