"""Cells of subnormal size, powers of two and not: a quotient's exponent is then no sum of the
coordinate's and the cell's.  All points lie in one pixel at one depth, so that the front one is
the first in the grid's order, and its colour tells which that is."""
import numpy as np
import pytest

import oracle
import synth

TINY = 2.0 ** -1074  # the smallest subnormal
W = H = 64


def scene(cell, steps):
    """One point per entry of steps, that many cells along x from the frame's origin."""
    xyz = np.zeros((len(steps), 3))
    xyz[:, 0] = np.asarray(steps) * cell
    rgb = np.arange(3 * len(steps), dtype=np.uint8).reshape(-1, 3) + 1
    frame = (np.zeros(3), np.array([8, 1, 1], np.int32))
    view = synth.camera.View(np.array([[1.0, 0, 0], [0, -1.0, 0], [0, 0, -1.0]]), np.array([0.0, 0.0, 1.0]))
    return xyz, rgb, None, cell, frame, view, synth.intrinsics_for(W, H)


CASES = [(2.0 ** -1023, [1, 0, 3, 2]), (2.0 ** -1022, [1, 0, 3, 2]), (2.0 ** -1030, [2, 0, 1]), (3 * TINY, [3, 1, 0]),
         (2.0 ** -1000, [1, 0, 3, 2])]


def expected(cell, steps):
    xyz, rgb, sid, cell, frame, view, intr = scene(cell, steps)
    g = oracle.build_grid(xyz, rgb, sid, cell, frame)
    assert list(np.asarray(steps)[g.order]) == sorted(steps)
    return g, oracle.render(g, view, intr, W, H, 0, 1.0)["keys"]


@pytest.mark.parametrize("cell,steps", CASES)
def test_the_oracle_sees_the_points_in_order(cell, steps):
    keys = expected(cell, steps)[1]
    assert (keys != ~np.uint64(0)).sum() == 1 and (keys[keys != ~np.uint64(0)] & np.uint64(0xFFFFFFFF))[0] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("cell,steps", CASES)
def test_grid_order(cell, steps):
    import paper_2502_11618_gb300 as lnr

    xyz, rgb, sid, cell, frame, view, intr = scene(cell, steps)
    g, keys = expected(cell, steps)
    r = lnr.Renderer(0)
    r.load_cloud(xyz, rgb, sid)
    r.build_grid_frame(cell, *frame)
    got = r.render_stage(view, intr, W, H, 0, 1.0, lnr.STAGE_KEYS)
    assert np.array_equal(got, keys)
    colours, _, filled = r.render_stage(view, intr, W, H, 0, 1.0, lnr.STAGE_RGBDA_RAW)
    assert np.array_equal(colours[filled > 0], rgb[[int(np.argmin(steps))]])
    r.close()
