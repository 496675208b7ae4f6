"""The device grid build against the oracle's, bit for bit, where its shortcuts can go wrong:
cell quotients on and one ulp around whole numbers (cells that are and are not powers of two,
with georeferenced coordinates), clouds of one point and around a sort tile's 4096, one cell
and many, axes with more cells than the origins' table holds, points outside a given frame,
and coordinates of either sign.  The cells and offsets show in the z-buffer's keys (depth
bits, sorted position), the colours and the cull counts of a view over the whole cloud."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def cloud(n, cell, seed, georef, span=20):
    """Points over span x span x 1 cells: a third anywhere, the rest on multiples of the cell
    along an axis or one ulp beside."""
    rng = np.random.default_rng(seed)
    off = np.array([512000.0, -5600000.0, 100.0]) if georef else np.array([-3.0, 2.0, 0.0])
    g0 = np.floor(off / cell) * cell
    k = rng.integers(0, span, (n, 3)) * np.array([1, 1, 0])
    xyz = g0 + (k + rng.uniform(0, 1, (n, 3))) * cell
    near = rng.integers(0, 3, n) > 0
    on = g0 + k * cell
    side = rng.integers(-1, 2, (n, 3))
    on = np.where(side < 0, np.nextafter(on, -np.inf), np.where(side > 0, np.nextafter(on, np.inf), on))
    ax = rng.integers(0, 2, n)
    xyz[near, ax[near]] = on[near, ax[near]]
    return xyz, rng.integers(0, 256, (n, 3), dtype=np.uint8), rng.integers(0, 4, n, dtype=np.uint8)


def check(xyz, rgb, sid, cell, frame=None):
    import paper_2502_11618_gb300 as lnr
    W = H = 256
    lo, hi = xyz.min(0), xyz.max(0)
    size = max(float((hi - lo)[:2].max()), cell)
    intr = synth.intrinsics_for(W, H, zfar=100.0 * size)
    view = synth.camera.View(np.array([[1.0, 0, 0], [0, -1.0, 0], [0, 0, -1.0]]),
                             np.array([*((lo + hi) / 2)[:2], hi[2] + size]))  # straight down on all of it
    g = oracle.build_grid(xyz, rgb, sid, cell, frame)
    r = lnr.Renderer(0)
    r.load_cloud(xyz, rgb, sid)
    if frame is None:
        r.build_grid(cell)
    else:
        r.build_grid_frame(cell, *frame)
    g0, dims = r.grid_info()
    assert np.array_equal(g0, g.g0) and np.array_equal(dims, g.dims)
    ref = oracle.render(g, view, intr, W, H, 0, 1.0)
    keys = r.render_stage(view, intr, W, H, 0, 1.0, lnr.STAGE_KEYS)
    assert (keys != ~np.uint64(0)).any()
    assert np.array_equal(keys, ref["keys"])
    rgb_g, d, a = r.render_stage(view, intr, W, H, 0, 1.0, lnr.STAGE_RGBDA_RAW)
    rgb_o, d_o, a_o = oracle.resolve(ref["keys"], g.rgbs, W, H)[:3]
    assert np.array_equal(np.asarray(rgb_g).reshape(-1), np.asarray(rgb_o).reshape(-1))
    vp = oracle.view_params(g, view.R, view.C)
    vis, _ = oracle.cull(g, vp, intr, W, H)
    cells, points = r.render_stage(view, intr, W, H, 0, 1.0, lnr.STAGE_CULL)
    counts = np.diff(g.cell_start.astype(np.int64))
    assert cells == int(((vis == 1) & (counts > 0)).sum()) and points == int(counts[vis == 1].sum())
    r.close()


@pytest.mark.parametrize("cell", [0.1, 0.25, 1.0 / 3.0, 0.7, 1.0, 3.0])
@pytest.mark.parametrize("georef", [False, True])
def test_quotients_near_whole_numbers(cell, georef):
    check(*cloud(60_000, cell, 3, georef), cell)


@pytest.mark.parametrize("n", [1, 2, 255, 4095, 4096, 4097, 12_289])
def test_cloud_sizes(n):
    check(*cloud(n, 0.3, n, False), 0.3)


def test_one_cell_and_a_long_axis():
    xyz, rgb, sid = cloud(5000, 0.25, 8, False)
    check(xyz, rgb, sid, 1000.0)
    xyz[:, 0] = np.linspace(-1000.0, 1000.0, 5000)   # 80001 cells along x: no origins' table
    check(xyz, rgb, sid, 0.025)


def test_points_outside_a_given_frame():
    xyz, rgb, sid = cloud(20_000, 0.5, 5, True)
    g0 = np.floor((xyz.min(0) + 2.0) / 0.5) * 0.5
    check(xyz, rgb, sid, 0.5, (g0, np.array([9, 11, 1], np.int32)))
