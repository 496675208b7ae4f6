"""lnr_filter_static's fused upsampling against the oracle's depth filter, bit for bit: image
sizes around its 64 x 64 tiles and odd at every level, all level counts, sparse and dense depth
with holes at the borders, in place, and strengths that keep nothing, some and everything."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 3), (63, 64), (64, 64), (65, 63), (66, 130), (127, 129), (191, 97), (333, 201), (640, 361)]


@pytest.mark.parametrize("W,H", SIZES)
def test_every_level_count(W, H):
    import torch

    import paper_2502_11618_gb300 as lnr
    fn = lnr.lib().lnr_filter_static
    rng = np.random.default_rng(W * 1000 + H)
    y, x = np.mgrid[0:H, 0:W]
    for n in range(0, min(6, int(np.log2(min(W, H)))) + 1):
        for fill, fs in ((0.05, 1.0), (0.4, 0.5), (0.95, 0.0), (0.4, 1e6)):
            D = (2.0 + 0.01 * x + 0.02 * y + 3.0 * (rng.random((H, W)) < 0.3)).astype(np.float32)
            D[rng.random((H, W)) >= fill] = np.inf
            want = oracle.depth_filter(D, n, fs)
            d = torch.from_numpy(D).cuda()
            for kept in (torch.full_like(d, -1.0), d):
                st = fn(ctypes.c_void_p(d.data_ptr()), W, H, n, ctypes.c_float(fs), ctypes.c_void_p(kept.data_ptr()),
                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
                assert st == 0
                assert np.array_equal(kept.cpu().numpy(), want), (n, fill, fs)
