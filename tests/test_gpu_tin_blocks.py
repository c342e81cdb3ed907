"""Piecewise-linear rectification (Sec. IV) where blocks of pixels are decided
at once: overlapping triangles whose lowest index must win, triangles wider
than a block, slivers, triangles that need 64-bit edge tests (extent above
16384), and outputs that end inside a block.  Against the oracle's per-pixel
first containing triangle."""
import numpy as np
import pytest

import oracle
import synth
from tests._util import cuda_or_skip
from tests.test_gpu_tin import NODATA, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("out_h,out_w", [(1, 1), (4, 32), (5, 33), (64, 64), (67, 95), (130, 201)])
@pytest.mark.parametrize("wide", [False, True])
def test_lowest_index_wins_over_blocks(out_h, out_w, wide):
    torch, P = cuda_or_skip()
    oracle.build()
    rng = np.random.default_rng(out_h * 1000 + out_w + wide)
    sen = synth.rect_texture(rng, 150, 230).astype(np.float32)
    n = 40
    pts = np.stack([rng.integers(0, out_w + 20, n), rng.integers(0, out_h + 20, n)], 1).astype(np.int32)
    if wide:   # a few vertices far outside the output
        pts[:6] = [(-9000, -8000), (9000, -8500), (-100, 9000), (17500, 40), (-20, 17000), (40, -17000)]
    d = rng.uniform(-3, 3, (n, 2))
    d[:6] *= 0.1
    res = np.zeros(n, dtype=synth.RESULT_DTYPE)
    res["sub_dx"], res["sub_dy"] = d[:, 0], d[:, 1]
    sen_xy = pts + np.stack([res["sub_dx"], res["sub_dy"]], 1).astype(np.float64)
    tris = rng.integers(0, n, (25, 3)).astype(np.int32)   # either orientation, some degenerate
    if wide:
        tris[12:16] = [(0, 1, 2), (3, 4, 0), (5, 3, 4), (0, 2, 1)]
    g = _run(torch, P, sen, pts, res, tris, out_h, out_w)
    o = oracle.tin_rectify(sen.astype(np.float64), pts, sen_xy, tris, out_h, out_w, NODATA)
    # the map of a triangle is evaluated in FP32 from one vertex: far vertices
    # cost position, so validity and values are compared away from the border
    # and to the slope of the image times 0.02 px
    both = (g != NODATA) & (o != NODATA)
    assert (both == (o != NODATA)).mean() > 0.99
    slope = 2 * max(np.abs(np.diff(sen, axis=0)).max(), np.abs(np.diff(sen, axis=1)).max())
    assert np.abs(g - o)[both].max(initial=0.0) <= 0.02 * slope
