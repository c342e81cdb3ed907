"""Which pixels a rectification fills, in both directions: exactly those in some
triangle, since the sensed image reaches beyond every mapped pixel and the edge tests
are exact.  Overlapping triangles of either orientation, outputs that end inside a
32 x 4 block, triangles with far vertices."""
import numpy as np
import pytest

import oracle
import synth
from tests._util import cuda_or_skip
from tests.test_gpu_tin import NODATA, _run

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24
PAD = 40    # of the sensed image beyond the output and the CPs around it


def _tolerance(pts, sen_xy, tris, out_h, out_w, rng_val):
    """Per pixel, from the triangle that fills it: 1e-4 of the image range, and what three
    FP32 roundings of the map's terms J (q - a) move the sample, at most the range per
    pixel along either axis."""
    y, x = np.mgrid[:out_h, :out_w].astype(np.int64)
    lim = np.zeros((out_h, out_w))
    p = pts.astype(np.int64)
    for t in tris[::-1]:   # the first triangle of the list wins
        a, b, c = (p[i] for i in t)
        if (b[0] - a[0]) * (c[1] - a[1]) - (b[1] - a[1]) * (c[0] - a[0]) <= 0:
            continue
        inside = np.ones(x.shape, bool)
        for u, v in ((a, b), (b, c), (c, a)):
            inside &= (v[0] - u[0]) * (y - u[1]) - (v[1] - u[1]) * (x - u[0]) >= 0
        e = np.stack([b - a, c - a], 1).astype(np.float64)
        s = np.stack([sen_xy[t[1]] - sen_xy[t[0]], sen_xy[t[2]] - sen_xy[t[0]]], 1)
        terms = np.abs(s @ np.linalg.inv(e)).max() * (np.abs(x - a[0]) + np.abs(y - a[1]))
        lim[inside] = rng_val * (1e-4 + 2 * 3 * EPS * (1 + terms[inside]))
    return lim


@pytest.mark.parametrize("out_h,out_w", [(1, 1), (4, 32), (5, 33), (64, 64), (67, 95), (130, 201)])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("n_tris", [3, 25, 60])
def test_filled_pixels(out_h, out_w, wide, n_tris):
    torch, P = cuda_or_skip()
    oracle.build()
    rng = np.random.default_rng(out_h * 1000 + out_w + 7 * n_tris + wide)
    sen = synth.rect_texture(rng, out_h + 20 + 2 * PAD, out_w + 20 + 2 * PAD).astype(np.float32)
    n = 40
    pts = np.stack([rng.integers(0, out_w + 20, n), rng.integers(0, out_h + 20, n)], 1).astype(np.int32)
    d = np.full((n, 2), PAD / 2) + rng.uniform(-3, 3, (n, 2))
    if wide:   # their offsets differ by less, so that pixels between them stay inside
        pts[:6] = [(-9000, -8000), (9000, -8500), (-100, 9000), (17500, 40), (-20, 17000), (40, -17000)]
    res = np.zeros(n, dtype=synth.RESULT_DTYPE)
    res["sub_dx"], res["sub_dy"] = d[:, 0], d[:, 1]
    sen_xy = pts + np.stack([res["sub_dx"], res["sub_dy"]], 1).astype(np.float64)
    tris = rng.integers(0, n, (n_tris, 3)).astype(np.int32)
    if wide:
        tris[-2:] = [(0, 1, 2), (5, 3, 4)]
    g = _run(torch, P, sen, pts, res, tris, out_h, out_w)
    o = oracle.tin_rectify(sen.astype(np.float64), pts, sen_xy, tris, out_h, out_w, NODATA)
    np.testing.assert_array_equal(g != NODATA, o != NODATA)
    both = o != NODATA
    if out_h >= 64 and n_tris > 3:
        assert both.sum() >= both.size // 4
    if not wide:   # far vertices cost position: their values are compared elsewhere
        lim = _tolerance(pts, sen_xy, tris, out_h, out_w, float(sen.max()) - float(sen.min()))
        assert (np.abs(g - o)[both] <= lim[both]).all()
