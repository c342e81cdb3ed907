"""Block-based Harris detection (Sec. IV) at the edges of its warp strips: chip
widths around one, two and three strips of 56 and 88 columns, row segments of
one row and more, cells on the image border, one and eight points per cell.
Every point against the oracle's responses (the k best, near-ties allowed)."""
import numpy as np
import pytest

import oracle
import synth
from tests._util import cuda_or_skip, to_dev

pytestmark = pytest.mark.gpu

# (h, w, grid_y, grid_x, margin): cell sides 1, 7, 55..57, 87..89, 112, 113, 177, 256
CASES = [(9, 12, 9, 12, 0), (35, 42, 5, 6, 0), (55, 57, 1, 1, 0), (112, 114, 2, 2, 0),
         (130, 131, 2, 2, 8), (88, 89, 1, 1, 0), (200, 202, 2, 2, 11), (112, 113, 1, 1, 0),
         (190, 450, 1, 2, 6), (256, 256, 1, 1, 0), (300, 276, 2, 1, 10)]


@pytest.mark.parametrize("dtype", ["f32", "u16"])
@pytest.mark.parametrize("k", [1, 3, 8])
@pytest.mark.parametrize("h,w,gy,gx,margin", CASES)
def test_points_are_the_best_of_their_cells(h, w, gy, gx, margin, k, dtype):
    torch, P = cuda_or_skip()
    oracle.build()
    A = synth.rect_texture(np.random.default_rng(h * 1000 + w), h, w).astype(np.float32)
    if dtype == "u16":
        A = np.rint(A * 16).astype(np.uint16)
    resp = oracle.harris(A.astype(np.float64))
    pts = P.cfog_detect_cps(to_dev(torch, A), gx, gy, k, 0, margin).cpu().numpy()
    ox, oy = oracle.detect(resp, gx, gy, k, 0, margin)
    for c in range(gx * gy):
        y0, y1, x0, x1 = oracle.cell_chip(h, w, gx, gy, 0, margin, *divmod(c, gx))
        scale = np.abs(resp[y0:y1, x0:x1]).max() + 1e-30
        got = [tuple(p) for p in pts[c * k:(c + 1) * k]]
        n = min(k, (y1 - y0) * (x1 - x0))
        assert got[n:] == [(-1, -1)] * (k - n)
        assert len(set(got[:n])) == n
        for (x, y), qx, qy in zip(got[:n], ox[c * k:], oy[c * k:]):
            assert x0 <= x < x1 and y0 <= y < y1
            assert (x, y) == (qx, qy) or abs(resp[y, x] - resp[qy, qx]) <= 1e-5 * scale
