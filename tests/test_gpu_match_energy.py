"""Matching of features whose norm is not 1: volumes scaled up and down, CFOG whose
eps outweighs the gradients, windows that are constant but for a patch.  Scores,
surfaces and sub-pixel offsets against the oracle on the GPU's own features.

Tolerance of a score: 2e-6 of the energies it is the difference of (sum T^2 plus the
largest window energy of the surface).  One FP32 rounding at that size is 6e-8; the
transforms add a few 2^-24 of it per level, about fourteen levels in the two
directions and axes."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests._util import TIE_REL, cuda_or_skip, to_dev

pytestmark = pytest.mark.gpu

REL = 2e-6
SUBPIX = 0.01
SIZE = 260
PTS = np.array([(130, 131), (101, 117), (150, 160)], np.int32)


def _images():
    im = synth.batched_pair(17, size=SIZE)
    return im.A.astype(np.float32), im.B.astype(np.float32)


def _patch():
    """Both images constant but for 40 x 36 pixels in the middle, moved by (2, -3)."""
    A, _ = _images()
    out = []
    for y, x in ((110, 112), (108, 115)):
        im = np.full((SIZE, SIZE), 100.0, np.float32)
        im[y:y + 40, x:x + 36] = A[60:100, 60:96]
        out.append(im)
    return out


def _scaled(f, s):
    return dataclasses.replace(f, data=f.data * s, sqnorm=f.sqnorm * (s * s))


def _check(torch, P, fa, fb, pts, N, r):
    da, db = fa.volume().double().cpu().numpy(), fb.volume().double().cpu().numpy()
    n = len(pts)
    full = lambda v, k: torch.full((k,), v, dtype=torch.int32, device="cuda")
    cps, L = torch.tensor(pts, device="cuda"), 2 * r + 1
    surf = torch.empty((n, L, L), device="cuda")
    one = P.cfog_match(fa, fb, cps, full(N, n), full(r, n), N, r, surface=surf)
    jobs = P.job_table([(fa, fb)])
    many = [P.cfog_match_batched(jobs, 1, cps.repeat(c, 1), full(N, c * n), full(r, c * n), N, r, variant=v)[:n]
            for v in (1, 2, 3, 4) for c in (1, 300)]
    torch.cuda.synchronize()
    surf = surf.cpu().numpy().astype(np.float64)
    for i, (x, y) in enumerate(pts):
        S, E = oracle.ssd_surface(da, db, int(x), int(y), N, r)
        o = oracle.match_one(da, db, int(x), int(y), N, r)
        tol = REL * E.max()      # E = sum T^2 + B(v)
        assert np.abs(surf[i] - S).max() <= tol, np.abs(surf[i] - S).max() / E.max()
        for res in [one] + many:
            g = {k: v[i].item() for k, v in P.unpack_results(res).items()}
            assert abs(g["ssd"] - o["ssd"]) <= tol
            if o["gap_rel"] < TIE_REL:
                continue
            assert (g["dx"], g["dy"], g["status"]) == (o["dx"], o["dy"], o["status"])
            if o["status"] == 0:
                assert abs(g["sub_dx"] - o["sub_dx"]) <= SUBPIX and abs(g["sub_dy"] - o["sub_dy"]) <= SUBPIX


@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e-2, 1e3, 1e6])
def test_scaled_volumes(scale):
    torch, P = cuda_or_skip()
    oracle.build()
    fa, fb = (_scaled(P.cfog_extract(to_dev(torch, im)), scale) for im in _images())
    _check(torch, P, fa, fb, PTS, 64, 12)


@pytest.mark.parametrize("times", [1, 10, 100, 1000])
def test_eps_outweighs_the_gradients(times):
    torch, P = cuda_or_skip()
    oracle.build()
    A, B = _images()
    p = P.default_params()
    p.eps = float(times * np.abs(np.gradient(A)).mean())
    fa, fb = (P.cfog_extract(to_dev(torch, im), p) for im in (A, B))
    _check(torch, P, fa, fb, PTS, 96, 16)


def test_windows_constant_but_for_a_patch():
    torch, P = cuda_or_skip()
    oracle.build()
    fa, fb = (P.cfog_extract(to_dev(torch, im)) for im in _patch())
    _check(torch, P, fa, fb, np.array([(128, 130), (120, 122)], np.int32), 160, 16)


@pytest.mark.parametrize("at,gain", [((20, 21), 1e5), ((20, 21), 100.0), ((22, 22), 1e5), ((22, 22), 200.0),
                                     ((21, 15), 1e5), ((21, 15), 200.0)])
def test_template_energy_in_a_few_pixels(at, gain):
    """Energy that a sample of the 64 x 64 template misses (even rows) or takes for
    typical (a sampled pixel, row 21 and column 15)."""
    torch, P = cuda_or_skip()
    oracle.build()
    fa, fb = (P.cfog_extract(to_dev(torch, im)) for im in _images())
    fa = _scaled(fa, 1.0)
    k = 2 if at == (20, 21) else 1
    y, x = PTS[0, 1] - 32 + at[0], PTS[0, 0] - 32 + at[1]
    fa.volume()[:, y:y + k, x:x + k] *= gain
    _check(torch, P, fa, fb, PTS[:1], 64, 12)
