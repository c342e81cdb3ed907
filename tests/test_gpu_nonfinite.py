"""Matching where the template or the search window holds NaN or infinite
pixels: no lag has a finite score, so the CP keeps its prior and reports
CFOG_CP_NONFINITE; every other CP of the launch returns the bytes it returns on
clean images.  All variants, both precisions, few and many CPs, and cfog_match."""
import numpy as np
import pytest

import synth
from tests._util import cuda_or_skip, to_dev

pytestmark = pytest.mark.gpu

N, R, MARK = 40, 6, (70, 71)   # (x, y) of the bad pixel; r < N / 2: every lag's window holds it
PTS = np.array([MARK, (160, 60), (60, 160), (150, 150)], np.int32)
VALUES = {"nan": np.nan, "inf": np.inf, "-inf": -np.inf}


def _features(torch, P, side, value):
    im = synth.batched_pair(5, size=220)
    A, B = im.A.copy(), im.B.copy()
    if side is not None:
        (A if side == "template" else B)[MARK[1], MARK[0]] = value
    return P.cfog_extract(to_dev(torch, A)), P.cfog_extract(to_dev(torch, B))


def _args(torch, copies):
    pts = torch.tensor(np.tile(PTS, (copies, 1)), device="cuda")
    full = lambda v: torch.full((len(pts),), v, dtype=torch.int32, device="cuda")
    return pts, full(N), full(R)


def _check(torch, P, got, clean, prior):
    L = P._lib
    d = {k: v.cpu().numpy() for k, v in P.unpack_results(got).items()}
    bad = np.arange(len(got)) % len(PTS) == 0
    assert (d["status"][bad] == L.CFOG_CP_NONFINITE).all()
    assert (d["dx"][bad] == prior[0]).all() and (d["dy"][bad] == prior[1]).all()
    assert (d["sub_dx"][bad] == prior[0]).all() and (d["sub_dy"][bad] == prior[1]).all()
    assert np.isposinf(d["ssd"][bad]).all()
    assert torch.equal(got.cpu()[~bad], clean.cpu()[~bad])


@pytest.mark.parametrize("value", list(VALUES))
@pytest.mark.parametrize("side", ["template", "window"])
@pytest.mark.parametrize("precision,variant", [(0, 1), (0, 2), (0, 3), (0, 4), (1, 0)])
def test_batched(precision, variant, side, value):
    torch, P = cuda_or_skip()
    out = []
    for s in (side, None):
        feats = _features(torch, P, s, VALUES[value])
        jobs = P.job_table([feats])
        for copies in (1, 200):
            pts, tm, rd = _args(torch, copies)
            prior = torch.tensor([[2, -1]], dtype=torch.int32, device="cuda").repeat(len(pts), 1)
            out.append(P.cfog_match_batched(jobs, 1, pts, tm, rd, N, R, prior=prior, precision=precision,
                                            variant=variant))
        torch.cuda.synchronize()   # feats outlives its launches
    for got, clean in zip(out[:2], out[2:]):
        _check(torch, P, got, clean, (2, -1))


@pytest.mark.parametrize("precision", [0, 1])
def test_single_pair(precision):
    torch, P = cuda_or_skip()
    pts, tm, rd = _args(torch, 1)
    feats = [_features(torch, P, s, np.nan) for s in ("window", None)]
    got, clean = (P.cfog_match(*f, pts, tm, rd, N, R, precision=precision) for f in feats)
    torch.cuda.synchronize()
    _check(torch, P, got, clean, (0, 0))
