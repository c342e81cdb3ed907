"""The FFT matcher's launch geometries and staging paths (Eq. 5-9): every FFT
length with compile-time radices and lengths that take the run-time path, CPs
on the image border, volumes whose rows are not 16-byte aligned, and the same
CP in a launch of few CPs (512-thread CTAs) and of many (256-thread CTAs).
Parity with the oracle by the suite's rules; equal bytes between geometries
and between alignments, since no sum's order depends on either."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests._util import check_match_parity, cuda_or_skip, gpu_results, to_dev

pytestmark = pytest.mark.gpu

# W = N + 2r just below and above the compiled lengths 48..180, a run-time
# length (24, 192), blocked plans, odd sides
CLASSES = [(16, 4), (31, 8), (32, 8), (33, 9), (44, 8), (49, 11), (64, 8), (65, 7), (63, 16),
           (88, 3), (80, 10), (84, 12), (96, 12), (97, 15), (100, 22), (112, 20), (150, 15), (160, 16)]


@pytest.fixture(scope="module")
def pair():
    torch, P = cuda_or_skip()
    oracle.build()
    im = synth.batched_pair(71, size=301)
    A, B = im.A[:281], im.B[:281]
    fa, fb = P.cfog_extract(to_dev(torch, A)), P.cfog_extract(to_dev(torch, B))
    return torch, P, fa, fb, oracle.cfog(A)[0], oracle.cfog(B)[0]


def _cps(N, r):
    """Centre, and the four corners of the region the window stays inside."""
    t0 = N // 2
    xs = (150, t0 + r, 301 - (N - t0) - r)
    ys = (140, t0 + r, 281 - (N - t0) - r)
    return np.array([(xs[0], ys[0])] + [(x, y) for x in xs[1:] for y in ys[1:]], np.int32)


def _run(torch, P, fa, fb, pts, N, r, variant, copies=1):
    pts = np.tile(pts, (copies, 1))
    n = len(pts)
    jobs = P.job_table([(fa, fb)])
    res = P.cfog_match_batched(jobs, 1, torch.tensor(pts, device="cuda"),
                               torch.full((n,), N, dtype=torch.int32, device="cuda"),
                               torch.full((n,), r, dtype=torch.int32, device="cuda"), N, r, variant=variant)
    torch.cuda.synchronize()
    return res


def _unaligned(torch, f):
    """The same volume at row pitch w (not a multiple of 4) from an address 4 bytes off."""
    rp, pp = f.w, f.w * f.h
    data = torch.empty(f.m * pp + 1, device="cuda")[1:]
    data.as_strided((f.m, f.h, f.w), (pp, rp, 1), data.storage_offset()).copy_(f.volume())
    sq = torch.empty(f.h * rp, device="cuda")
    sq.as_strided((f.h, f.w), (rp, 1)).copy_(f.sq())
    return dataclasses.replace(f, data=data, sqnorm=sq, row_pitch=rp, plane_pitch=pp)


@pytest.mark.parametrize("variant", [1, 2, 3, 4])
@pytest.mark.parametrize("N,r", CLASSES)
def test_class_parity_and_equal_bytes(pair, N, r, variant):
    torch, P, fa, fb, da, db = pair
    pts = _cps(N, r)
    few = _run(torch, P, fa, fb, pts, N, r, variant)
    o = oracle.match_many(da, db, pts[:, 0], pts[:, 1], np.full(len(pts), N), np.full(len(pts), r))
    check_match_parity(gpu_results(P, few), o)
    copies = 2 * torch.cuda.get_device_properties(0).multi_processor_count // len(pts) + 1
    many = _run(torch, P, fa, fb, pts, N, r, variant, copies)
    assert torch.equal(many, few.repeat(copies, 1))
    loose = _run(torch, P, _unaligned(torch, fa), _unaligned(torch, fb), pts, N, r, variant)
    assert torch.equal(loose, few)
