"""A job's rejection does not depend on its neighbours: jobs on both sides of the
size (2048 CPs) from which a job takes more threads, alone and in one launch, with
the same bytes; the mixed launch is complete for what follows on its stream."""
import numpy as np
import pytest

import synth
from tests._util import cuda_or_skip

pytestmark = pytest.mark.gpu

SIZES = [700, 2047, 2048, 0, 300, 2600, 1500, 12000, 57]


def _dev(torch, cps, res):
    r = np.ascontiguousarray(res).view(np.int32).reshape(-1, 6)
    return torch.from_numpy(cps.astype(np.int32)).cuda(), torch.from_numpy(r.copy()).cuda()


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("seed", [200, 220])
def test_job_alone_and_with_neighbours(seed, degree):
    torch, P = cuda_or_skip()
    sets = [synth.cp_set(seed + k, n, noise=0.05, outlier_frac=0.05) for k, n in enumerate(SIZES)]
    start = np.concatenate([[0], np.cumsum(SIZES)]).tolist()
    c, r = _dev(torch, np.concatenate([s[0] for s in sets]), np.concatenate([s[1] for s in sets]))
    keep, order, models = (t.clone() for t in P.cfog_reject_outliers(c, r, start, degree, 0.25))
    torch.cuda.synchronize()
    together = P.unpack_models(models)
    removed = 0
    for j, (a, b) in enumerate(zip(start, start[1:])):
        if a == b:
            continue
        k1, o1, m1 = P.cfog_reject_outliers(c[a:b].contiguous(), r[a:b].contiguous(), None, degree, 0.25)
        torch.cuda.synchronize()
        n = together[j]["n_removed"]
        removed += n
        assert P.unpack_models(m1)[0] == together[j]
        assert torch.equal(k1, keep[a:b])
        assert torch.equal(o1[:n], order[a:a + n] - a)
    assert removed > 100


@pytest.mark.parametrize("decades", [(-4, 4), (-6, 1)])
def test_many_jobs_with_and_without_a_large_one(decades):
    """2000 jobs of residuals over many magnitudes, whose sums of squares round by the
    order of the terms, with and without a job of 2500 CPs in the launch."""
    torch, P = cuda_or_skip()
    rng = np.random.default_rng(5)
    sizes = [int(v) for v in rng.integers(1800, 2047, 2000)] + [2500]
    n = sum(sizes)
    cps = rng.integers(0, 20000, (n, 2)).astype(np.int32)
    res = np.zeros(n, dtype=synth.RESULT_DTYPE)
    for f in ("sub_dx", "sub_dy"):
        res[f] = 10.0 ** rng.uniform(*decades, n) * rng.choice([-1.0, 1.0], n)
    start = np.concatenate([[0], np.cumsum(sizes)]).tolist()
    c, r = _dev(torch, cps, res)
    end = start[-2]
    _, _, both = P.cfog_reject_outliers(c, r, start, 1, 1e9)
    _, _, small = P.cfog_reject_outliers(c[:end].contiguous(), r[:end].contiguous(), start[:-1], 1, 1e9)
    assert P.unpack_models(both)[:2000] == P.unpack_models(small)
