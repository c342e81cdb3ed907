"""Windows in which more lags tie than the nomination buffer holds (64): a
structureless pair, whose every lag scores zero, and a periodic pair, where every
fourth lag along both axes is an exact match.  The reported lag depends neither
on timing nor on the launch's geometry."""
import numpy as np
import pytest

from tests._util import cuda_or_skip, to_dev

pytestmark = pytest.mark.gpu

COPIES = 400
PTS = [(100, 100), (90, 111), (77, 83)]


def _match(torch, P, img, N, r, variant, copies):
    f = P.cfog_extract(to_dev(torch, img))
    pts = torch.tensor(np.tile(np.array(PTS, np.int32), (copies, 1)), device="cuda")
    full = lambda v: torch.full((len(pts),), v, dtype=torch.int32, device="cuda")
    res = P.cfog_match_batched(P.job_table([(f, f)]), 1, pts, full(N), full(r), N, r, variant=variant)
    torch.cuda.synchronize()
    return res.cpu().numpy()


@pytest.mark.parametrize("variant", [1, 2, 3, 4])
@pytest.mark.parametrize("N,r", [(48, 20), (33, 9), (64, 5)])
def test_flat_window_reports_the_first_lag(N, r, variant):
    torch, P = cuda_or_skip()
    img = np.full((200, 210), 37.0, np.float32)
    for copies in (1, COPIES):
        res = _match(torch, P, img, N, r, variant, copies)
        assert (res[:, 0] == -r).all() and (res[:, 1] == -r).all()
        assert (res[:, 4].view(np.float32) == 0.0).all()
        assert (res[:, 5] == P._lib.CFOG_CP_EDGE_PEAK).all()


@pytest.mark.parametrize("variant", [1, 2, 3, 4])
@pytest.mark.parametrize("N,r", [(48, 20), (40, 25)])
def test_periodic_window_same_lag_in_every_launch(N, r, variant):
    torch, P = cuda_or_skip()
    cell = np.random.default_rng(9).integers(0, 4096, (4, 4)).astype(np.float32)
    img = np.tile(cell, (50, 53))
    few = _match(torch, P, img, N, r, variant, 1)
    assert (few[:, :2] % 4 == 0).all()
    many = _match(torch, P, img, N, r, variant, COPIES)
    assert np.array_equal(many, np.tile(few, (COPIES, 1)))
