"""Rectification over more triangles than 32-bit thread numbers of one warp each
reach (2^27): the last two of 2^27 + 3 hold the output, the others are degenerate."""
import numpy as np
import pytest

import synth
from tests._util import cuda_or_skip, to_dev

pytestmark = pytest.mark.gpu


def test_triangles_behind_2_27():
    torch, P = cuda_or_skip()
    if torch.cuda.mem_get_info()[0] < 24e9:
        pytest.skip("needs 12 GB on the device")
    sen = np.random.default_rng(3).integers(0, 4096, (70, 80)).astype(np.float32)
    cps = np.array([(0, 0), (63, 0), (63, 47), (0, 47)], np.int32)
    res = np.zeros(4, dtype=synth.RESULT_DTYPE)
    r = torch.from_numpy(res.view(np.int32).reshape(-1, 6)).cuda()
    n = 2 ** 27 + 3
    tris = torch.zeros((n, 3), dtype=torch.int32, device="cuda")
    tris[-2:] = torch.tensor([(0, 1, 2), (0, 2, 3)], dtype=torch.int32)
    out = P.cfog_tin_rectify(to_dev(torch, sen), torch.from_numpy(cps).cuda(), r, tris, 48, 64, -1.0)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), sen[:48, :64])   # offsets of zero
    del tris, out
    torch.cuda.empty_cache()
