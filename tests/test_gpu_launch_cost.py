"""Host time of a launch: the plans of a launch's bounds are searched once, for either
CTA size, and a change of the tuned plans does not repeat the search."""
import time

import pytest

import synth
from tests._util import cuda_or_skip, to_dev

pytestmark = pytest.mark.gpu


def test_plans_are_searched_once_per_bounds():
    torch, P = cuda_or_skip()
    L = P._lib
    im = synth.batched_pair(3, size=300)
    f = P.cfog_extract(to_dev(torch, im.A)), P.cfog_extract(to_dev(torch, im.B))
    jobs = P.job_table([f])
    many = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    cps = torch.full((many, 2), 150, dtype=torch.int32, device="cuda")
    tm = torch.full((many,), 16, dtype=torch.int32, device="cuda")
    rd = torch.full((many,), 4, dtype=torch.int32, device="cuda")
    out, ws = torch.empty((many, 6), dtype=torch.int32, device="cuda"), P.match_workspace(many)

    def call(n, bounds):
        torch.cuda.synchronize()
        t = time.perf_counter()
        P.cfog_match_batched(jobs, 1, cps[:n], tm[:n], rd[:n], *bounds, variant=1, out=out[:n], workspace=ws)
        return time.perf_counter() - t

    for n in (many, 8):
        call(n, (40, 8))                       # both kernels loaded
    ratios = []
    for side in (251, 253, 255):
        bounds = (side, 22)
        first = call(many, bounds)             # searches the classes
        few = call(8, bounds)                  # 512-thread CTAs: the same search
        L.check(L.lib().cfog_match_set_plan(1, 9, 20, 5, -1), "cfog_match_set_plan")
        again = call(many, bounds)             # tuned plans changed
        ratios.append(max(few, again) / first)
    assert sorted(ratios)[1] < 0.5, ratios
