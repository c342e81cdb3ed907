"""Plans of the 16384-element planes by radius (no GPU).  From radius 26 on a plane that
leaves an SM one CTA costs a twelfth more than its arithmetic, so no plan costs more
than that above the class's least; below, it costs double."""
import ctypes

import pytest

from tests._hostcc import host_lib

CODE = """
#include "cfog_plan.cuh"
using namespace cfog;
// cost of the plan at a limit of shared memory, without the charge, and its shared memory
extern "C" long long cost_of_plan(int N, int r, int m, int smem_cap, int *smem) {
    MatchPlan p;
    if (!make_plan_host(N, r, m, PlanLimits{16384, smem_cap, 128, 256}, &p)) return -1;
    *smem = plan_smem_bytes(p, N, r, 256, p.G);
    return (long long)p.y.P * p.x.P * (fft_len_cost(p.y.A, p.y.B) + fft_len_cost(p.x.A, p.x.B)) *
           (p.y.nb * p.x.nb * m + 1);
}
"""
CAP, ANY = 109 * 1024, 1 << 30


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib = host_lib(tmp_path_factory.mktemp("radius"), "radius", CODE)
    lib.cost_of_plan.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("m", [9, 36])
@pytest.mark.parametrize("r", range(33))
def test_charge_by_radius(lib, r, m):
    smem = ctypes.c_int()
    for N in range(1, 257):
        least = lib.cost_of_plan(N, r, m, ANY, ctypes.byref(smem))
        cost = lib.cost_of_plan(N, r, m, CAP, ctypes.byref(smem))
        assert least <= cost <= (least + least // 12 if r >= 26 else 2 * least), N
