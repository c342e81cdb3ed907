"""The host's search for FFT plans (no GPU): the search that drops beaten codes early
finds the plan of least (cost, code) over all codes, in well under the time of working
every code out."""
import ctypes
import time

import pytest

from tests._hostcc import host_lib

CODE = """
#include "cfog_plan.cuh"
using namespace cfog;
static void row(const MatchPlan &p, int *out) {
    const int v[8] = {p.y.nb, p.x.nb, p.y.P, p.x.P, p.y.A, p.x.A, p.ld, p.G};
    for (int i = 0; i < 8; ++i) out[i] = v[i];
}
extern "C" int searched(int N, int r, int m, const int *l, int *out) {
    MatchPlan p;
    const bool ok = make_plan_host(N, r, m, PlanLimits{l[0], l[1], l[2], l[3]}, &p);
    if (ok) row(p, out);
    return ok;
}
extern "C" int every_code(int N, int r, int m, const int *l, int *out) {
    long long best = -1;
    MatchPlan keep;
    for (int code = 0; code < kPlanCodes; ++code) {
        MatchPlan p;
        const long long c = plan_for_code(N, r, m, code, PlanLimits{l[0], l[1], l[2], l[3]}, &p);
        if (c >= 0 && (best < 0 || c < best)) {
            best = c;
            keep = p;
        }
    }
    if (best >= 0) row(keep, out);
    return best >= 0;
}
extern "C" int all_classes(int search, int nmax, int rmax, const int *l) {
    int n = 0, out[8];
    for (int N = 1; N <= nmax; ++N)
        for (int r = 0; r <= rmax; ++r) n += search ? searched(N, r, 9, l, out) : every_code(N, r, 9, l, out);
    return n;
}
"""
# plane bound, shared memory, accumulator columns per thread, threads: WIDE, PAIR, TRIO
LIMITS = {"wide": (16384, 109 * 1024, 128, 256), "pair": (9216, 109 * 1024, 128, 256),
          "trio": (7680, 71 * 1024, 64, 256)}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_lib(tmp_path_factory.mktemp("plan"), "plan", CODE)


@pytest.mark.parametrize("limits", list(LIMITS))
@pytest.mark.parametrize("m", [1, 9, 36])
def test_same_plan_as_every_code(lib, limits, m):
    l = (ctypes.c_int * 4)(*LIMITS[limits])
    a, b = (ctypes.c_int * 8)(), (ctypes.c_int * 8)()
    for N in list(range(1, 257, 5)) + [64, 96, 128, 256]:
        for r in range(33):
            assert lib.searched(N, r, m, l, a) == lib.every_code(N, r, m, l, b)
            assert list(a) == list(b), (N, r)


def test_search_time(lib):
    l = (ctypes.c_int * 4)(*LIMITS["wide"])

    def best(search):
        ts = []
        for _ in range(5):
            t = time.perf_counter()
            assert lib.all_classes(search, 128, 20, l) == 128 * 21
            ts.append(time.perf_counter() - t)
        return min(ts)

    assert best(1) < 0.6 * best(0)
