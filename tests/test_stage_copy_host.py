"""The addresses of the FFT matcher's staging copies (no GPU): every copy of a
raw row starts on a boundary of its own size inside the row, reads wanted
columns only, and the copies together read every wanted column."""
import ctypes

import pytest

from tests._hostcc import host_lib

CODE = """
#include "cfog_plan.cuh"
extern "C" void copy_of(int F, int x, int x0, int x1, int *out) {
    const cfog::StageCopy c = cfog::stage_copy(F, x, x0, x1);
    out[0] = c.col;
    out[1] = c.bytes;
}
extern "C" int raw_len_of(int Px) { return cfog::raw_len(Px); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_lib(tmp_path_factory.mktemp("stage"), "stage", CODE)


@pytest.mark.parametrize("F", [4, 1])
@pytest.mark.parametrize("Px", [2, 24, 50, 96, 128, 256])
def test_copies_are_aligned_and_read_the_wanted_columns(lib, F, Px):
    out = (ctypes.c_int * 2)()
    for x0 in range(4):
        for width in sorted({1, 2, 3, Px // 2, Px - 1, Px} - {0}):
            x1, read = x0 + width, set()
            for x in range(0, lib.raw_len_of(Px), F):
                lib.copy_of(F, x, x0, x1, out)
                col, size = out[0], out[1]
                assert col % F == 0 and 0 <= col < x1
                assert size % 4 == 0 and 0 <= size <= 4 * F
                if size:
                    assert col == x and col + size // 4 <= x1
                    read |= set(range(col, col + size // 4))
            assert set(range(x0, x1)) <= read
