"""Index arithmetic of the sort's and the push's passes over a share of a species
(csrc/span.cuh), on the host: at the top of the accepted range (2^31 - 1 particles) the
last rounds of a loop step past the end, and no position they form may pass for a
particle's.  The signed form `p = base + step; p < end` does not hold there."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1308_5892_gb300", "csrc")

SOURCE = """
#include "span.cuh"
using namespace pic;
extern "C" int rows(int n) { return slot_rows(n); }
// positions outside [first, end) that the rounds of `step` elements over the share's last part form;
// *seen: visited positions less those there are
extern "C" long long walk(int first, int end, unsigned step, long long *seen) {
    long long bad = 0;
    const unsigned count = (unsigned)(end - first), last = count < 3 * step ? 0u : (count - 2 * step) / step * step;
    *seen = (long long)last - count;
    for (Slot base = slot_at((Slot)first, last); slot_before(base, end); base = slot_at(base, step))
        for (unsigned o = 0; o < step; ++o) {
            const Slot p = slot_at(base, o);
            if (!slot_before(p, end)) continue;
            ++*seen;
            if ((long long)p < first || (long long)p >= end) ++bad;
        }
    return bad;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("span")
    (d / "span.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "span.so"), str(d / "span.cpp")], check=True)
    L = ctypes.CDLL(str(d / "span.so"))
    L.walk.restype = ctypes.c_longlong
    L.walk.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_uint, ctypes.POINTER(ctypes.c_longlong)]
    return L


TOP = 2 ** 31 - 1


@pytest.mark.parametrize("first,end", [(0, 1), (7, 8199), (0, 8193), (0, TOP), (0, TOP - 8191), (TOP - 5, TOP),
                                       (TOP - 100000, TOP), (1, TOP - 1)])
@pytest.mark.parametrize("step", [32, 1024, 4096, 8192])   # rows and items of the push, rounds of the sort
def test_rounds_past_the_end_form_no_position(lib, first, end, step):
    over = ctypes.c_longlong()
    assert lib.walk(first, end, step, ctypes.byref(over)) == 0
    assert over.value == 0   # and every element is visited once


def test_rows_at_the_ends_of_the_range(lib):
    assert [lib.rows(n) for n in (0, 1, 32, 33, TOP - 31, TOP)] == [0, 1, 1, 2, 2 ** 26 - 1, 2 ** 26]


def test_no_rows_for_offsets_out_of_order(lib):
    assert [lib.rows(n) for n in (-1, -31, -32, -TOP)] == [0, 0, 0, 0]
