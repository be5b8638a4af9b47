"""Which host arrays a batch is read from, and rows written to, in place
(host_view.h), on the host: only those that lie in page-locked memory from
their first byte to their last, and aligned to their values."""

import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_08808_gb300", "csrc")

# page-locked ranges [lo, hi) at a device address each
DRIVER = r"""
#include <cstdint>
#include "host_view.h"
struct Range { uintptr_t lo, hi, dev; };
extern "C" uintptr_t view_of(const Range *r, int n, uintptr_t p, int64_t count, size_t size) {
    auto view = [&](void *q) -> void * {
        for (int k = 0; k < n; k++)
            if ((uintptr_t)q >= r[k].lo && (uintptr_t)q < r[k].hi) return (void *)(r[k].dev + ((uintptr_t)q - r[k].lo));
        return nullptr;
    };
    return (uintptr_t)dspg::array_view(view, (void *)p, count, size);
}
"""


@pytest.fixture(scope="module")
def view_of(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_view")
    src, lib = d / "driver.cpp", d / "driver.so"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fPIC", "-shared", "-I", CSRC, "-o", str(lib), str(src)],
                   check=True)
    f = ctypes.CDLL(str(lib)).view_of
    f.restype = ctypes.c_size_t

    def call(ranges, p, count, size=1):
        flat = (ctypes.c_size_t * (3 * len(ranges)))(*[x for r in ranges for x in r])
        return f(flat, len(ranges), ctypes.c_size_t(p), ctypes.c_int64(count), ctypes.c_size_t(size))

    return call


@pytest.mark.parametrize("dev", [0x1000, 0x900000])
@pytest.mark.parametrize("p, nbytes, inside", [
    (0x1000, 0x1000, True), (0x1000, 1, True), (0x1fff, 1, True), (0x1ffc, 4, True), (0x1800, 0x800, True),
    (0x1000, 0x1001, False), (0x1ffc, 5, False), (0x1fff, 2, False), (0xfff, 2, False), (0x2000, 1, False),
    (0xfff, 0x1002, False), (0x1800, 0x100000, False),
])
def test_an_array_is_used_in_place_only_when_all_of_it_is_page_locked(view_of, dev, p, nbytes, inside):
    assert view_of([(0x1000, 0x2000, dev)], p, nbytes) == (dev + p - 0x1000 if inside else 0)


def test_two_ranges_count_as_one_only_where_the_gpu_sees_them_side_by_side(view_of):
    for dev2, want in ((0x6000, 0x5800), (0x9000, 0)):
        assert view_of([(0x1000, 0x2000, 0x5000), (0x2000, 0x3000, dev2)], 0x1800, 0x1000) == want


def test_only_aligned_arrays_of_a_size_that_can_be(view_of):
    r = [(0x1000, 0x9000, 0x5000)]
    assert view_of(r, 0x1000, 0x1000, 8) == 0x5000 and view_of(r, 0x1008, 0xfff, 8) == 0x5008
    for p, count, size in ((0x1004, 16, 8), (0x1002, 16, 4), (0x1001, 1, 4), (0x1008, 0x1000, 8), (0x1000, -1, 4),
                           (0x1000, (1 << 61) + 1, 8), (0x1000, 2**63 - 1, 4), (0, 4, 4)):
        assert view_of(r, p, count, size) == 0, (p, count, size)
    assert view_of(r, 0x1000, 0, 8) == 0x5000  # nothing is accessed
