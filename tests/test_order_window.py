"""The windows of columns that a read puts a long row in order by
(order_window.h), run on the host: any 32-bit values whatever leave every mark
inside the window's shared memory and end the loop over the windows, and a
row's distinct columns get their places in column order.  The keys of rows
sorted together sort by row first, whatever a value holds."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_08808_gb300", "csrc")

# k_order_long's steps on one row, by the same functions, every index checked
DRIVER = r"""
#include <vector>
#include "order_window.h"
using namespace dspg;
extern "C" int order_row(const int32_t *v, int64_t len, int64_t ncols, int64_t *place, int *windows) {
    const int32_t W = (int32_t)(ncols < OL_W ? (ncols + OL_STRETCH - 1) / OL_STRETCH * OL_STRETCH : OL_W);
    int32_t mn = INT32_MAX, mx = -1;
    for (int64_t e = 0; e < len; e++)
        if (ow_is_column(v[e], ncols)) {
            mn = v[e] < mn ? v[e] : mn;
            mx = v[e] > mx ? v[e] : mx;
        }
    *windows = 0;
    for (int64_t e = 0; e < len; e++) place[e] = -1;
    if (mn > mx) return 0;
    int64_t before = 0;
    for (int32_t wb = ow_first(mn); wb <= mx; wb += W) {
        if (++*windows > 1 << 12) return 1;  // does not end
        const int32_t nb = ow_stretches(wb, mx, W);
        if (nb < 1 || nb > W / OL_STRETCH) return 2;
        const uint32_t in = (uint32_t)nb * OL_STRETCH;
        std::vector<int> marks(W, 0);
        for (int64_t e = 0; e < len; e++) {
            const uint32_t c = ow_place(v[e], wb);
            if (c < in) {
                if (c >= (uint32_t)W) return 3;
                marks[c] = 1;
            }
        }
        std::vector<int64_t> first(W, 0);
        int64_t n = before;
        for (int32_t c = 0; c < W; c++) {
            first[c] = n;
            n += marks[c];
        }
        for (int64_t e = 0; e < len; e++) {
            const uint32_t c = ow_place(v[e], wb);
            if (c < in) place[e] = first[c];
        }
        before = n;
        if ((int64_t)wb + W > INT32_MAX) return 4;  // the step would overflow
    }
    return 0;
}
extern "C" uint64_t list_key(uint64_t k, int32_t v, int cb) { return ow_list_key(k, v, cb); }
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("order_window")
    src, lib = d / "driver.cpp", d / "driver.so"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fwrapv", "-fPIC", "-shared", "-I", CSRC, "-o", str(lib),
                    str(src)], check=True)
    return ctypes.CDLL(str(lib))


@pytest.fixture(scope="module")
def order_row(driver):
    f = driver.order_row

    def call(v, ncols):
        v = np.ascontiguousarray(v, np.int32)
        place, windows = np.zeros(v.size, np.int64), ctypes.c_int()
        rc = f(v.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(v.size), ctypes.c_int64(ncols),
               place.ctypes.data_as(ctypes.c_void_p), ctypes.byref(windows))
        return rc, place, windows.value

    return call


WIDTHS = [1, 65, 1024, 1025, 20480, (1 << 18) - 1, 1 << 18, (1 << 18) + 1, 600001, (1 << 22) - 1, 1 << 22]
EDGES = [-2**31, -2**31 + 1, -2_000_000_000, -1024, -1, 0, 1, 1023, 1024, (1 << 18) - 1, 1 << 18, (1 << 22) - 1, 1 << 22,
         (1 << 22) + 1023, 2_000_000_000, 2**31 - (1 << 18), 2**31 - 1025, 2**31 - 1024, 2**31 - 2, 2**31 - 1]


@pytest.mark.parametrize("ncols", WIDTHS)
def test_any_values_stay_inside_the_window(order_row, ncols):
    rng = np.random.default_rng(ncols)
    rows = [np.array(p) for p in [[a, b] for a in EDGES for b in EDGES]]
    rows += [np.array(EDGES), np.array(EDGES[::-1]), np.array([-1] * 70), np.zeros(70, np.int64)]
    rows += [rng.integers(-2**31, 2**31, 200) for _ in range(20)]
    rows += [np.concatenate([rng.integers(-2**31, 2**31, 100), rng.integers(0, ncols, 100)]) for _ in range(20)]
    for v in rows:
        rc, _, windows = order_row(v, ncols)
        assert rc == 0, (v, rc)
        assert windows <= -(-ncols // (1 << 18)) + 1


@pytest.mark.parametrize("ncols", WIDTHS)
def test_columns_get_their_places_in_order(order_row, ncols):
    rng = np.random.default_rng(ncols + 1)
    for n in (1, 2, 66, 400):
        v = rng.permutation(np.unique(np.concatenate([[0, ncols - 1], rng.integers(0, ncols, n)])))
        rc, place, _ = order_row(v, ncols)
        assert rc == 0
        assert np.array_equal(place, np.argsort(np.argsort(v)))


@pytest.mark.parametrize("cb", [1, 23, 31])
def test_keys_sort_by_row_first(driver, cb):
    f = driver.list_key
    f.restype = ctypes.c_uint64
    for k in (0, 1, 5, (1 << 16) - 1):
        for v in EDGES + [(1 << cb) - 1, 1 << (cb - 1)]:
            key = f(ctypes.c_uint64(k), ctypes.c_int32(v), cb)
            assert key >> cb == k
            if 0 <= v < 1 << cb:
                assert key & ((1 << cb) - 1) == v
