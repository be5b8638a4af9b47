// order_window.h -- the columns that a read puts a row in order by, window
// after window (k_order_long).  Plain arithmetic, so that a host program can
// run it on any 32-bit values.
//
// A read of C may meet a row whose columns are still being written (an
// asynchronous batch has moved it to memory that holds anything).  So the
// row's first and last column are taken over real columns only, the windows
// lie between those two, and whatever the other values are, they fall outside.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DSPG_HD __host__ __device__ __forceinline__
#else
#define DSPG_HD inline
#endif

namespace dspg {

constexpr int OL_W = 1 << 18;       // columns of a window
constexpr int OL_STRETCH = 1024;    // columns of a stretch, whose marks are counted together

// Whether v is a column of a C of ncols columns (at most 2^31 - 1 of them).
DSPG_HD bool ow_is_column(int32_t v, int64_t ncols) { return (uint32_t)v < (uint32_t)ncols; }

// Where the first window starts, mn being the row's first column (not negative).
DSPG_HD int32_t ow_first(int32_t mn) { return mn & ~(OL_STRETCH - 1); }

// Stretches of the window of W columns (whole stretches) at wb, mx >= wb being the row's last column.
DSPG_HD int32_t ow_stretches(int32_t wb, int32_t mx, int32_t W) {
    const int32_t to_end = ((mx - wb) >> 10) + 1, most = W >> 10;
    return to_end < most ? to_end : most;
}

// The place of v in the window of nb stretches at wb; in it when below nb * OL_STRETCH.
DSPG_HD uint32_t ow_place(int32_t v, int32_t wb) { return (uint32_t)v - (uint32_t)wb; }

// Whether a row of len entries whose columns span that many windows is put in
// order by a sorting network over its entries instead: up to 256 entries a
// window, and at most OL_NET.  Each side of the line as measured, 20,000 rows
// into device memory, us (network / windows, whose cost is nearly that of
// going over them):
//    2 windows:  400 entries  490 / 583,   768 entries  923 / 722
//    4 windows: 1024 entries  950 / 1244, 1536 entries 1973 / 1443
//    8 windows: 2048 entries 2047 / 2710, 3000 entries 4358 / 3208
//   16 windows: 2048 entries 2043 / 4442, 4000 entries 4619 / 6408
constexpr int OL_NET = 4096;
DSPG_HD bool ow_by_network(int64_t len, int windows) {
    return windows > 1 && len <= OL_NET && len <= (int64_t)windows << 8;
}

// The key that sorts value v of the k-th listed row: by row first, whatever v
// holds, so that a row that is being written displaces no entry of another.
DSPG_HD uint64_t ow_list_key(uint64_t k, int32_t v, int cb) {
    return k << cb | ((uint32_t)v & (((uint64_t)1 << cb) - 1));
}

static_assert(OL_STRETCH == 1 << 10 && OL_W % OL_STRETCH == 0, "windows of whole stretches");

}  // namespace dspg
