// layout.cu -- building slack-CSRs from row-wise sources and reading them back.
//
// These kernels move whole rows between a CSR-like source (row start + row
// length) and a destination layout, one warp per row, and sort read rows by
// column; they carry no semiring arithmetic.
#include <algorithm>

#include "internal.h"
#include "order_window.h"

namespace dspg {

static unsigned blocks_for(int64_t n, int nt, int64_t cap = 1 << 20) {
    int64_t g = (n + nt - 1) / nt;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (unsigned)g;
}

__global__ void k_iota(int32_t *a, int64_t n) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        a[x] = (int32_t)x;
}
// First and last steps of a batch.  The host keeps the batch pointers and
// receives the control block in pinned, mapped memory; these two small
// kernels move them (the pointers read uncached, as the host rewrites them
// between batches), which costs less on the stream than a memset and two
// copy-engine transfers.
static_assert(sizeof(Ctl) % sizeof(unsigned long long) == 0, "control block in 8-byte words");
constexpr int CTL_WORDS = (int)(sizeof(Ctl) / sizeof(unsigned long long));
constexpr int ARG_WORDS = (int)(3 * sizeof(InArgs) / sizeof(unsigned long long));

__global__ void k_begin_batch(const InArgs *host_args, InArgs *dev_args, Ctl *ctl) {
    pdl_begin();
    unsigned long long *c = (unsigned long long *)ctl;
    for (int k = threadIdx.x; k < CTL_WORDS; k += blockDim.x) c[k] = 0ull;
    if (threadIdx.x < ARG_WORDS)
        ((unsigned long long *)dev_args)[threadIdx.x] = __ldcv((const unsigned long long *)host_args + threadIdx.x);
}

__global__ void k_end_batch(const Ctl *ctl, Ctl *host_ctl) {
    pdl_begin();
    const unsigned long long *c = (const unsigned long long *)ctl;
    for (int k = threadIdx.x; k < CTL_WORDS; k += blockDim.x) ((unsigned long long *)host_ctl)[k] = c[k];
    __threadfence_system();
}

void begin_batch(const InArgs *host_args, InArgs *dev_args, Ctl *ctl, cudaStream_t s) {
    launch_k(k_begin_batch, 1, 128, 0, s, host_args, dev_args, ctl);
}

void end_batch(const Ctl *ctl, Ctl *host_ctl, cudaStream_t s) { launch_k(k_end_batch, 1, 128, 0, s, ctl, host_ctl); }

void fill_iota(int32_t *a, int64_t n, cudaStream_t s) {
    if (n > 0) launch_k(k_iota, blocks_for(n, 256, 8192), 256, 0, s, a, n);
}

__global__ void k_caps(const int32_t *len, int32_t *cap, int64_t n, int smin, int sdiv) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        cap[x] = slack_cap(len[x], smin, sdiv);
}
void caps_from_lens(const int32_t *len, int32_t *cap, int64_t n, int smin, int sdiv, cudaStream_t s) {
    if (n > 0) launch_k(k_caps, blocks_for(n, 256, 8192), 256, 0, s, len, cap, n, smin, sdiv);
}

__global__ void k_lens_rowptr(const int64_t *rowptr, int32_t *len, int64_t n) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        len[x] = (int32_t)(rowptr[x + 1] - rowptr[x]);
}
void lens_from_rowptr(const int64_t *rowptr, int32_t *len, int64_t n, cudaStream_t s) {
    if (n > 0) launch_k(k_lens_rowptr, blocks_for(n, 256, 8192), 256, 0, s, rowptr, len, n);
}

__global__ void k_lens_of_rows(const int32_t *rows, int64_t n, const int32_t *len, int32_t *out) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        out[x] = len[rows[x]];
}
void lens_of_rows(const int32_t *rows, int64_t n, const int32_t *len, int32_t *out, cudaStream_t s) {
    if (n > 0) launch_k(k_lens_of_rows, blocks_for(n, 256, 8192), 256, 0, s, rows, n, len, out);
}

// R in row order from its collection: each chunk of 8192 rows wrote its
// (ascending) rows at chunk[2c] in R, chunk[2c+1] of them, so laying the
// chunks end to end in chunk order sorts R.  k_chunk_counts lists the
// counts for a scan, k_chunk_copy moves each chunk (a block per chunk).
__global__ void k_chunk_counts(const long long *chunk, int64_t nch, int64_t *cnt) {
    pdl_begin();
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nch; c += (int64_t)gridDim.x * blockDim.x)
        cnt[c] = chunk[2 * c + 1];
}

__global__ void k_chunk_copy(const int32_t *R, const long long *chunk, int64_t nch, const int64_t *ex, int64_t n,
                             int32_t *out) {
    pdl_begin();
    for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
        const long long b = chunk[2 * c], k = chunk[2 * c + 1];
        const int64_t o = ex[c];
        if (k <= 0 || b < 0 || b + k > n || o + k > n) continue;  // not one collection: the caller checks ex[nch]
        for (long long t = threadIdx.x; t < k; t += blockDim.x) out[o + t] = R[b + t];
    }
}

void rows_in_order(const int32_t *R, const long long *chunk, int64_t nch, int64_t n, int64_t *cnt, int64_t *ex,
                   int64_t *tmp, int32_t *out, cudaStream_t s) {
    if (nch <= 0) return;
    launch_k(k_chunk_counts, blocks_for(nch, 256, 1024), 256, 0, s, chunk, nch, cnt);
    scan_i64(cnt, ex, nch, tmp, s);
    launch_k(k_chunk_copy, (unsigned)std::min<int64_t>(nch, 8192), 256, 0, s, R, chunk, nch, ex, n, out);
}

// R in row order and its row pointers for a read, in two launches while
// the chunk table is small enough for one block to scan (READ_NCH_MAX
// chunks): every block scans the chunk counts itself, so no scan launches
// come between.  k_read_order lays each chunk's rows at the scan of the
// counts, looks up their lengths in C and sums them per chunk;
// k_read_rowptr scans the sums and each chunk's lengths into the rows' first
// entries.  Both also write the caller's page-locked arrays when given
// (h_rows, h_rp: device addresses), and both leave everything untouched when
// the counts do not add up to n (R was not collected in one pass; the caller
// sees *r_total != n).
constexpr int RD_NT = 1024;
constexpr int RD_IPT = 2;

int64_t read_nch_max() { return (int64_t)RD_NT * RD_IPT; }

// Exclusive scan of the m <= RD_NT * RD_IPT values load(0..m) into s_ex;
// returns their total.  Every thread of the block calls it.
template <class F>
__device__ __forceinline__ int64_t rd_scan_table(F load, int m, int64_t *s_ex, int64_t *s_w) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int64_t v[RD_IPT];
    int64_t sum = 0;
#pragma unroll
    for (int j = 0; j < RD_IPT; j++) {
        const int c = tid * RD_IPT + j;
        v[j] = c < m ? load(c) : 0;
        sum += v[j];
    }
    const int64_t incl = warp_incl_scan<int64_t>(sum);
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int64_t t = s_w[lane];
        const int64_t ti = warp_incl_scan<int64_t>(t);
        s_w[lane] = ti - t;
        if (lane == 31) s_w[32] = ti;
    }
    __syncthreads();
    int64_t e = s_w[w] + incl - sum;
#pragma unroll
    for (int j = 0; j < RD_IPT; j++) {
        const int c = tid * RD_IPT + j;
        if (c < m) s_ex[c] = e;
        e += v[j];
    }
    const int64_t total = s_w[32];
    __syncthreads();
    return total;
}

// Exclusive scan of one value per thread; *total gets the block's sum.
__device__ __forceinline__ int64_t rd_block_scan(int64_t v, int64_t *s_w, int64_t *total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t incl = warp_incl_scan<int64_t>(v);
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int64_t t = s_w[lane];
        const int64_t ti = warp_incl_scan<int64_t>(t);
        s_w[lane] = ti - t;
        if (lane == 31) s_w[32] = ti;
    }
    __syncthreads();
    const int64_t r = s_w[w] + incl - v;
    *total = s_w[32];
    __syncthreads();
    return r;
}

// chunk c of R holds k = chunk[2c+1] rows at chunk[2c]; they go to o = ex[c]
__device__ __forceinline__ bool rd_chunk_ok(long long b, long long k, int64_t o, int64_t n) {
    return k > 0 && b >= 0 && b + k <= n && o + k <= n;
}

__global__ void __launch_bounds__(RD_NT)
k_read_order(const int32_t *R, const long long *chunk, int nch, int64_t n_arg, const long long *n_dev, int64_t rows_cap,
             const unsigned *status, const int32_t *len, int32_t *out, int32_t *lens, int64_t *S, int64_t *r_total,
             int32_t *h_rows, ReadOut *res) {
    pdl_begin();
    __shared__ int64_t s_ex[RD_NT * RD_IPT];
    __shared__ int64_t s_w[33];
    const int64_t n = n_dev ? (int64_t)*n_dev : n_arg;
    // enqueued behind an apply (n on the device): nothing is read after a
    // failed batch or when R would not fit the buffers sized for it
    const bool skip = (status && *status) || n < 0 || n > rows_cap;
    const int64_t tot = rd_scan_table([&](int c) { return (int64_t)chunk[2 * c + 1]; }, nch, s_ex, s_w);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *r_total = skip ? -1 : tot;
        if (res) {
            ReadOut z{};
            z.nr = n;
            *res = z;
        }
    }
    if (skip || tot != n) return;
    for (int c = blockIdx.x; c < nch; c += gridDim.x) {
        const long long b = chunk[2 * c], k = chunk[2 * c + 1];
        const int64_t o = s_ex[c];
        int64_t sum = 0;
        if (rd_chunk_ok(b, k, o, n))
            for (long long t = threadIdx.x; t < k; t += RD_NT) {
                const int32_t r = R[b + t];
                out[o + t] = r;
                if (h_rows) h_rows[o + t] = r;
                const int32_t L = len[r];
                lens[o + t] = L;
                sum += L;
            }
        sum = warp_sum<int64_t>(sum);
        if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = sum;
        __syncthreads();
        if (threadIdx.x < 32) {
            int64_t t = s_w[threadIdx.x];
            t = warp_sum<int64_t>(t);
            if (threadIdx.x == 0) S[c] = t;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(RD_NT)
k_read_rowptr(const long long *chunk, int nch, int64_t n_arg, const long long *n_dev, const int32_t *lens,
              const int64_t *S, const int64_t *r_total, int64_t *rp, int64_t *h_rp) {
    pdl_begin();
    __shared__ int64_t s_ex[RD_NT * RD_IPT];
    __shared__ int64_t s_base[RD_NT * RD_IPT];
    __shared__ int64_t s_w[33];
    const int64_t n = n_dev ? (int64_t)*n_dev : n_arg;
    if (*r_total != n) return;
    rd_scan_table([&](int c) { return (int64_t)chunk[2 * c + 1]; }, nch, s_ex, s_w);
    const int64_t nnz = rd_scan_table([&](int c) { return S[c]; }, nch, s_base, s_w);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        rp[n] = nnz;
        if (h_rp) h_rp[n] = nnz;
    }
    for (int c = blockIdx.x; c < nch; c += gridDim.x) {
        const long long b = chunk[2 * c], k = chunk[2 * c + 1];
        const int64_t o = s_ex[c];
        if (!rd_chunk_ok(b, k, o, n)) continue;  // the same for the whole block
        int64_t carry = s_base[c];
        for (long long t0 = 0; t0 < k; t0 += RD_NT) {
            const long long t = t0 + threadIdx.x;
            const int64_t L = t < k ? lens[o + t] : 0;
            int64_t round = 0;
            const int64_t e = rd_block_scan(L, s_w, &round);
            if (t < k) {
                rp[o + t] = carry + e;
                if (h_rp) h_rp[o + t] = carry + e;
            }
            carry += round;
        }
    }
}

// The same for at most RS_MAX rows, in one launch of one block: a thread
// takes four consecutive places of R, finds their chunk by a search of the
// scanned counts in shared memory, and the four loads of each step are in
// flight together.  Two launches of many blocks take 9 us on a few thousand
// rows, most of it their own latency; this one 6.
constexpr int64_t RS_MAX = 4 * RD_NT;

__global__ void __launch_bounds__(RD_NT)
k_read_small(const int32_t *R, const long long *chunk, int nch, int64_t n_arg, const long long *n_dev, int64_t rows_cap,
             const unsigned *status, const int32_t *len, int32_t *out, int64_t *r_total, int64_t *rp, int32_t *h_rows,
             int64_t *h_rp, ReadOut *res) {
    pdl_begin();
    __shared__ int64_t s_ex[RD_NT * RD_IPT], s_b[RD_NT * RD_IPT];
    __shared__ int64_t s_w[33];
    const int tid = threadIdx.x;
    const int64_t n = n_dev ? (int64_t)*n_dev : n_arg;
    const bool skip = (status && *status) || n < 0 || n > rows_cap || n > RS_MAX;
    for (int c = tid; c < nch; c += RD_NT) s_b[c] = chunk[2 * c];
    const int64_t tot = rd_scan_table([&](int c) { return (int64_t)chunk[2 * c + 1]; }, nch, s_ex, s_w);
    if (tid == 0) {
        *r_total = skip ? -1 : tot;
        if (res) {
            ReadOut z{};
            z.nr = n;
            *res = z;
        }
    }
    if (skip || tot != n) return;
    int32_t r[4];
    int64_t L[4], sum = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int64_t t = (int64_t)tid * 4 + j;
        r[j] = 0;
        if (t < n) {
            const int c = (int)upper_bound_dev<int64_t>(s_ex, 0, nch, t) - 1;  // the last chunk that starts at or before t
            const int64_t b = s_b[c] + t - s_ex[c];
            r[j] = R[b >= 0 && b < n ? b : 0];
        }
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int64_t t = (int64_t)tid * 4 + j;
        L[j] = t < n ? len[r[j]] : 0;
        sum += L[j];
        if (t < n) {
            out[t] = r[j];
            if (h_rows) h_rows[t] = r[j];
        }
    }
    int64_t nnz = 0;
    int64_t e = rd_block_scan(sum, s_w, &nnz);
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int64_t t = (int64_t)tid * 4 + j;
        if (t < n) {
            rp[t] = e;
            if (h_rp) h_rp[t] = e;
        }
        e += L[j];
    }
    if (tid == 0) {
        rp[n] = nnz;
        if (h_rp) h_rp[n] = nnz;
    }
}

void read_order_rowptr(const int32_t *R, const long long *chunk, int64_t nch, int64_t n, const long long *n_dev,
                       int64_t rows_cap, const unsigned *status, const int32_t *len, int32_t *out, int32_t *lens,
                       int64_t *S, int64_t *r_total, int64_t *rp, int32_t *h_rows, int64_t *h_rp, ReadOut *res,
                       cudaStream_t s, int num_sms) {
    if (n <= RS_MAX) {
        launch_k(k_read_small, 1, RD_NT, 0, s, R, chunk, (int)nch, n, n_dev, rows_cap, status, len, out, r_total, rp,
                 h_rows, h_rp, res);
        return;
    }
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nch, (int64_t)num_sms * 2));
    launch_k(k_read_order, g, RD_NT, 0, s, R, chunk, (int)nch, n, n_dev, rows_cap, status, len, out, lens, S, r_total,
             h_rows, res);
    launch_k(k_read_rowptr, g, RD_NT, 0, s, chunk, (int)nch, n, n_dev, (const int32_t *)lens, (const int64_t *)S,
             (const int64_t *)r_total, rp, h_rp);
}

template <typename T>
__global__ void k_copy_rows(const int32_t *rows, int64_t n, const int64_t *src_off, const int32_t *len,
                            const int32_t *src_col, const T *src_val, const int64_t *dst_off, int32_t *dst_col,
                            T *dst_val) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < n; x += nwarps) {
        const int64_t r = rows ? rows[x] : x;
        const int64_t so = src_off[r], d = dst_off[r];
        const int L = len[r];
        for (int e = lane; e < L; e += 32) {
            dst_col[d + e] = src_col[so + e];
            if (dst_val) dst_val[d + e] = src_val[so + e];
        }
    }
}

void copy_rows(const int32_t *rows, int64_t n, const int64_t *src_off, const int32_t *len, const int32_t *src_col,
               const void *src_val, const int64_t *dst_off, int32_t *dst_col, void *dst_val, int vsize,
               cudaStream_t s, int num_sms) {
    if (n <= 0) return;
    unsigned g = blocks_for(n * 32, 256, (int64_t)num_sms * 16);
    if (vsize == 8)
        launch_k(k_copy_rows<double>, g, 256, 0, s, rows, n, src_off, len, src_col, (const double *)src_val, dst_off,
                                              dst_col, (double *)dst_val);
    else
        launch_k(k_copy_rows<int32_t>, g, 256, 0, s, rows, n, src_off, len, src_col, (const int32_t *)src_val, dst_off,
                                               dst_col, (int32_t *)dst_val);
}

__global__ void k_gather_cols(int64_t n, MatView M, const int64_t *out_rowptr, int32_t *out_col) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += nwarps) {
        const int64_t so = M.off[r], d = out_rowptr[r];
        const int L = M.len[r];
        for (int e = lane; e < L; e += 32) out_col[d + e] = M.col[so + e];
    }
}

void gather_cols_out(int64_t n, const MatView &M, const int64_t *out_rowptr, int32_t *out_col, cudaStream_t s,
                     int num_sms) {
    if (n <= 0) return;
    launch_k(k_gather_cols, blocks_for(n * 32, 256, (int64_t)num_sms * 16), 256, 0, s, n, M, out_rowptr, out_col);
}

// ------------------------------------------------- rows out, in column order

// C's rows are stored in any column order (the hash bins write long rows in
// table order); every read returns canonical rows.  Two launches take the
// rows straight from the arena to their places in the result, which is
// device memory or, through the C2C link, the caller's page-locked arrays:
// k_read_short the rows of up to SORT_SHORT entries, which it also counts
// and lists the longer ones of, and k_order_long (or k_sort_long where C is
// very wide) those.
constexpr int SORT_SHORT = 64;     // rows up to this length: a warp each
constexpr int SORT_MAX = 16384;    // very wide C: longer rows are listed and sorted together (sort_listed_rows)
constexpr int RS_NT = 256;         // threads of a k_read_short block
constexpr int RS_ROWS = 32;        // rows of its tile
constexpr int RS_PW = RS_ROWS / (RS_NT / 32);  // rows of a warp

// A read may run while an asynchronous batch rewrites other rows of C, and a
// read of all of C then meets rows that change under it, or that have been
// moved to a place whose entries are not written yet: their entries come out
// undefined, but every access stays inside the arena, the row's stretch of
// the result, whose lengths (rp) were taken before, and the windows of
// columns in shared memory (order_window.h).
__device__ __forceinline__ int64_t row_start(const MatView &M, int64_t r, int64_t len) {
    const int64_t so = M.off[r], most = M.arena_cap - len;
    return so <= most ? so : (most > 0 ? most : 0);
}

// A tile of RS_ROWS consecutive rows per block and round: each warp loads
// its four rows together, ranks the columns of those out of order by
// shuffles, and puts the entries at their places in shared memory; the
// block then stores the tile's stretch of the result, whole 128-byte lines
// at a time.  What bounds it is the far side of the stores: into host
// memory rows stored one by one (each starting and ending inside a line)
// reached 144 GB/s on the rows of a 10^4-update stencil batch (17.5 MB: 122
// us) against the link's 190; now 95 us.  Into device memory it is one pass
// instead of a gather and an in-place sort (the 51.7 million entries of the
// 128^3 stencil's square: 0.39 instead of 1.41 ms).  A tile with a longer row
// stores its short rows directly.  Nothing is written when R is not the
// ordered list of its collection (r_total != n) or the entries do not fit
// nnz_cap; the flags say which.
template <typename T>
__global__ void __launch_bounds__(RS_NT)
k_read_short(const int32_t *rows, int64_t n_arg, const long long *n_dev, MatView M, const int64_t *rp,
             const int64_t *r_total, int64_t nnz_cap, int32_t *out_col, T *out_val, int64_t *long_list, ReadOut *res,
             ReadOut *host_res) {
    pdl_begin();
    __shared__ T s_val[RS_ROWS * SORT_SHORT];
    __shared__ int32_t s_col[RS_ROWS * SORT_SHORT];
    const int64_t n = n_dev ? (int64_t)*n_dev : n_arg;
    // rp[n] exists only when R was placed (r_total == n)
    const bool unordered = r_total && *r_total != n;
    const int64_t nnz = unordered ? 0 : rp[n];
    const unsigned bad = (unordered ? READ_UNORDERED : 0u) | (nnz > nnz_cap ? READ_TOO_SMALL : 0u);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        res->nnz = nnz;
        if (bad) atomicOr(&res->flags, bad);
        if (host_res) {  // all that the host needs, but for a very wide C's longest rows
            ReadOut z{};
            z.nnz = nnz;
            z.flags = bad;
            z.nr = n;
            *host_res = z;
        }
    }
    if (bad) return;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const T *mv = (const T *)M.val;
    for (int64_t x0 = (int64_t)blockIdx.x * RS_ROWS; x0 < n; x0 += (int64_t)gridDim.x * RS_ROWS) {
        const int64_t x1 = x0 + RS_ROWS < n ? x0 + RS_ROWS : n;
        const int64_t base = rp[x0], end = rp[x1];
        // lanes 0..RS_PW - 1 hold the warp's rows
        int64_t h_so = 0, h_d = 0;
        int64_t h_len = 0;
        const int64_t hx = x0 + w * RS_PW + lane;
        if (lane < RS_PW && hx < x1) {
            h_d = rp[hx];
            h_len = rp[hx + 1] - h_d;
            h_so = row_start(M, rows ? (int64_t)rows[hx] : hx, h_len);
        }
        const bool lng = h_len > SORT_SHORT;
        const unsigned lm = __ballot_sync(0xffffffffu, lng);
        if (lm) {  // the long rows of this warp: one atomic
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&res->n_long, (unsigned)__popc(lm));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (lng) long_list[at + __popc(lm & lanemask_lt())] = hx;
        }
        const bool staged = !__syncthreads_or(lng);  // then the tile has at most RS_ROWS * SORT_SHORT entries
        const int len_l = lng ? 0 : (int)h_len;
        int len[RS_PW];
        int32_t k0[RS_PW], k1[RS_PW];
        T v0[RS_PW], v1[RS_PW];
#pragma unroll
        for (int j = 0; j < RS_PW; j++) {  // every load of the warp's rows before any use
            const int L = __shfl_sync(0xffffffffu, len_l, j);
            const int64_t so = __shfl_sync(0xffffffffu, h_so, j);
            len[j] = L;
            k0[j] = lane < L ? M.col[so + lane] : INT32_MAX;
            k1[j] = lane + 32 < L ? M.col[so + lane + 32] : INT32_MAX;
            v0[j] = out_val && lane < L ? mv[so + lane] : T(0);
            v1[j] = out_val && lane + 32 < L ? mv[so + lane + 32] : T(0);
        }
#pragma unroll
        for (int j = 0; j < RS_PW; j++) {
            const int L = len[j];
            const int64_t d = __shfl_sync(0xffffffffu, h_d, j);
            // entry e + 1 after entry e: the next lane's, across the halves at lane 31
            const int32_t up0 = __shfl_down_sync(0xffffffffu, k0[j], 1);
            const int32_t lo1 = __shfl_sync(0xffffffffu, k1[j], 0);
            const int32_t up1 = __shfl_down_sync(0xffffffffu, k1[j], 1);
            const int32_t n0 = lane == 31 ? lo1 : up0;
            const bool out_of_order = (lane + 1 < L && k0[j] > n0) || (lane + 33 < L && k1[j] > up1);
            int r0 = lane, r1 = lane + 32;
            if (__any_sync(0xffffffffu, out_of_order)) {  // rank among the row's (distinct) columns
                r0 = 0;
                r1 = 0;
                for (int q = 0; q < 32; q++) {
                    const int32_t a = __shfl_sync(0xffffffffu, k0[j], q), b = __shfl_sync(0xffffffffu, k1[j], q);
                    r0 += (a < k0[j]) + (b < k0[j]);
                    r1 += (a < k1[j]) + (b < k1[j]);
                }
            }
            if (staged) {
                const int o = (int)(d - base);
                if (lane < L) {
                    s_col[o + r0] = k0[j];
                    s_val[o + r0] = v0[j];
                }
                if (lane + 32 < L) {
                    s_col[o + r1] = k1[j];
                    s_val[o + r1] = v1[j];
                }
            } else {
                if (lane < L) {
                    out_col[d + r0] = k0[j];
                    if (out_val) out_val[d + r0] = v0[j];
                }
                if (lane + 32 < L) {
                    out_col[d + r1] = k1[j];
                    if (out_val) out_val[d + r1] = v1[j];
                }
            }
        }
        if (staged) {
            __syncthreads();
            // from the 32-entry boundary at or below base, so that a warp's stores fill lines
            const int cnt = (int)(end - base);
            for (int i = tid - (int)(base & 31); i < cnt; i += RS_NT)
                if (i >= 0) {
                    out_col[base + i] = s_col[i];
                    if (out_val) out_val[base + i] = s_val[i];
                }
        }
        __syncthreads();
    }
}

// Bitonic sort by column of the N (a power of two) keys in sk, with their
// values in sv when hv, in the block's shared memory (padding keys INT32_MAX).
template <typename T>
__device__ __forceinline__ void block_sort_row(int32_t *sk, T *sv, int N, bool hv) {
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int size = 2; size <= N; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int q = tid; q < N / 2; q += nt) {
                const int a = 2 * q - (q & (stride - 1)), b = a + stride;
                const bool up = (a & size) == 0;
                const int32_t ka = sk[a], kb = sk[b];
                if ((ka > kb) == up) {
                    sk[a] = kb;
                    sk[b] = ka;
                    if (hv) {
                        const T t = sv[a];
                        sv[a] = sv[b];
                        sv[b] = t;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// The listed rows of more than SORT_SHORT entries, a block each (taken by a
// ticket, as their lengths differ by orders of magnitude).  The columns of a
// row are distinct, so the place of an entry in column order is the number
// of the row's columns below its own: the columns are marked in a bitmap in
// shared memory, the marks counted (per 1024 columns by the marking itself,
// inside those by a warp each, only where there are any), and each entry
// looks up the marks below its bit and goes straight to its place.  Work per
// row: its entries three times from L1/L2 and two shared-memory atomics per
// entry, against the log^2 passes of a sorting network over the next power
// of two (300-edge batches of R-MAT 18, 27 million entries in rows of 2,000
// on average into host memory: 4.2 ms with the network in 196 KB of shared
// memory, one block per SM; 1.55 ms now, the link's rate.  A warp's register
// network for rows of up to 512 entries measured the same there).  Columns
// are taken in windows of W, from the row's first to its last, and a window
// keeps 4 blocks of 512 threads on an SM (50 KB at W = 2^18, OL_W).  A window
// takes about 3 us however few of the row's columns lie in it, so a short row
// over several of them goes through a network in the bitmap's memory instead
// (ow_by_network; 20,000 rows of 72 entries in a C of 2^22 columns: 831 us
// with the network in 196 KB, 1929 by windows, 250 so).  A row already in
// order (the dense kernels' rows) is copied.  With host arrays (out_col) the
// row is put together in device memory (dst_col, dst_val: it stays in L2) and
// stored to the host in order.
constexpr int OL_NT = 512;
// C wider than this: k_sort_long.  At this width 5000 rows of 6000 entries take
// 2.1 ms by their 16 windows and 4.1 by the network in 196 KB; at twice the
// width the windows would take as long.
constexpr int64_t OL_MAX_COLS = (int64_t)1 << 22;

static_assert(2 * OL_NET <= OL_W / 32, "the network's columns and places fit the bitmap of a whole window");

static size_t order_long_smem(int W) { return (size_t)W / 32 * 6 + (size_t)W / 1024 * 8; }

template <typename T>
__global__ void __launch_bounds__(OL_NT)
k_order_long(const int32_t *rows, MatView M, const int64_t *rp, const int64_t *long_list, int32_t *dst_col, T *dst_val,
             int32_t *out_col, T *out_val, bool has_val, ReadOut *res, int W) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *bm = (uint32_t *)smem;          // W / 32 words: the marked columns of the window
    uint32_t *cnt = bm + W / 32;              // W / 1024: marks per 1024 columns
    uint32_t *first = cnt + W / 1024;         // W / 1024: marks before them
    uint16_t *pre = (uint16_t *)(first + W / 1024);  // W / 32: marks before a word inside its 1024 columns
    __shared__ unsigned s_t;
    __shared__ int s_mn, s_mx;
    __shared__ uint32_t s_w[OL_NT / 32 + 1];
    if (res->flags) return;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned nl = res->n_long;
    const T *mv = (const T *)M.val;
    for (int q = tid; q < W / 32; q += OL_NT) bm[q] = 0u;
    for (int q = tid; q < W / 1024; q += OL_NT) cnt[q] = 0u;
    while (true) {
        if (tid == 0) {
            s_t = atomicAdd(&res->next, 1u);
            s_mn = INT32_MAX;
            s_mx = -1;
        }
        __syncthreads();
        const unsigned t = s_t;
        if (t >= nl) return;
        const int64_t x = long_list[t];
        const int64_t lo = rp[x];
        const int64_t len = rp[x + 1] - lo;
        const int64_t so = row_start(M, rows ? (int64_t)rows[x] : x, len);
        const int32_t *mc = M.col + so;
        int unsorted = 0;
        int mn = INT32_MAX, mx = -1;
#pragma unroll 4
        for (int64_t e = tid; e < len; e += OL_NT) {
            const int32_t c = mc[e];
            const int32_t nx = e + 1 < len ? mc[e + 1] : INT32_MAX;
            unsorted |= c > nx;
            if (ow_is_column(c, M.ncols)) {  // always, for a row that does not change meanwhile
                mn = min(mn, c);
                mx = max(mx, c);
            }
        }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) {
            atomicMin(&s_mn, mn);
            atomicMax(&s_mx, mx);
        }
        if (!__syncthreads_or(unsorted)) {
            int32_t *oc = out_col ? out_col : dst_col;
            T *ov = out_col ? out_val : dst_val;
#pragma unroll 4
            for (int64_t e = tid - (int64_t)(lo & 31); e < len; e += OL_NT)
                if (e >= 0) {
                    oc[lo + e] = mc[e];
                    if (has_val) ov[lo + e] = mv[so + e];
                }
            __syncthreads();  // every thread has read s_t, s_mn and s_mx
            continue;
        }
        mn = s_mn;
        mx = s_mx;
        if (mn > mx) {  // no column at all: a row that is being written
            __syncthreads();  // as above
            continue;
        }
        if (ow_by_network(len, (mx - ow_first(mn)) / W + 1)) {
            int N = 128;
            while (N < len) N <<= 1;
            int32_t *sk = (int32_t *)bm, *se = sk + N;  // columns, and where in the row they are
            for (int e = tid; e < N; e += OL_NT) {
                sk[e] = e < len ? mc[e] : INT32_MAX;
                se[e] = e < len ? e : 0;
            }
            __syncthreads();
            block_sort_row<int32_t>(sk, se, N, true);
            int32_t *oc = out_col ? out_col : dst_col;
            T *ov = out_col ? out_val : dst_val;
            for (int64_t e = tid - (int64_t)(lo & 31); e < len; e += OL_NT)
                if (e >= 0) {
                    oc[lo + e] = sk[e];
                    if (has_val) ov[lo + e] = mv[so + se[e]];
                }
            __syncthreads();
            for (int q = tid; q < 2 * N; q += OL_NT) bm[q] = 0u;
            continue;  // the next row's marks follow a barrier
        }
        uint32_t carry = 0;  // entries of the windows before
        for (int wb = ow_first(mn); wb <= mx; wb += W) {  // mx < M.ncols <= OL_MAX_COLS: no step overflows
            const int nb = ow_stretches(wb, mx, W);
            const uint32_t in = (uint32_t)nb * OL_STRETCH;
#pragma unroll 4
            for (int64_t e = tid; e < len; e += OL_NT) {
                const uint32_t c = ow_place(mc[e], wb);
                if (c < in) {
                    atomicOr(&bm[c >> 5], 1u << (c & 31));
                    atomicAdd(&cnt[c >> 10], 1u);
                }
            }
            __syncthreads();
            for (int b = w; b < nb; b += OL_NT / 32)
                if (cnt[b]) {
                    const uint32_t p = __popc(bm[b * 32 + lane]);
                    pre[b * 32 + lane] = (uint16_t)(warp_incl_scan<uint32_t>(p) - p);
                }
            // marks before each stretch: nb <= OL_W / 1024 <= OL_NT, one a thread
            const uint32_t v = tid < nb ? cnt[tid] : 0u;
            const uint32_t incl = warp_incl_scan<uint32_t>(v);
            if (lane == 31) s_w[w] = incl;
            __syncthreads();
            if (w == 0) {
                const uint32_t a = lane < OL_NT / 32 ? s_w[lane] : 0u;
                const uint32_t ai = warp_incl_scan<uint32_t>(a);
                if (lane < OL_NT / 32) s_w[lane] = ai - a;
                if (lane == 31) s_w[OL_NT / 32] = ai;
            }
            __syncthreads();
            if (tid < nb) first[tid] = carry + s_w[w] + incl - v;
            carry += s_w[OL_NT / 32];
            __syncthreads();
#pragma unroll 4
            for (int64_t e = tid; e < len; e += OL_NT) {
                const int32_t col = mc[e];
                const uint32_t c = ow_place(col, wb);
                if (c < in) {
                    const uint32_t o = first[c >> 10] + pre[c >> 5] + __popc(bm[c >> 5] & ((1u << (c & 31)) - 1u));
                    if (o < (uint64_t)len) {  // always, for a row that does not change meanwhile
                        dst_col[lo + o] = col;
                        if (has_val) dst_val[lo + o] = mv[so + e];
                    }
                }
            }
            __syncthreads();
            for (int b = w; b < nb; b += OL_NT / 32)
                if (cnt[b]) {
                    bm[b * 32 + lane] = 0u;
                    __syncwarp();
                    if (lane == 0) cnt[b] = 0u;
                }
            __syncthreads();
        }
        if (out_col) {
#pragma unroll 4
            for (int64_t e = tid - (int64_t)(lo & 31); e < len; e += OL_NT)
                if (e >= 0) {
                    out_col[lo + e] = __ldcg(dst_col + lo + e);
                    if (has_val) out_val[lo + e] = __ldcg(dst_val + lo + e);
                }
        }
    }
}

// The listed rows of a C wider than OL_MAX_COLS, a block each: put in column
// order in shared memory (unless in order already); rows over SORT_MAX
// entries are copied as they are to dst and listed again (huge_list) for
// sort_listed_rows.
template <typename T>
__global__ void __launch_bounds__(512)
k_sort_long(const int32_t *rows, MatView M, const int64_t *rp, const int64_t *long_list, int32_t *dst_col, T *dst_val,
            int32_t *out_col, T *out_val, bool has_val, int64_t *huge_list, ReadOut *res) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    T *sv = (T *)smem;
    int32_t *sk = (int32_t *)(sv + SORT_MAX);
    if (res->flags) return;
    const unsigned nl = res->n_long;
    const int tid = threadIdx.x, nt = blockDim.x;
    const T *mv = (const T *)M.val;
    int32_t *oc = out_col ? out_col : dst_col;
    T *ov = out_col ? out_val : dst_val;
    for (unsigned j = blockIdx.x; j < nl; j += gridDim.x) {
        const int64_t x = long_list[j];
        const int64_t lo = rp[x];
        const int64_t len = rp[x + 1] - lo;
        const int64_t so = row_start(M, rows ? (int64_t)rows[x] : x, len);
        int unsorted = 0;
        for (int64_t e = tid; e + 1 < len; e += nt) unsorted |= M.col[so + e] > M.col[so + e + 1];
        const bool sort = __syncthreads_or(unsorted);
        if (!sort || len > SORT_MAX) {
            int32_t *tc = sort ? dst_col : oc;
            T *tv = sort ? dst_val : ov;
            for (int64_t e = tid; e < len; e += nt) {
                tc[lo + e] = M.col[so + e];
                if (has_val) tv[lo + e] = mv[so + e];
            }
            if (sort && tid == 0) huge_list[atomicAdd(&res->n_huge, 1u)] = x;
            continue;
        }
        int N = 128;
        while (N < len) N <<= 1;
        for (int e = tid; e < N; e += nt) {
            sk[e] = e < len ? M.col[so + e] : INT32_MAX;
            if (has_val && e < len) sv[e] = mv[so + e];
        }
        __syncthreads();
        block_sort_row<T>(sk, sv, N, has_val);
        for (int e = tid; e < len; e += nt) {
            oc[lo + e] = sk[e];
            if (has_val) ov[lo + e] = sv[e];
        }
        __syncthreads();
    }
}

template <typename T>
static void read_rows_out_t(const int32_t *rows, int64_t n, const long long *n_dev, const MatView &M, bool has_val,
                            const int64_t *rp, const int64_t *r_total, int64_t nnz_cap, int32_t *dst_col, T *dst_val,
                            int32_t *out_col, T *out_val, int64_t *long_list, int64_t *huge_list, ReadOut *res,
                            ReadOut *host_res, cudaStream_t s, int num_sms) {
    // n on the device: n is the host's bound on it, which sizes the grids.
    // One wave of resident blocks: a partial second one left SMs idle (the
    // 128^3 stencil's square into device memory: 398 us with 8 blocks an SM
    // launched of which 5 fit, 354 so).
    static const int per_sm = resident_blocks(k_read_short<T>, RS_NT);
    launch_k(k_read_short<T>, blocks_for(std::max<int64_t>(n, 1), RS_ROWS, (int64_t)num_sms * per_sm), RS_NT, 0, s, rows, n,
             n_dev, M, rp, r_total, nnz_cap, out_col ? out_col : dst_col,
             has_val ? (out_col ? out_val : dst_val) : (T *)nullptr, long_list, res, host_res);
    if (M.ncols <= OL_MAX_COLS) {
        const int W = (int)std::min<int64_t>(OL_W, std::max<int64_t>(1, (M.ncols + 1023) / 1024) * 1024);
        const size_t smem = order_long_smem(W);
        static bool set = false;
        if (!set) {
            cudaFuncSetAttribute(k_order_long<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)order_long_smem(OL_W));
            set = true;
        }
        launch_k(k_order_long<T>, (unsigned)std::max<int64_t>(1, std::min<int64_t>(n, (int64_t)num_sms * 4)), OL_NT,
                 smem, s, rows, M, rp, (const int64_t *)long_list, dst_col, dst_val, out_col, out_val, has_val, res, W);
        return;
    }
    const size_t smem = (size_t)SORT_MAX * (sizeof(T) + sizeof(int32_t));
    static bool set = false;
    if (!set) {
        cudaFuncSetAttribute(k_sort_long<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        set = true;
    }
    launch_k(k_sort_long<T>, (unsigned)std::max<int64_t>(1, std::min<int64_t>(n, (int64_t)num_sms * 2)), 512, smem, s,
             rows, M, rp, (const int64_t *)long_list, dst_col, dst_val, out_col, out_val, has_val, huge_list, res);
}

bool read_has_huge(int64_t ncols) { return ncols > OL_MAX_COLS; }

void read_rows_out(const int32_t *rows, int64_t n, const long long *n_dev, const MatView &M, int vsize,
                   const int64_t *rp, const int64_t *r_total, int64_t nnz_cap, int32_t *dst_col, void *dst_val,
                   int32_t *out_col, void *out_val, int64_t *long_list, int64_t *huge_list, ReadOut *res,
                   ReadOut *host_res, cudaStream_t s, int num_sms) {
    const bool has_val = vsize && M.val && (out_col ? out_val != nullptr : dst_val != nullptr);
    if (vsize == 8)
        read_rows_out_t<double>(rows, n, n_dev, M, has_val, rp, r_total, nnz_cap, dst_col, (double *)dst_val, out_col,
                                (double *)out_val, long_list, huge_list, res, host_res, s, num_sms);
    else
        read_rows_out_t<int32_t>(rows, n, n_dev, M, has_val, rp, r_total, nnz_cap, dst_col, (int32_t *)dst_val, out_col,
                                 (int32_t *)out_val, long_list, huge_list, res, host_res, s, num_sms);
}

// Rows too long for a CTA's shared memory, sorted all at once: the packed
// key (list index << cb | column) of every entry of the listed rows goes
// through the LSD radix sort with its place in the rows' concatenation,
// then each entry is gathered into its sorted place and copied back.
// pre[k] = entries of the listed rows before row k (pre[nl] = their total).
__device__ __forceinline__ int list_of(const int64_t *pre, int nl, int64_t q) {
    int lo = 0, hi = nl;  // the k with pre[k] <= q < pre[k + 1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (pre[mid] <= q) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void k_listed_keys(const int64_t *rowptr, const int64_t *listed, const int64_t *pre, int nl, int cb,
                              const int32_t *col, uint64_t *keys, uint32_t *idx) {
    pdl_begin();
    const int64_t E = pre[nl];
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < E; q += (int64_t)gridDim.x * blockDim.x) {
        const int k = list_of(pre, nl, q);
        const int64_t p = rowptr[listed[k]] + (q - pre[k]);
        keys[q] = ow_list_key((uint64_t)k, col[p], cb);
        idx[q] = (uint32_t)q;
    }
}

template <typename T>
__global__ void k_listed_gather(const int64_t *rowptr, const int64_t *listed, const int64_t *pre, int nl,
                                const uint32_t *idx, const int32_t *col, const T *val, int32_t *tcol, T *tval) {
    pdl_begin();
    const int64_t E = pre[nl];
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < E; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t src = idx[q];  // the same row as q: the keys sort by list index first
        const int k = list_of(pre, nl, src);
        const int64_t p = rowptr[listed[k]] + (src - pre[k]);
        tcol[q] = col[p];
        if (val) tval[q] = val[p];
    }
}

template <typename T>
__global__ void k_listed_back(const int64_t *rowptr, const int64_t *listed, const int64_t *pre, int nl,
                              const int32_t *tcol, const T *tval, int32_t *col, T *val) {
    pdl_begin();
    const int64_t E = pre[nl];
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < E; q += (int64_t)gridDim.x * blockDim.x) {
        const int k = list_of(pre, nl, q);
        const int64_t p = rowptr[listed[k]] + (q - pre[k]);
        col[p] = tcol[q];
        if (val) val[p] = tval[q];
    }
}

void sort_listed_rows(const int64_t *rowptr, const int64_t *listed, const int64_t *pre, int nl, int64_t total,
                      int cb, int32_t *col, void *val, int vsize, const SortScratch &w, cudaStream_t s, int num_sms) {
    if (nl <= 0 || total <= 0) return;
    const unsigned g = blocks_for(total, 256, (int64_t)num_sms * 8);
    launch_k(k_listed_keys, g, 256, 0, s, rowptr, listed, pre, nl, cb, col, w.k0, w.i0);
    bool alt = false;
    radix_sort_pairs(w.k0, w.i0, w.k1, w.i1, total, bits_for(nl) + cb, w.counts, w.scan_tmp, w.scan_out, s, &alt);
    const uint32_t *idx = alt ? w.i1 : w.i0;
    if (vsize == 8) {
        launch_k(k_listed_gather<double>, g, 256, 0, s, rowptr, listed, pre, nl, idx, col, (const double *)val, w.tcol,
                 (double *)w.tval);
        launch_k(k_listed_back<double>, g, 256, 0, s, rowptr, listed, pre, nl, (const int32_t *)w.tcol,
                 (const double *)w.tval, col, (double *)val);
    } else {
        launch_k(k_listed_gather<int32_t>, g, 256, 0, s, rowptr, listed, pre, nl, idx, col, (const int32_t *)val,
                 w.tcol, (int32_t *)w.tval);
        launch_k(k_listed_back<int32_t>, g, 256, 0, s, rowptr, listed, pre, nl, (const int32_t *)w.tcol,
                 (const int32_t *)w.tval, col, (int32_t *)val);
    }
}

// Canonical-CSR check: rowptr[0] = 0 and non-decreasing, rowptr[n] = nnz,
// columns in range and strictly ascending per row, values valid for the
// semiring.  Sets *bad = 1 on the first violation seen.
__global__ void k_validate_rows(int64_t nrows, int64_t ncols, int64_t nnz, const int64_t *rowptr, unsigned *bad) {
    pdl_begin();
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= nrows;
         r += (int64_t)gridDim.x * blockDim.x) {
        if (r == 0 && rowptr[0] != 0) atomicOr(bad, 1u);
        if (r == nrows && rowptr[nrows] != nnz) atomicOr(bad, 1u);
        if (r < nrows && rowptr[r + 1] < rowptr[r]) atomicOr(bad, 1u);
    }
}

__global__ void k_validate_entries(int64_t nrows, int64_t ncols, const int64_t *rowptr, const int32_t *col,
                                   const void *val, int sr, unsigned *bad) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nrows; r += nwarps) {
        const int64_t lo = rowptr[r], hi = rowptr[r + 1];
        if (hi < lo) continue;
        for (int64_t p = lo + lane; p < hi; p += 32) {
            const int32_t c = col[p];
            bool ok = c >= 0 && (int64_t)c < ncols && (p == lo || col[p - 1] < c);
            if (sr == SR_PT) ok = ok && isfinite(((const double *)val)[p]);
            else {
                const int32_t v = ((const int32_t *)val)[p];
                ok = ok && v > -MP_LIMIT && v < MP_LIMIT;
            }
            if (!ok) atomicOr(bad, 1u);
        }
    }
}

// Entry check, run only after the row bounds have been verified on the host.
void validate_csr_entries(int64_t nrows, int64_t ncols, const int64_t *rowptr, const int32_t *col, const void *val,
                          int sr, unsigned *bad, cudaStream_t s) {
    if (nrows > 0)
        launch_k(k_validate_entries, blocks_for(nrows * 32, 256, 8192), 256, 0, s, nrows, ncols, rowptr, col, val, sr, bad);
}

void validate_rowptr(int64_t nrows, int64_t nnz, const int64_t *rowptr, unsigned *bad, cudaStream_t s) {
    launch_k(k_validate_rows, blocks_for(nrows + 1, 256, 4096), 256, 0, s, nrows, 0, nnz, rowptr, bad);
}

__global__ void k_hist_cols(const int32_t *col, int64_t nnz, int32_t *counts) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nnz; x += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&counts[col[x]], 1);
}
void hist_cols(const int32_t *col, int64_t nnz, int32_t *counts, cudaStream_t s) {
    if (nnz > 0) launch_k(k_hist_cols, blocks_for(nnz, 256, 8192), 256, 0, s, col, nnz, counts);
}

__global__ void k_rows_of_entries(const int64_t *rowptr, int64_t nrows, uint32_t *rows_out) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nrows; r += nwarps)
        for (int64_t p = rowptr[r] + lane; p < rowptr[r + 1]; p += 32) rows_out[p] = (uint32_t)r;
}
void rows_of_entries(const int64_t *rowptr, int64_t nrows, uint32_t *rows_out, cudaStream_t s, int num_sms) {
    if (nrows > 0)
        launch_k(k_rows_of_entries, blocks_for(nrows * 32, 256, (int64_t)num_sms * 16), 256, 0, s, rowptr, nrows, rows_out);
}

__global__ void k_keys_from_cols(const int32_t *col, int64_t nnz, uint64_t *keys) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nnz; x += (int64_t)gridDim.x * blockDim.x)
        keys[x] = (uint64_t)(uint32_t)col[x];
}
void keys_from_cols(const int32_t *col, int64_t nnz, uint64_t *keys, cudaStream_t s) {
    if (nnz > 0) launch_k(k_keys_from_cols, blocks_for(nnz, 256, 8192), 256, 0, s, col, nnz, keys);
}

__global__ void k_keys_from_i32(const int32_t *a, int64_t n, uint64_t *keys, uint32_t *idx) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        keys[x] = (uint64_t)(uint32_t)a[x];
        idx[x] = (uint32_t)x;
    }
}
__global__ void k_keys_to_i32(const uint64_t *keys, int64_t n, int32_t *a) {
    pdl_begin();
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        a[x] = (int32_t)keys[x];
}
void sort_i32_values(int32_t *a, int64_t n, int bits, uint64_t *k0, uint64_t *k1, uint32_t *i0, uint32_t *i1,
                     uint32_t *counts, int64_t *scan_tmp, int64_t *scan_out, cudaStream_t s) {
    if (n <= 1) return;
    launch_k(k_keys_from_i32, blocks_for(n, 256, 8192), 256, 0, s, a, n, k0, i0);
    bool alt = false;
    radix_sort_pairs(k0, i0, k1, i1, n, bits, counts, scan_tmp, scan_out, s, &alt);
    launch_k(k_keys_to_i32, blocks_for(n, 256, 8192), 256, 0, s, alt ? k1 : k0, n, a);
}

}  // namespace dspg
