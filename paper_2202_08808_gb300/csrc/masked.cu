// masked.cu -- general updates by the entry-level masked recompute
// (Section 5.2, Algorithm 2), and the Bloom filter F that it keeps.
//
// F has C's pattern and a 64-bit word per entry: bit (k mod 64) of F(i,j)
// is set when the term A(i,k) B(k,j) contributes to C(i,j) (Section 5.2,
// l = 64).  On one GPU the words sit beside C's values in C's arena (same
// offsets), so every move of a row of C moves its words too.
//
// A batch of general updates (inserts, deletes, value changes of A and B)
// is applied in the paper's order:
//
//  1. computePattern: the pattern of C* = A* B' + A B* (Eq. 1), with F*:
//     each changed entry (i,k) of A meets the row k of B' (contribution
//     (i, j, bit k)); each changed entry (k,j) of B meets the rows i with
//     A(i,k) != 0 before the batch, read from the transposed pattern of A
//     before it is updated (contribution (i, j, bit k)).  The contributions
//     are sorted by (i, j) with the radix sort of the batch and equal keys
//     are merged (bits OR-ed): C* as sorted runs, one run per row.
//  2. E = (F | F*) at the entries of C*, and R_i = OR of E over row i
//     (k_mask_scan: the row of C is scanned once, each of its columns looked
//     up in the row's run of C*).
//  3. A^R: the entries (i,k) of A' whose bit (k mod 64) is set in R_i
//     (k_mask_keep).
//  4. Z, H = A^R B' masked at C* (k_mask_product): each kept (i,k,a) meets
//     row k of B'; a product whose column j is in row i's run of C* is
//     folded into Z(i,j) and sets bit k of H(i,j).
//  5. Merge Z into C and H into F at C*'s entries (k_mask_plan,
//     k_mask_splice): an entry of C* that received a product takes its new
//     value and word (written in place, or where C had no entry there, in
//     the place of one that leaves or at the row's end); one that received
//     none leaves C, and the row's last entries move into the places left.
//     The other entries of C outside C* are not touched.
//
// Every k that contributes to an entry of C* at the end has its bit in E
// (it contributed before, or one of its two factors changed), so A^R keeps
// every term of every masked entry; terms it keeps beyond those (bits
// shared modulo 64) reach no masked column or are genuine terms anyway.
//
// The static product's F comes from k_bloom_warp (a warp per row, the
// row's columns in a shared-memory table) and k_bloom_cta (rows longer than
// BL_WARP entries, a CTA with a dense column-to-place map in global memory).
#include "internal.h"

namespace dspg {

namespace {

constexpr int BL_WARP = 512;    // rows up to this many entries: the warp kernel
constexpr int BL_SLOTS = 1024;  // its table: at most half full
constexpr int BL_NW = 2;        // warps per block of the warp kernel (static shared memory)

__device__ __forceinline__ unsigned long long kbit(int32_t k) { return 1ull << (k & 63); }

__device__ __forceinline__ unsigned long long warp_or(unsigned long long v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// Slot of column j in a warp's table (inserting it when absent and
// insert is set); -1 when absent (or the table is full, which the row
// bound rules out).
__device__ __forceinline__ int bl_slot(int32_t *keys, int32_t j, bool insert) {
    uint32_t h = ((uint32_t)j * 2654435761u) >> (32 - 10);
    for (int probe = 0; probe < BL_SLOTS; probe++) {
        const int32_t k = ((volatile int32_t *)keys)[h];
        if (k == j) return (int)h;
        if (k == -1) {
            if (!insert) return -1;
            const int32_t old = atomicCAS(&keys[h], -1, j);
            if (old == -1 || old == j) return (int)h;
        }
        h = (h + probe + 1) & (BL_SLOTS - 1);
    }
    return -1;
}

__global__ void __launch_bounds__(BL_NW * 32)
k_bloom_warp(MatView A, MatView B, MatView C, unsigned long long *F, int32_t *rows_long, long long *n_long,
             long long cap_long) {
    pdl_begin();
    __shared__ int32_t s_key[BL_NW][BL_SLOTS];
    __shared__ unsigned long long s_bits[BL_NW][BL_SLOTS];
    __shared__ int16_t s_slot[BL_NW][BL_WARP];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t *keys = s_key[w];
    unsigned long long *bits = s_bits[w];
    int16_t *slot = s_slot[w];
    for (int q = lane; q < BL_SLOTS; q += 32) {
        keys[q] = -1;
        bits[q] = 0ull;
    }
    __syncwarp();
    const long long nw = (long long)gridDim.x * BL_NW;
    for (long long i = (long long)blockIdx.x * BL_NW + w; i < C.nrows; i += nw) {
        const int L = C.len[i];
        if (L == 0) continue;
        if (L > BL_WARP) {
            if (lane == 0) {
                const long long t = atomicAdd((unsigned long long *)n_long, 1ull);
                if (t < cap_long) rows_long[t] = (int32_t)i;
            }
            continue;
        }
        const int64_t coff = C.off[i];
        for (int p = lane; p < L; p += 32) slot[p] = (int16_t)bl_slot(keys, C.col[coff + p], true);
        __syncwarp();
        const int64_t aoff = A.off[i];
        const int alen = A.len[i];
        for (int a = 0; a < alen; a++) {
            const int32_t k = A.col[aoff + a];
            const unsigned long long b = kbit(k);
            const int64_t bo = B.off[k];
            const int bl = B.len[k];
            for (int q = lane; q < bl; q += 32) {
                const int h = bl_slot(keys, B.col[bo + q], false);
                if (h >= 0) atomicOr(&bits[h], b);
            }
        }
        __syncwarp();
        for (int p = lane; p < L; p += 32) {
            const int h = slot[p];
            if (h >= 0) {
                F[coff + p] = bits[h];
                keys[h] = -1;
                bits[h] = 0ull;
            }
        }
        __syncwarp();
    }
}

// Rows longer than BL_WARP: a CTA per row, with pos[j] = the place of
// column j in the row (this CTA's m entries of posmap, -1 elsewhere).
__global__ void __launch_bounds__(512)
k_bloom_cta(MatView A, MatView B, MatView C, unsigned long long *F, const int32_t *rows_long, const long long *n_long,
            long long cap_long, int32_t *posmap) {
    pdl_begin();
    int32_t *pos = posmap + (int64_t)blockIdx.x * C.ncols;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
    const long long n = *n_long < cap_long ? *n_long : cap_long;
    for (long long t = blockIdx.x; t < n; t += gridDim.x) {
        const int32_t i = rows_long[t];
        const int64_t coff = C.off[i];
        const int L = C.len[i];
        for (int p = tid; p < L; p += blockDim.x) {
            pos[C.col[coff + p]] = p;
            F[coff + p] = 0ull;
        }
        __syncthreads();
        const int64_t aoff = A.off[i];
        const int alen = A.len[i];
        for (int a = w; a < alen; a += nw) {
            const int32_t k = A.col[aoff + a];
            const unsigned long long b = kbit(k);
            const int64_t bo = B.off[k];
            const int bl = B.len[k];
            for (int q = lane; q < bl; q += 32) {
                const int32_t p = pos[B.col[bo + q]];
                if (p >= 0) atomicOr(&F[coff + p], b);
            }
        }
        __syncthreads();
        for (int p = tid; p < L; p += blockDim.x) pos[C.col[coff + p]] = -1;
        __syncthreads();
    }
}

// ------------------------------------------------------- computePattern

__device__ __forceinline__ void pat_emit(const PatJob &J, Ctl *ctl, bool ok, int32_t i, int32_t j, int32_t k) {
    const long long t = warp_fetch_add(&ctl->mask_n, ok ? 1 : 0);
    if (ok) {
        if (t < J.cap) {
            J.key[t] = ((uint64_t)(uint32_t)i << J.cb) | (uint32_t)j;
            J.bits[t] = kbit(k);
        } else {
            set_status(ctl, ST_MASK_FULL);
        }
    }
}

// A warp per batch entry that changes its matrix: the X term (A batch
// against B') and the Y term (B batch against the old pattern of A).
__global__ void k_pat_contrib(PatJob J, MatView B, MatView AT, Ctl *ctl, unsigned mask) {
    pdl_begin();
    if (__any_sync(0xffffffffu, failed(ctl, mask))) return;
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (long long e = w0; e < J.xn; e += nwarps) {
        if (J.xk[e] == K_NOP) continue;  // the same e on every lane
        const int32_t i = J.xr[e], k = J.xc[e];
        const int64_t bo = B.off[k];
        const int bl = B.len[k];
        for (int q0 = 0; q0 < bl; q0 += 32) {
            const int q = q0 + lane;
            const bool ok = q < bl;
            pat_emit(J, ctl, ok, i, ok ? B.col[bo + q] : 0, k);
        }
    }
    for (long long e = w0; e < J.yn; e += nwarps) {
        if (J.yk[e] == K_NOP) continue;
        const int32_t k = J.yr[e], j = J.yc[e];
        const int64_t to = AT.off[k];
        const int tl = AT.len[k];
        for (int q0 = 0; q0 < tl; q0 += 32) {
            const int q = q0 + lane;
            const bool ok = q < tl;
            pat_emit(J, ctl, ok, ok ? AT.col[to + q] : 0, j, k);
        }
    }
}

__global__ void k_iota(uint32_t *v, int64_t n) {
    pdl_begin();
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        v[t] = (uint32_t)t;
}

// flag[s] = 1 where a run of equal keys starts.
__global__ void k_pat_heads(const uint64_t *K, int64_t n, int32_t *flag) {
    pdl_begin();
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x)
        flag[s] = (s == 0 || K[s] != K[s - 1]) ? 1 : 0;
}

// Each run of equal keys becomes entry u = ex[s] of C*: its row and
// column, and F* = OR of the run's bits; rflag[u] = 1 where a row starts.
__global__ void k_pat_unique(const uint64_t *K, const uint32_t *I, const uint64_t *bits, int64_t n,
                             const int64_t *ex, int cb, MaskJob M, int32_t *rflag) {
    pdl_begin();
    const uint64_t cmask = (uint64_t(1) << cb) - 1;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = K[s];
        if (s > 0 && K[s - 1] == key) continue;
        unsigned long long f = 0;
        for (int64_t t = s; t < n && K[t] == key; t++) f |= bits[I[t]];
        const int64_t u = ex[s];
        M.urow[u] = (int32_t)(key >> cb);
        M.ucol[u] = (int32_t)(key & cmask);
        M.ufs[u] = f;
        rflag[u] = (s == 0 || (K[s - 1] >> cb) != (key >> cb)) ? 1 : 0;
    }
}

// Runs of C* per row: start and row of run r = rex[u]; the row's bit in
// bm; and the end of the last run.
__global__ void k_pat_runs(MaskJob M, const int32_t *rflag, const int64_t *rex, uint32_t *bm) {
    pdl_begin();
    const int64_t nu = *M.nu_dev;
    if (blockIdx.x == 0 && threadIdx.x == 0) M.run_start[*M.nruns_dev] = nu;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += (int64_t)gridDim.x * blockDim.x) {
        if (!rflag[u]) continue;
        const int64_t r = rex[u];
        const int32_t i = M.urow[u];
        M.run_start[r] = u;
        M.run_row[r] = i;
        atomicOr(&bm[i >> 5], 1u << (i & 31));
    }
}

// --------------------------------------------------- E, R and A^R

// The entries of a row of C that are in its run of C*: their places and
// words of F.  The row is read once, MS_U loads a thread in flight, and a
// column goes on to the search of the run only when its bit of a filter of
// the run's columns (nw words of shared memory, a bit per column) is set:
// runs are a few entries long (2 on R-MAT with 1000 edges) and rows
// thousands.  The nt threads t (a warp, or the block with BLOCK) share the row.
constexpr int MS_NT = 256;
constexpr int MS_U = 8;
constexpr int MS_LONG = 2048;  // rows of more entries are read by the whole block (8192, with 4 loads in flight: 190 us)

template <bool BLOCK>
__device__ __forceinline__ void mask_scan_row(const MaskJob &M, const MatView &C, const unsigned long long *F, int64_t u0,
                                              int64_t u1, int64_t coff, int L, uint32_t *filter, int lognw, int t) {
    constexpr int NT = BLOCK ? MS_NT : 32;
    auto sync = [&]() {
        if (BLOCK) __syncthreads();
        else __syncwarp();
    };
    const int shift = 32 - 5 - lognw;
    for (int q = t; q < (1 << lognw); q += NT) filter[q] = 0u;
    sync();
    for (int64_t u = u0 + t; u < u1; u += NT) {
        const uint32_t hsh = ((uint32_t)M.ucol[u] * 2654435761u) >> shift;
        atomicOr(&filter[hsh >> 5], 1u << (hsh & 31));
    }
    sync();
    for (int p0 = t; p0 < L; p0 += NT * MS_U) {
        int32_t j[MS_U];
#pragma unroll
        for (int q = 0; q < MS_U; q++) j[q] = p0 + q * NT < L ? C.col[coff + p0 + q * NT] : -1;
#pragma unroll
        for (int q = 0; q < MS_U; q++) {
            const uint32_t hsh = ((uint32_t)j[q] * 2654435761u) >> shift;
            if (j[q] < 0 || !((filter[hsh >> 5] >> (hsh & 31)) & 1u)) continue;
            const int64_t u = lower_bound_dev<int32_t>(M.ucol, u0, u1, j[q]);
            if (u < u1 && M.ucol[u] == j[q]) {
                M.upos[u] = p0 + q * NT;
                M.ue[u] = F[coff + p0 + q * NT];
            }
        }
    }
    sync();
}

// R_i = OR over the run of (F | F*), by a warp.
__device__ __forceinline__ void mask_row_bits(const MaskJob &M, int64_t r, int64_t u0, int64_t u1, int lane) {
    unsigned long long rb = 0;
    for (int64_t u = u0 + lane; u < u1; u += 32) rb |= M.ue[u] | M.ufs[u];
    rb = warp_or(rb);
    if (lane == 0) M.rbits[r] = rb;
}

// A warp per run, the rows of more than MS_LONG entries by the whole block at
// the end of its round.  Bound by the read of the rows (4 bytes an entry);
// with a search per entry in global memory, a load after the other, the
// kernel took 448 us on 1000 edges of R-MAT 17, 124 us now.
__global__ void __launch_bounds__(MS_NT) k_mask_scan(MaskJob M, MatView C, const unsigned long long *F) {
    pdl_begin();
    __shared__ uint32_t s_filter[MS_NT / 32 * 32];
    __shared__ long long s_long[MS_NT / 32];
    __shared__ int s_nlong;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long nr = *M.nruns_dev;
    for (long long r0 = (long long)blockIdx.x * (MS_NT / 32); r0 < nr; r0 += (long long)gridDim.x * (MS_NT / 32)) {
        if (tid == 0) s_nlong = 0;
        __syncthreads();
        const long long r = r0 + w;
        if (r < nr) {
            const int64_t u0 = M.run_start[r], u1 = M.run_start[r + 1];
            const int32_t i = M.run_row[r];
            const int64_t coff = C.off[i];
            const int L = C.len[i];
            if (L > MS_LONG) {
                if (lane == 0) s_long[atomicAdd(&s_nlong, 1)] = r;
            } else {
                mask_scan_row<false>(M, C, F, u0, u1, coff, L, s_filter + w * 32, 5, lane);
                mask_row_bits(M, r, u0, u1, lane);
            }
        }
        __syncthreads();
        const int nl = s_nlong;
        for (int q = 0; q < nl; q++) {
            const long long rl = s_long[q];
            const int64_t u0 = M.run_start[rl], u1 = M.run_start[rl + 1];
            const int32_t i = M.run_row[rl];
            mask_scan_row<true>(M, C, F, u0, u1, C.off[i], C.len[i], s_filter, 8, tid);
            if (w == 0) mask_row_bits(M, rl, u0, u1, lane);
        }
        __syncthreads();
    }
}
static_assert(MS_NT / 32 * 32 == 1 << 8, "the block's filter");

// A warp per run: the entries of row i of A' whose bit is set in R_i.  They
// are counted first, so that a block takes its runs' places with one atomic:
// an atomic per 32 entries on the one counter took 414 us on 1000 edges of
// R-MAT 17, 14 us now.
constexpr int MK_U = 4;
__global__ void __launch_bounds__(256) k_mask_keep(MaskJob M, MatView A, Ctl *ctl) {
    pdl_begin();
    __shared__ int s_n[8];
    __shared__ long long s_base;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const long long nr = *M.nruns_dev;
    for (long long r0 = (long long)blockIdx.x * 8; r0 < nr; r0 += (long long)gridDim.x * 8) {
        const long long r = r0 + w;
        unsigned long long rb = 0ull;
        int64_t aoff = 0;
        int alen = 0;
        if (r < nr) {
            const int32_t i = M.run_row[r];
            rb = M.rbits[r];
            aoff = A.off[i];
            alen = A.len[i];
        }
        int n = 0;
        for (int q0 = lane; q0 < alen; q0 += 32 * MK_U) {
            int32_t k[MK_U];
#pragma unroll
            for (int q = 0; q < MK_U; q++) k[q] = q0 + 32 * q < alen ? A.col[aoff + q0 + 32 * q] : -1;
#pragma unroll
            for (int q = 0; q < MK_U; q++) n += k[q] >= 0 && (rb & kbit(k[q])) != 0ull;
        }
        n = warp_sum<int>(n);
        if (lane == 0) s_n[w] = n;
        __syncthreads();
        if (tid == 0) {
            int tot = 0;
            for (int q = 0; q < 8; q++) {
                const int v = s_n[q];
                s_n[q] = tot;
                tot += v;
            }
            s_base = tot ? (long long)atomicAdd((unsigned long long *)&ctl->mask_kept, (unsigned long long)tot) : 0;
        }
        __syncthreads();
        long long t = s_base + s_n[w];
        if (n > 0) {
            for (int q0 = 0; q0 < alen; q0 += 32) {
                const int q = q0 + lane;
                const bool keep = q < alen && ((rb & kbit(A.col[aoff + q])) != 0ull);
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                const long long at = t + __popc(bal & lanemask_lt());
                if (keep) {
                    if (at < M.kcap) {
                        M.kept_run[at] = (int32_t)r;
                        M.kept_a[at] = aoff + q;
                    } else {
                        set_status(ctl, ST_MASK_FULL);
                    }
                }
                t += __popc(bal);
            }
        }
        __syncthreads();  // s_n and s_base are read before the next round writes them
    }
}

// ------------------------------------------------ the masked product

template <int SR>
struct MSr;
template <>
struct MSr<SR_PT> {
    using T = double;
    __device__ static T mul(T a, T b) { return __dmul_rn(a, b); }
    __device__ static void acc(T *p, T v) { atomicAdd(p, v); }
};
template <>
struct MSr<SR_MP> {
    using T = int32_t;
    __device__ static T mul(T a, T b) { return a + b; }
    __device__ static void acc(T *p, T v) { atomicMin(p, v); }
};

// A warp per kept entry (i, k, a): the products with row k of B' whose
// column is in row i's run of C*.
template <int SR>
__global__ void k_mask_product(MaskJob M, MatView A, MatView B, Ctl *ctl, unsigned mask) {
    pdl_begin();
    using T = typename MSr<SR>::T;
    if (failed(ctl, mask)) return;  // no barrier or shuffle below
    const int lane = threadIdx.x & 31;
    const long long nk = *M.nkept_dev < M.kcap ? *M.nkept_dev : M.kcap;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const T *Av = (const T *)A.val;
    const T *Bv = (const T *)B.val;
    T *z = (T *)M.z;
    long long prods = 0;
    for (long long t = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nk; t += nwarps) {
        const int32_t r = M.kept_run[t];
        const int64_t ae = M.kept_a[t];
        const int32_t k = A.col[ae];
        const T a = Av[ae];
        const unsigned long long b = kbit(k);
        const int64_t u0 = M.run_start[r], u1 = M.run_start[r + 1];
        const int64_t bo = B.off[k];
        const int bl = B.len[k];
        for (int q = lane; q < bl; q += 32) {
            const int32_t j = B.col[bo + q];
            const int64_t u = lower_bound_dev<int32_t>(M.ucol, u0, u1, j);
            if (u < u1 && M.ucol[u] == j) {
                MSr<SR>::acc(z + u, MSr<SR>::mul(a, Bv[bo + q]));
                atomicOr(&M.h[u], b);
                M.hit[u] = 1;
            }
        }
        prods += bl;
    }
    if (lane == 0 && prods) atomicAdd((unsigned long long *)&ctl->products, (unsigned long long)prods);
}

// ------------------------------------------------------------ merge

// A warp per run: the row's length after the merge (deleted entries out,
// new entries in); a row that outgrows its capacity gets a place at the
// arena tail (nothing is written when the arena is exhausted).
__global__ void k_mask_plan(MaskJob M, MatView C, Ctl *ctl, unsigned mask, int slack_min, int slack_div) {
    pdl_begin();
    if (__any_sync(0xffffffffu, failed(ctl, mask))) return;  // a warp leaves as a whole
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long nr = *M.nruns_dev;
    for (long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nr; r += nwarps) {
        const int64_t u0 = M.run_start[r], u1 = M.run_start[r + 1];
        int ndel = 0, nins = 0;
        for (int64_t u = u0 + lane; u < u1; u += 32) {
            const bool in_c = M.upos[u] >= 0, hit = M.hit[u] != 0;
            ndel += in_c && !hit;
            nins += !in_c && hit;
        }
        ndel = warp_sum<int>(ndel);
        nins = warp_sum<int>(nins);
        if (lane == 0) {
            const int32_t i = M.run_row[r];
            const int64_t L2 = (int64_t)C.len[i] - ndel + nins;
            int64_t dest = -1;
            int32_t cap = C.cap[i];
            if (L2 > cap) {
                cap = slack_cap(L2, slack_min, slack_div);
                dest = (int64_t)atomicAdd((unsigned long long *)C.top, (unsigned long long)cap);
                if (dest + cap > C.arena_cap) set_status(ctl, ST_C_ARENA);
                atomicAdd((unsigned long long *)&ctl->c_reloc, 1ull);
            }
            M.dest[r] = dest;
            M.dcap[r] = cap;
        }
    }
}

// A warp per run: (moves the row to its new place first, when it has one)
// writes the new values and words in place.  The entries that received no
// product leave holes: the new entries go into holes first, then to the
// row's end, and when there are more holes than new entries, the row's last
// entries move into the holes that remain (C's rows carry no column order).
// So only the run and as many entries at the row's end are touched; the
// compaction of the whole row in order that this replaces took 646 us on
// 1000 edges of R-MAT 17, 25 us now.  The holes' places are listed in
// the run's words ue, which are not needed any more.
template <int SR>
__global__ void k_mask_splice(MaskJob M, MatView C, unsigned long long *F, Ctl *ctl, unsigned mask) {
    pdl_begin();
    using T = typename MSr<SR>::T;
    if (__any_sync(0xffffffffu, failed(ctl, mask))) return;
    const int lane = threadIdx.x & 31;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    T *Cv = (T *)C.val;
    const T *z = (const T *)M.z;
    long long written = 0;
    const long long nr = *M.nruns_dev;
    for (long long r = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nr; r += nwarps) {
        const int64_t u0 = M.run_start[r], u1 = M.run_start[r + 1];
        const int32_t i = M.run_row[r];
        const int L = C.len[i];
        int64_t base = C.off[i];
        const int64_t dest = M.dest[r];
        if (dest >= 0) {
            for (int p = lane; p < L; p += 32) {
                C.col[dest + p] = C.col[base + p];
                Cv[dest + p] = Cv[base + p];
                F[dest + p] = F[base + p];
            }
            base = dest;
            __syncwarp();
        }
        unsigned long long *hole = M.ue + u0;  // the holes' places, in the run's order
        int ndel = 0, nins = 0;
        for (int64_t uc = u0; uc < u1; uc += 32) {
            const int64_t u = uc + lane;
            const int p = u < u1 ? M.upos[u] : -1;
            const bool hit = u < u1 && M.hit[u] != 0;
            const bool del = p >= 0 && !hit;
            if (p >= 0 && hit) {
                Cv[base + p] = z[u];
                F[base + p] = M.h[u];
                written++;
            }
            const unsigned bd = __ballot_sync(0xffffffffu, del);
            if (del) hole[ndel + __popc(bd & lanemask_lt())] = (unsigned long long)p;
            ndel += __popc(bd);
            nins += __popc(__ballot_sync(0xffffffffu, u < u1 && p < 0 && hit));
        }
        __syncwarp();
        const int len = L - ndel + nins;
        if (nins > 0) {
            int m = 0;  // new entries placed
            for (int64_t uc = u0; uc < u1; uc += 32) {
                const int64_t u = uc + lane;
                const bool ins = u < u1 && M.upos[u] < 0 && M.hit[u];
                const unsigned bal = __ballot_sync(0xffffffffu, ins);
                if (ins) {
                    const int x = m + __popc(bal & lanemask_lt());
                    const int d = x < ndel ? (int)hole[x] : L + x - ndel;
                    C.col[base + d] = M.ucol[u];
                    Cv[base + d] = z[u];
                    F[base + d] = M.h[u];
                    written++;
                }
                m += __popc(bal);
            }
        }
        if (ndel > nins) {
            // the remaining holes: marked, and those below the new length
            // listed again (a hole's new place in the list is never above its
            // old one, and each round reads before it writes)
            int nh = 0;
            for (int x0 = nins; x0 < ndel; x0 += 32) {
                const int x = x0 + lane;
                const int p = x < ndel ? (int)hole[x] : INT32_MAX;
                if (x < ndel) C.col[base + p] = -1;
                const bool low = p < len;
                const unsigned bal = __ballot_sync(0xffffffffu, low);
                __syncwarp();
                if (low) hole[nh + __popc(bal & lanemask_lt())] = (unsigned long long)p;
                nh += __popc(bal);
                __syncwarp();
            }
            // the entries past the new length that stay, one into each of them
            int m = 0;
            for (int p0 = len; p0 < L && m < nh; p0 += 32) {
                const int p = p0 + lane;
                const int32_t c = p < L ? C.col[base + p] : -1;
                const unsigned bal = __ballot_sync(0xffffffffu, c >= 0);
                if (c >= 0) {
                    const int d = (int)hole[m + __popc(bal & lanemask_lt())];
                    C.col[base + d] = c;
                    Cv[base + d] = Cv[base + p];
                    F[base + d] = F[base + p];
                }
                m += __popc(bal);
            }
        }
        __syncwarp();
        if (lane == 0) {
            dcheck(ctl, base + len <= C.arena_cap && len <= (dest >= 0 ? M.dcap[r] : C.cap[i]), DBG_MASK_ROOM, i);
            C.len[i] = len;
            if (dest >= 0) {
                C.off[i] = dest;
                C.cap[i] = M.dcap[r];
            }
        }
    }
    written = warp_sum<long long>(written);
    if (lane == 0 && written) atomicAdd((unsigned long long *)&ctl->nnz_written, (unsigned long long)written);
}

template <typename T>
__global__ void k_fill_val(T *p, int64_t n, T v) {
    pdl_begin();
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        p[t] = v;
}

unsigned grid_of(int64_t items, int per_block, int num_sms, int waves = 16) {
    int64_t g = (items + per_block - 1) / per_block;
    if (g > (int64_t)num_sms * waves) g = (int64_t)num_sms * waves;
    if (g < 1) g = 1;
    return (unsigned)g;
}

}  // namespace

void bloom_rows(const MatView &A, const MatView &B, const MatView &C, unsigned long long *F, int32_t *rows_long,
                long long *n_long, long long cap_long, cudaStream_t s, int num_sms) {
    if (C.nrows <= 0) return;
    launch_k(k_bloom_warp, grid_of(C.nrows, BL_NW, num_sms, 8), BL_NW * 32, 0, s, A, B, C, F, rows_long, n_long,
             cap_long);
}

void bloom_long_rows(const MatView &A, const MatView &B, const MatView &C, unsigned long long *F,
                     const int32_t *rows_long, const long long *n_long, long long cap_long, int32_t *posmap,
                     int ctas, cudaStream_t s) {
    launch_k(k_bloom_cta, (unsigned)std::max(ctas, 1), 512, 0, s, A, B, C, F, rows_long, n_long, cap_long, posmap);
}

void pat_contrib(const PatJob &J, const MatView &B, const MatView &AT, Ctl *ctl, unsigned mask, cudaStream_t s,
                 int num_sms) {
    const int64_t warps = std::max(J.xn, J.yn);
    if (warps <= 0) return;
    launch_k(k_pat_contrib, grid_of(warps, 8, num_sms, 8), 256, 0, s, J, B, AT, ctl, mask);
}

void iota_u32(uint32_t *v, int64_t n, cudaStream_t s, int num_sms) {
    if (n <= 0) return;
    launch_k(k_iota, grid_of(n, 256, num_sms), 256, 0, s, v, n);
}

void pat_heads(const uint64_t *K, int64_t n, int32_t *flag, cudaStream_t s, int num_sms) {
    if (n <= 0) return;
    launch_k(k_pat_heads, grid_of(n, 256, num_sms), 256, 0, s, K, n, flag);
}

void pat_unique(const uint64_t *K, const uint32_t *I, const uint64_t *bits, int64_t n, const int64_t *ex, int cb,
                const MaskJob &M, int32_t *rflag, cudaStream_t s, int num_sms) {
    if (n <= 0) return;
    launch_k(k_pat_unique, grid_of(n, 256, num_sms), 256, 0, s, K, I, bits, n, ex, cb, M, rflag);
}

void pat_runs(const MaskJob &M, const int32_t *rflag, const int64_t *rex, int64_t max_u, uint32_t *bm, cudaStream_t s,
              int num_sms) {
    if (max_u <= 0) return;
    launch_k(k_pat_runs, grid_of(max_u, 256, num_sms), 256, 0, s, M, rflag, rex, bm);
}

void mask_scan(const MaskJob &M, const MatView &C, const unsigned long long *F, cudaStream_t s, int num_sms) {
    if (M.max_runs <= 0) return;
    launch_k(k_mask_scan, grid_of(M.max_runs, 8, num_sms), 256, 0, s, M, C, F);
}

void mask_keep(const MaskJob &M, const MatView &A, Ctl *ctl, cudaStream_t s, int num_sms) {
    if (M.max_runs <= 0) return;
    launch_k(k_mask_keep, grid_of(M.max_runs, 8, num_sms), 256, 0, s, M, A, ctl);
}

void mask_product(int sr, const MaskJob &M, const MatView &A, const MatView &B, Ctl *ctl, unsigned mask,
                  cudaStream_t s, int num_sms) {
    if (M.kcap <= 0) return;
    if (sr == SR_PT)
        launch_k(k_mask_product<SR_PT>, grid_of(M.kcap, 8, num_sms), 256, 0, s, M, A, B, ctl, mask);
    else
        launch_k(k_mask_product<SR_MP>, grid_of(M.kcap, 8, num_sms), 256, 0, s, M, A, B, ctl, mask);
}

void mask_init_acc(int sr, const MaskJob &M, int64_t nu, cudaStream_t s, int num_sms) {
    if (nu <= 0) return;
    if (sr == SR_PT) launch_k(k_fill_val<double>, grid_of(nu, 256, num_sms), 256, 0, s, (double *)M.z, nu, 0.0);
    else launch_k(k_fill_val<int32_t>, grid_of(nu, 256, num_sms), 256, 0, s, (int32_t *)M.z, nu, MP_INF);
}

void mask_plan(const MaskJob &M, const MatView &C, Ctl *ctl, unsigned mask, int slack_min, int slack_div,
               cudaStream_t s, int num_sms) {
    if (M.max_runs <= 0) return;
    launch_k(k_mask_plan, grid_of(M.max_runs, 8, num_sms), 256, 0, s, M, C, ctl, mask, slack_min, slack_div);
}

void mask_splice(int sr, const MaskJob &M, const MatView &C, unsigned long long *F, Ctl *ctl, unsigned mask,
                 cudaStream_t s, int num_sms) {
    if (M.max_runs <= 0) return;
    if (sr == SR_PT) launch_k(k_mask_splice<SR_PT>, grid_of(M.max_runs, 8, num_sms), 256, 0, s, M, C, F, ctl, mask);
    else launch_k(k_mask_splice<SR_MP>, grid_of(M.max_runs, 8, num_sms), 256, 0, s, M, C, F, ctl, mask);
}

}  // namespace dspg
