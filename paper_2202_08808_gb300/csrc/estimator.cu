// estimator.cu -- training and evaluation of the learned row-size estimator
// (the network is in estimator.cuh), and the features of rows of C.
//
// Training is plain SGD on the mean squared error between the network's
// output and log2(1 + nnz(C_i)), where nnz(C_i) are exact row sizes that the
// library itself produced (the lengths of the rows of C after a build or a
// batch, which are exact symbolic counts).  One step runs two kernels:
//   k_est_rows  tiles of 32 rows: forward, dL/do, dL/dz2, dL/dz1
//   k_est_step  one thread per parameter: its sum over the rows in order;
//               master <- master - lr * grad and the bfloat16 copy
// Every sum over rows runs in row order in one thread, so a step is
// deterministic.  The forward uses the bfloat16-rounded weights and the
// gradient is taken at them (applied to the float32 master copy).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <string>

#include "estimator.cuh"
#include "internal.h"

using namespace dspg;

namespace {

struct EErr {
    dspg_status st;
    std::string msg;
};

#define ECK(x)                                                                                          \
    do {                                                                                                \
        cudaError_t e_ = (x);                                                                           \
        if (e_ != cudaSuccess) throw EErr{DSPG_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e_)}; \
    } while (0)

template <typename T>
void ealloc(T **p, size_t n) {
    if (cudaMalloc((void **)p, sizeof(T) * (n ? n : 1)) != cudaSuccess) {
        cudaGetLastError();
        throw EErr{DSPG_ERR_OOM, "estimator: device allocation failed"};
    }
}

// Device memory of one call.
struct EBuf {
    float *p = nullptr;
    ~EBuf() {
        if (p) cudaFree(p);
    }
};

constexpr int EST_NT = 128;  // threads of a feature block

// What a training step keeps between its kernels, each a column of `ld` rows
// per unit (so that a sum over rows reads consecutive words): the inputs,
// h1, h2, dL/dz1, dL/dz2 and dL/do.
struct EstCols {
    float *x, *h1, *h2, *dz1, *dz2, *d;
    int64_t ld;  // a multiple of ER_ROWS, at least n
};
constexpr int EST_COLS = EST_IN + 4 * EST_HID + 1;

// A block takes tiles of ER_ROWS rows.  The two 64 x 64 products of a tile
// (z2 = h1 W2', dh1 = dz2 W2) run on the FP32 units out of shared memory, a
// thread for 2 rows x 4 units, so that an operand loaded serves several
// multiply-adds; each output sums its terms in the order of est_forward.
// Bound by the latency of its eight phases: 7 us for 4096 rows, a tile on
// each of 128 SMs.  A thread per row, as before, left 120 of the 152 SMs
// idle on such a batch.
constexpr int ER_NT = 256;
constexpr int ER_ROWS = 32;
constexpr int ER_LD = EST_HID + 4;  // row stride in shared memory: 16-byte rows, fewer bank conflicts down a column
constexpr int ER_W = EST_W2 + EST_HID + EST_HID + 4;  // W1, b1, b2, W3, b3 (and padding)
constexpr int ER_B2 = EST_W2, ER_W3 = ER_B2 + EST_HID, ER_B3 = ER_W3 + EST_HID;  // their places in shared memory
constexpr size_t ER_SMEM =
    (size_t)(ER_W + EST_HID * ER_LD + ER_ROWS * EST_IN + 4 * ER_ROWS * ER_LD + ER_ROWS) * sizeof(float);

// One weight to its place: W2 in rows of ER_LD, the others as they follow.
__device__ __forceinline__ void place_weight(float *W, float *W2, int k, float v) {
    if (k < EST_W2) W[k] = v;
    else if (k < EST_B2) W2[(k - EST_W2) / EST_HID * ER_LD + (k - EST_W2) % EST_HID] = v;
    else W[k - EST_HID * EST_HID] = v;
}

// col[j * ld + row] for the tile's rows, from t[row * ER_LD + j]
__device__ __forceinline__ void store_columns(float *col, int64_t ld, int64_t base, const float *t) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int j = w; j < EST_HID; j += ER_NT / 32) col[j * ld + base + lane] = t[lane * ER_LD + j];
}

template <bool GRAD>
__global__ void __launch_bounds__(ER_NT)
k_est_rows(const uint16_t *w, const float *X, const float *y, int64_t n, float *O, EstCols C, double *lpart) {
    pdl_begin();
    extern __shared__ __align__(16) float sm[];
    float *W = sm;                        // W1, b1, b2, W3, b3
    float *W2 = W + ER_W;                 // rows of ER_LD
    float *x = W2 + EST_HID * ER_LD;      // the tile's inputs
    float *h1 = x + ER_ROWS * EST_IN, *h2 = h1 + ER_ROWS * ER_LD;
    float *dz1 = h2 + ER_ROWS * ER_LD, *dz2 = dz1 + ER_ROWS * ER_LD;
    float *d = dz2 + ER_ROWS * ER_LD;     // dL/do
    const int tid = threadIdx.x;
    int64_t base = (int64_t)blockIdx.x * ER_ROWS;  // the grid has no more blocks than tiles
    // the first tile's inputs are fetched beside the weights, the next ones' beside a tile's work
    auto input = [&](int64_t b) { return tid < ER_ROWS * EST_IN && b * EST_IN + tid < n * EST_IN ? X[b * EST_IN + tid] : 0.0f; };
    float xv = input(base);
#pragma unroll
    for (int q = tid; q < EST_PARAMS / 8; q += ER_NT) {
        const uint4 v = *((const uint4 *)w + q);
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            place_weight(W, W2, q * 8 + 2 * i, bf16_bits_to_float((uint16_t)(u[i] & 0xffffu)));
            place_weight(W, W2, q * 8 + 2 * i + 1, bf16_bits_to_float((uint16_t)(u[i] >> 16)));
        }
    }
    if (tid < EST_PARAMS % 8) {
        const int k = EST_PARAMS / 8 * 8 + tid;
        place_weight(W, W2, k, bf16_bits_to_float(w[k]));
    }
    // this thread's 2 rows of a tile, and its 4 units: jq, jq + 16, ... of z2 (so that the rows of W2 that a
    // quarter-warp reads lie in different banks), 4 jq, ... of dh1
    const int r0 = (tid >> 4) * 2, jq = tid & 15, q1 = jq * 4;
    double loss = 0.0;
    for (; base < n; base += (int64_t)gridDim.x * ER_ROWS) {
        const int nr = (int)(n - base < ER_ROWS ? n - base : ER_ROWS);
        const float yv = y && tid < nr ? y[base + tid] : 0.0f;
        if (tid < ER_ROWS * EST_IN) x[tid] = xv;
        xv = input(base + (int64_t)gridDim.x * ER_ROWS);
        __syncthreads();
        {
            const int j = tid & 63;
            float wj[EST_IN];
#pragma unroll
            for (int c = 0; c < EST_IN; c++) wj[c] = W[EST_W1 + j * EST_IN + c];
            const float bj = W[EST_B1 + j];
#pragma unroll
            for (int q = 0; q < ER_ROWS / 4; q++) {
                const int r = (tid >> 6) * (ER_ROWS / 4) + q;
                float z = bj;
#pragma unroll
                for (int c = 0; c < EST_IN; c++) z = fmaf(wj[c], x[r * EST_IN + c], z);
                h1[r * ER_LD + j] = fmaxf(z, 0.0f);
            }
        }
        __syncthreads();
        {
            float z[2][4];
#pragma unroll
            for (int i = 0; i < 4; i++) z[0][i] = z[1][i] = W[ER_B2 + jq + 16 * i];
#pragma unroll 4
            for (int k = 0; k < EST_HID; k += 4) {
                const float4 a = *(const float4 *)(h1 + r0 * ER_LD + k), b = *(const float4 *)(h1 + (r0 + 1) * ER_LD + k);
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float4 v = *(const float4 *)(W2 + (jq + 16 * i) * ER_LD + k);
                    z[0][i] = fmaf(v.x, a.x, z[0][i]);
                    z[1][i] = fmaf(v.x, b.x, z[1][i]);
                    z[0][i] = fmaf(v.y, a.y, z[0][i]);
                    z[1][i] = fmaf(v.y, b.y, z[1][i]);
                    z[0][i] = fmaf(v.z, a.z, z[0][i]);
                    z[1][i] = fmaf(v.z, b.z, z[1][i]);
                    z[0][i] = fmaf(v.w, a.w, z[0][i]);
                    z[1][i] = fmaf(v.w, b.w, z[1][i]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                h2[r0 * ER_LD + jq + 16 * i] = fmaxf(z[0][i], 0.f);
                h2[(r0 + 1) * ER_LD + jq + 16 * i] = fmaxf(z[1][i], 0.f);
            }
        }
        __syncthreads();
        if (tid < ER_ROWS) {
            float o = W[ER_B3];
#pragma unroll 4
            for (int j = 0; j < EST_HID; j += 4) {
                const float4 v = *(const float4 *)(W + ER_W3 + j), h = *(const float4 *)(h2 + tid * ER_LD + j);
                o = fmaf(v.x, h.x, o);
                o = fmaf(v.y, h.y, o);
                o = fmaf(v.z, h.z, o);
                o = fmaf(v.w, h.w, o);
            }
            float dd = 0.0f;
            if (tid < nr) {
                if (O) O[base + tid] = o;
                if (y) {
                    const float e = o - yv;
                    dd = 2.0f * e / (float)n;
                    loss += (double)e * (double)e;
                }
            }
            d[tid] = dd;
            if (GRAD) C.d[base + tid] = dd;
        } else if (GRAD) {  // the other warps' share of the columns meanwhile
            const int lane = tid & 31, wp = tid >> 5;
            for (int j = wp - 1; j < EST_HID; j += ER_NT / 32 - 1) {
                C.h1[j * C.ld + base + lane] = h1[lane * ER_LD + j];
                C.h2[j * C.ld + base + lane] = h2[lane * ER_LD + j];
            }
            if (wp == 1)
#pragma unroll
                for (int c = 0; c < EST_IN; c++) C.x[c * C.ld + base + lane] = x[lane * EST_IN + c];
        }
        if (GRAD) {
            __syncthreads();
            const float4 w3 = *(const float4 *)(W + ER_W3 + q1);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const float4 h = *(const float4 *)(h2 + (r0 + q) * ER_LD + q1);
                const float e = d[r0 + q];
                *(float4 *)(dz2 + (r0 + q) * ER_LD + q1) =
                    make_float4(h.x > 0.f ? e * w3.x : 0.f, h.y > 0.f ? e * w3.y : 0.f, h.z > 0.f ? e * w3.z : 0.f,
                                h.w > 0.f ? e * w3.w : 0.f);
            }
            __syncthreads();
            store_columns(C.dz2, C.ld, base, dz2);
            float4 ga = make_float4(0.f, 0.f, 0.f, 0.f), gb = ga;
#pragma unroll 4
            for (int j = 0; j < EST_HID; j += 4) {
                const float4 a4 = *(const float4 *)(dz2 + r0 * ER_LD + j), b4 = *(const float4 *)(dz2 + (r0 + 1) * ER_LD + j);
                const float as[4] = {a4.x, a4.y, a4.z, a4.w}, bs[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float4 v = *(const float4 *)(W2 + (j + i) * ER_LD + q1);
                    ga.x = fmaf(as[i], v.x, ga.x);
                    ga.y = fmaf(as[i], v.y, ga.y);
                    ga.z = fmaf(as[i], v.z, ga.z);
                    ga.w = fmaf(as[i], v.w, ga.w);
                    gb.x = fmaf(bs[i], v.x, gb.x);
                    gb.y = fmaf(bs[i], v.y, gb.y);
                    gb.z = fmaf(bs[i], v.z, gb.z);
                    gb.w = fmaf(bs[i], v.w, gb.w);
                }
            }
            const float4 ha = *(const float4 *)(h1 + r0 * ER_LD + q1), hb = *(const float4 *)(h1 + (r0 + 1) * ER_LD + q1);
            *(float4 *)(dz1 + r0 * ER_LD + q1) = make_float4(ha.x > 0.f ? ga.x : 0.f, ha.y > 0.f ? ga.y : 0.f,
                                                             ha.z > 0.f ? ga.z : 0.f, ha.w > 0.f ? ga.w : 0.f);
            *(float4 *)(dz1 + (r0 + 1) * ER_LD + q1) = make_float4(hb.x > 0.f ? gb.x : 0.f, hb.y > 0.f ? gb.y : 0.f,
                                                                   hb.z > 0.f ? gb.z : 0.f, hb.w > 0.f ? gb.w : 0.f);
            __syncthreads();
            store_columns(C.dz1, C.ld, base, dz1);
        }
        __syncthreads();  // the tile's arrays are read before the next one fills them
    }
    if (y && tid < 32) {
        loss = warp_sum<double>(loss);
        if (tid == 0) lpart[blockIdx.x] = loss;
    }
}
static_assert(ER_ROWS == 32 && ER_ROWS / 2 * EST_HID / 4 == ER_NT, "k_est_rows' thread layout");

// One thread per parameter sums its term over the rows in order:
//   W2[j][k] = sum_r dz2[r][j] h1[r][k]   b2[j] = sum_r dz2[r][j]
//   W1[j][c] = sum_r dz1[r][j] x[r][c]    b1[j] = sum_r dz1[r][j]
//   W3[j]    = sum_r d[r] h2[r][j]        b3    = sum_r d[r]
// A block has the parameters of at most 12 columns (4 of dz2 by 8 of h1, 8
// of dz1 by the inputs, 8 of h2 by d) and streams those columns through
// shared memory, ES_ST stages of ES_R rows by asynchronous copies of its
// warps 2 and 3; 144 blocks keep every SM but a few busy.  What bounds it is the chain of one
// multiply-add after the other: 4.3 cycles a row out of registers, 4.4 out of
// shared memory with the stage's loop unrolled, 6.2 with two rounds of it (a
// warp alone).  The loads of a thread per parameter straight from row-major
// arrays made it 13 times as long (32 steps of 4096 rows and the loss of
// 32768: 7.7 ms, 0.84 ms with the loop not unrolled, 0.73 now).  Stages of
// 128 or 512 rows (0.79 and 0.85 ms) and 6 of them (0.87) are slower.  With lr > 0 the
// parameter's owner then makes the step and its bfloat16 copy.
constexpr int ES_NT = 128;
constexpr int ES_R = 256;
constexpr int ES_LD = ES_R + 4;   // 16-byte reads of 8 columns side by side meet no bank twice
constexpr int ES_ST = 4;
constexpr int ES_MAXC = 12;
constexpr size_t ES_SMEM = (size_t)(ES_ST * ES_MAXC + 1) * ES_LD * sizeof(float);
constexpr int ES_W2B = (EST_HID / 4) * (EST_HID / 8), ES_W1B = EST_HID / 8, ES_W3B = EST_HID / 8;

__global__ void __launch_bounds__(ES_NT)
k_est_step(EstCols C, int64_t n, float lr, float *grad, float *master, uint16_t *w) {
    pdl_begin();
    extern __shared__ __align__(16) float sm[];
    const int tid = threadIdx.x, b = blockIdx.x;
    // the block's columns: na of `ca`, then nb of `cb`; this thread's
    // parameter p (-1: none) and its columns ia and ib (ib < 0: a column of
    // ones, which makes the multiply-add the plain sum)
    const float *ca, *cb;
    int na, nb, p = -1, ia = 0, ib = -1;
    if (b < ES_W2B) {
        const int j = (b / (EST_HID / 8)) * 4, k = (b % (EST_HID / 8)) * 8;
        ca = C.dz2 + j * C.ld;
        cb = C.h1 + k * C.ld;
        na = 4;
        nb = 8;
        if (tid < 32) {
            ia = tid >> 3;
            ib = 4 + (tid & 7);
            p = EST_W2 + (j + ia) * EST_HID + k + (tid & 7);
        } else if (k == 0 && tid < 36) {
            ia = tid - 32;
            p = EST_B2 + j + ia;
        }
    } else if (b < ES_W2B + ES_W1B) {
        const int j = (b - ES_W2B) * 8;
        ca = C.dz1 + j * C.ld;
        cb = C.x;
        na = 8;
        nb = EST_IN;
        if (tid < 32) {
            ia = tid >> 2;
            ib = 8 + (tid & 3);
            p = EST_W1 + (j + ia) * EST_IN + (tid & 3);
        } else if (tid < 40) {
            ia = tid - 32;
            p = EST_B1 + j + ia;
        }
    } else {
        const int j = (b - ES_W2B - ES_W1B) * 8;
        ca = C.h2 + j * C.ld;
        cb = C.d;
        na = 8;
        nb = 1;
        if (tid < 8) {
            ia = tid;
            ib = 8;
            p = EST_W3 + j + tid;
        } else if (j == 0 && tid == 32) {
            ia = 8;
            p = EST_B3;
        }
    }
    float *ones = sm + ES_ST * ES_MAXC * ES_LD;
    for (int r = tid; r < ES_LD; r += ES_NT) ones[r] = 1.0f;
    const int64_t stages = (n + ES_R - 1) / ES_R;
    auto fetch = [&](int64_t s) {  // stage s into its slot; whole tiles of ER_ROWS rows exist past n
        if (s < stages && tid >= ES_NT / 2) {
            const int64_t r0 = s * ES_R;
            const int rows = (int)(C.ld - r0 < ES_R ? C.ld - r0 : ES_R);
            float *dst = sm + (s % ES_ST) * ES_MAXC * ES_LD;
            for (int q = tid - ES_NT / 2; q < (na + nb) * (ES_R / 4); q += ES_NT / 2) {
                const int c = q / (ES_R / 4), r = (q % (ES_R / 4)) * 4;
                const float *src = (c < na ? ca + c * C.ld : cb + (c - na) * C.ld) + r0 + r;
                if (r < rows) {
                    const unsigned to = (unsigned)__cvta_generic_to_shared(dst + c * ES_LD + r);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(to), "l"(src) : "memory");
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    for (int s = 0; s < ES_ST - 1; s++) fetch(s);
    float g = 0.0f;
    for (int64_t s = 0; s < stages; s++) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(ES_ST - 2) : "memory");
        __syncthreads();  // stage s is here, and every thread has left the slot that the next fetch fills
        fetch(s + ES_ST - 1);
        if (p >= 0) {
            const float *A = sm + (s % ES_ST) * ES_MAXC * ES_LD + ia * ES_LD;
            const float *B = ib < 0 ? ones : sm + (s % ES_ST) * ES_MAXC * ES_LD + ib * ES_LD;
            const int rows = (int)(n - s * ES_R < ES_R ? n - s * ES_R : ES_R);
            int r = 0;
            // 16 rows at a time, the next 16 loaded meanwhile (64 cycles of the chain); unrolled over the whole
            // stage, as the copies of the loaded words and the loop's own instructions took a third of the chain
            if (rows == ES_R) {
                float4 a[4], q[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    a[i] = *(const float4 *)(A + 4 * i);
                    q[i] = *(const float4 *)(B + 4 * i);
                }
#pragma unroll
                for (; r < ES_R; r += 16) {
                    float4 a2[4], q2[4];
                    const int nx = r + 16 < ES_R ? r + 16 : 0;
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        a2[i] = *(const float4 *)(A + nx + 4 * i);
                        q2[i] = *(const float4 *)(B + nx + 4 * i);
                    }
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        g = fmaf(a[i].x, q[i].x, g);
                        g = fmaf(a[i].y, q[i].y, g);
                        g = fmaf(a[i].z, q[i].z, g);
                        g = fmaf(a[i].w, q[i].w, g);
                        a[i] = a2[i];
                        q[i] = q2[i];
                    }
                }
            }
            for (; r < rows; r++) g = fmaf(A[r], B[r], g);
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    if (p >= 0) {
        grad[p] = g;
        if (lr > 0.0f) {
            const float v = master[p] - lr * g;
            master[p] = v;
            w[p] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
        }
    }
}

__global__ void k_est_loss(const double *lpart, int np, int64_t n, double *loss) {
    pdl_begin();
    double s = 0.0;
    for (int b = threadIdx.x; b < np; b += 32) s += lpart[b];
    s = warp_sum<double>(s);
    if (threadIdx.x == 0) *loss = s / (double)n;
}

__global__ void k_est_round(const float *master, uint16_t *w) {
    pdl_begin();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < EST_PARAMS) w[p] = __bfloat16_as_ushort(__float2bfloat16_rn(master[p]));
}

// Features of rows (all rows when rows == nullptr) and, when y != nullptr,
// the target log2(1 + len(C_i)).  A row index out of range sets *bad and
// gets zeros.
__global__ void k_row_features(MatView A, MatView B, MatView C, const int32_t *rows, int64_t n, float *X, float *y,
                               unsigned *bad) {
    pdl_begin();
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = rows ? rows[t] : (int32_t)t;
        if (i < 0 || i >= A.nrows) {
            atomicOr(bad, 1u);
            for (int c = 0; c < EST_IN; c++) X[t * EST_IN + c] = 0.0f;
            if (y) y[t] = 0.0f;
            continue;
        }
        const int64_t off = A.off[i];
        const int alen = A.len[i];
        long long sum = 0, mx = 0;
        for (int a = 0; a < alen; a++) {
            const long long l = B.len[A.col[off + a]];
            sum += l;
            mx = l > mx ? l : mx;
        }
        float x[EST_IN];
        est_features(x, alen, sum, mx);
        for (int c = 0; c < EST_IN; c++) X[t * EST_IN + c] = x[c];
        if (y) y[t] = log2f(1.0f + (float)C.len[i]);
    }
}

unsigned grid_rows(int64_t n) {
    int64_t g = (n + EST_NT - 1) / EST_NT;
    if (g > 4096) g = 4096;
    return (unsigned)(g < 1 ? 1 : g);
}

// Blocks of k_est_rows at most: two to an SM (their shared memory).
int most_blocks() {
    static int most = 0;
    if (!most) {
        int dev = 0, sms = 0;
        ECK(cudaGetDevice(&dev));
        ECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        ECK(cudaFuncSetAttribute(k_est_rows<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ER_SMEM));
        ECK(cudaFuncSetAttribute(k_est_rows<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ER_SMEM));
        ECK(cudaFuncSetAttribute(k_est_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ES_SMEM));
        most = 2 * sms;
    }
    return most;
}

// Room for the columns of n rows.
EstCols columns(dspg_estimator *e, int64_t n) {
    const int64_t ld = (n + ER_ROWS - 1) / ER_ROWS * ER_ROWS;
    if (ld > e->cap) {
        if (e->cols) cudaFree(e->cols);
        e->cols = nullptr;
        e->cap = 0;
        const int64_t cap = ld + ld / 2;
        ealloc(&e->cols, (size_t)cap * EST_COLS);
        e->cap = cap;
    }
    EstCols C;
    C.ld = ld;
    C.x = e->cols;
    C.h1 = C.x + EST_IN * ld;
    C.h2 = C.h1 + EST_HID * ld;
    C.dz1 = C.h2 + EST_HID * ld;
    C.dz2 = C.dz1 + EST_HID * ld;
    C.d = C.dz2 + EST_HID * ld;
    return C;
}

// forward (outputs to O when given, loss when y and loss) and, with grad, the
// gradient and, with lr > 0, the step of the weights
void run_rows(dspg_estimator *e, const float *X, const float *y, int64_t n, float *O, bool grad, float lr, bool loss,
              cudaStream_t s) {
    const int most = most_blocks();
    if (!e->lpart) ealloc(&e->lpart, (size_t)most);
    const EstCols C = grad ? columns(e, n) : EstCols{};
    const int g = (int)std::min<int64_t>((n + ER_ROWS - 1) / ER_ROWS, most);
    launch_k(grad ? k_est_rows<true> : k_est_rows<false>, g, ER_NT, ER_SMEM, s, (const uint16_t *)e->w, X, y, n, O, C,
             e->lpart);
    if (grad) launch_k(k_est_step, ES_W2B + ES_W1B + ES_W3B, ES_NT, ES_SMEM, s, C, n, lr, e->grad, e->master, e->w);
    if (loss) launch_k(k_est_loss, 1, 32, 0, s, (const double *)e->lpart, g, n, e->loss_d);
}

dspg_status efail(dspg_estimator *e, const EErr &x) {
    if (e) e->err = x.msg;
    dspg::set_thread_error(x.msg.c_str());
    return x.st;
}

void check_rows(const float *X, int64_t n) {
    if (n <= 0 || !X) throw EErr{DSPG_ERR_INVALID, "estimator: need n > 0 rows and X"};
}

}  // namespace

void dspg::row_features(const MatView &A, const MatView &B, const MatView &C, const int32_t *rows, int64_t n, float *X,
                        float *y, unsigned *bad, cudaStream_t s) {
    if (n > 0) launch_k(k_row_features, grid_rows(n), EST_NT, 0, s, A, B, C, rows, n, X, y, bad);
}

extern "C" {

dspg_status dspg_estimator_create(dspg_estimator **out, const float *params) {
    dspg_estimator *e = nullptr;
    try {
        if (!out || !params) throw EErr{DSPG_ERR_INVALID, "estimator: out and params must not be NULL"};
        *out = nullptr;
        e = new dspg_estimator();
        ealloc(&e->master, EST_PARAMS);
        ealloc(&e->grad, EST_PARAMS);
        ealloc(&e->w, EST_PARAMS);
        ealloc(&e->loss_d, 1);
        ECK(cudaMemcpy(e->master, params, sizeof(float) * EST_PARAMS, cudaMemcpyHostToDevice));
        ECK(cudaMemset(e->grad, 0, sizeof(float) * EST_PARAMS));
        launch_k(k_est_round, (EST_PARAMS + 127) / 128, 128, 0, (cudaStream_t)0, (const float *)e->master, e->w);
        ECK(cudaGetLastError());
        ECK(cudaDeviceSynchronize());
        *out = e;
        return DSPG_OK;
    } catch (const EErr &x) {
        dspg_status st = efail(nullptr, x);
        dspg_estimator_destroy(e);
        return st;
    }
}

dspg_status dspg_estimator_params(dspg_estimator *e, float *params, void *stream) {
    if (!e || !params) return DSPG_ERR_INVALID;
    try {
        cudaStream_t s = (cudaStream_t)stream;
        ECK(cudaMemcpyAsync(params, e->master, sizeof(float) * EST_PARAMS, cudaMemcpyDeviceToHost, s));
        ECK(cudaStreamSynchronize(s));
        return DSPG_OK;
    } catch (const EErr &x) {
        return efail(e, x);
    }
}

dspg_status dspg_estimator_grad(dspg_estimator *e, const float *X, const float *y, int64_t n, float *grad,
                                double *loss, void *stream) {
    if (!e) return DSPG_ERR_INVALID;
    try {
        check_rows(X, n);
        if (!y) throw EErr{DSPG_ERR_INVALID, "estimator: y is NULL"};
        cudaStream_t s = (cudaStream_t)stream;
        run_rows(e, X, y, n, nullptr, true, 0.0f, true, s);
        if (grad) ECK(cudaMemcpyAsync(grad, e->grad, sizeof(float) * EST_PARAMS, cudaMemcpyDeviceToHost, s));
        if (loss) ECK(cudaMemcpyAsync(loss, e->loss_d, sizeof(double), cudaMemcpyDeviceToHost, s));
        ECK(cudaStreamSynchronize(s));
        return DSPG_OK;
    } catch (const EErr &x) {
        return efail(e, x);
    }
}

dspg_status dspg_estimator_train(dspg_estimator *e, const float *X, const float *y, int64_t n, int64_t batch,
                                 int64_t steps, float lr, double *loss, void *stream) {
    if (!e) return DSPG_ERR_INVALID;
    try {
        check_rows(X, n);
        if (!y || batch <= 0 || steps < 0 || !(lr > 0.0f)) throw EErr{DSPG_ERR_INVALID, "estimator: bad training arguments"};
        cudaStream_t s = (cudaStream_t)stream;
        const int64_t nb = (n + batch - 1) / batch;
        for (int64_t k = 0; k < steps; k++) {
            const int64_t b = k % nb;
            const int64_t lo = b * batch, m = (lo + batch <= n) ? batch : n - lo;
            run_rows(e, X + lo * EST_IN, y + lo, m, nullptr, true, lr, false, s);
        }
        ECK(cudaGetLastError());
        if (loss) {  // loss of the whole set after training
            run_rows(e, X, y, n, nullptr, false, 0.0f, true, s);
            ECK(cudaMemcpyAsync(loss, e->loss_d, sizeof(double), cudaMemcpyDeviceToHost, s));
        }
        ECK(cudaStreamSynchronize(s));
        return DSPG_OK;
    } catch (const EErr &x) {
        return efail(e, x);
    }
}

dspg_status dspg_estimator_predict(dspg_estimator *e, const float *X, int64_t n, float *out, void *stream) {
    if (!e || !out) return DSPG_ERR_INVALID;
    try {
        check_rows(X, n);
        cudaStream_t s = (cudaStream_t)stream;
        // outputs over the inputs: a block stores its tile's while others have
        // theirs to read, so they go through memory of their own
        const uintptr_t x0 = (uintptr_t)X, o0 = (uintptr_t)out;
        const bool over = o0 < x0 + sizeof(float) * EST_IN * n && x0 < o0 + sizeof(float) * n;
        EBuf o;
        if (over) ealloc(&o.p, (size_t)n);
        run_rows(e, X, nullptr, n, over ? o.p : out, false, 0.0f, false, s);
        if (over) ECK(cudaMemcpyAsync(out, o.p, sizeof(float) * n, cudaMemcpyDeviceToDevice, s));
        ECK(cudaGetLastError());
        ECK(cudaStreamSynchronize(s));
        return DSPG_OK;
    } catch (const EErr &x) {
        return efail(e, x);
    }
}

const char *dspg_estimator_last_error(const dspg_estimator *e) { return e ? e->err.c_str() : dspg_last_error(nullptr); }

void dspg_estimator_destroy(dspg_estimator *e) {
    if (!e) return;
    cudaDeviceSynchronize();
    for (float *p : {e->master, e->grad, e->cols})
        if (p) cudaFree(p);
    if (e->lpart) cudaFree(e->lpart);
    if (e->w) cudaFree(e->w);
    if (e->loss_d) cudaFree(e->loss_d);
    delete e;
}

}  // extern "C"
