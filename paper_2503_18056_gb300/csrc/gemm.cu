// FP64 contractions of the Gram-SVD rounding (App. A.2 of arXiv 2503.18056) on
// the FP64 tensor pipe (mma.sync m8n8k4.f64): the products below the sizes at
// which digits.cu takes over, and whatever it cannot split.
//
// GB300's FP64 pipe issues one warp instruction in 64 clocks per SM
// sub-partition (19 per SM; a DMMA of 256 FMAs takes eight times that), so a
// product's time is the longest chain of DMMAs that a sub-partition is given,
// and loads hardly matter: a 16 x 16 tile's step of 16 indices is 2,048 clocks
// of each of its four warps against four loads a lane from L2.  So the work
// is cut as finely as possible and nothing is staged in shared memory: a CTA
// owns a 16 x 16 tile and a range of the contraction, its four warps take
// every fourth group of four indices, and the contraction is split over CTAs
// (prod_split) until the 608 sub-partitions share the DMMAs evenly.  The CTA
// that arrives last at a tile adds the splits' partials in split order
// (reproducible), so a split product is one launch.
//
// Measured (GB300, us a library call, 64 x 64 tiles staged in shared memory
// before): 133 x 97 x 389 474 -> 27; Gram of 1024 x 61 300 -> 26 (most of both
// the host's call); the small-grid 2D step 8.5 -> 6.1 ms, the 16-problem
// captured batch 26.3 -> 21.1 ms.
#include <algorithm>
#include <atomic>

#include "internal.h"

namespace ttsn {

namespace {

constexpr int BT = 16;       // output tile edge
constexpr int BK = 16;       // contraction indices of a CTA's step (four warps x four)
constexpr int THREADS = 128;

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile(
        "mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
        : "+d"(c[0]), "+d"(c[1])
        : "d"(a), "d"(b));
}

__host__ __device__ inline int floor_log2(long x) {
    int b = 0;
    while (x > 1) {
        x >>= 1;
        ++b;
    }
    return b;
}
__host__ __device__ inline long prod_tiles(long M, long N, int tri) {
    const long tm = (M + BT - 1) / BT, tn = (N + BT - 1) / BT;
    return tri ? tm * (tm + 1) / 2 : tm * tn;
}
__host__ __device__ inline int prod_chunk(long K, int ks) {
    const long c = (K + ks - 1) / ks;
    return (int)((c + BK - 1) / BK * BK);
}
// Time of a product at ks splits in units of 128 clocks: the waves of one CTA
// per SM (four warps fill its four sub-partitions) times a CTA's steps (16
// units each) and its start and in-CTA sum (8), then the last arrival's sum
// (two DADDs a thread and split).
__host__ __device__ inline unsigned prod_cost(long tiles, long K, int ks) {
    const long steps = prod_chunk(K, ks) / BK;
    const long waves = (tiles * ks + 151) / 152;
    const long c = waves * (16 * steps + 8) + (ks > 1 ? ks + 12 : 0);
    return c > 0x03ffffffL ? 0x03ffffffu : (unsigned)c;
}
constexpr int MAX_SPLIT = 64;
__host__ __device__ inline int prod_limit(long tiles, long K) {
    long k = K / BK;
    if (k > SPLIT_ITEMS / tiles) k = SPLIT_ITEMS / tiles;
    if (k > MAX_SPLIT) k = MAX_SPLIT;
    return k < 1 ? 1 : (int)k;
}

}  // namespace

// Autotuned splits (tt_autotune): for a product of t < 152 output tiles of 64
// x 64 (bucket floor(log2 t)) and depth K (bucket floor(log2 K)), the split
// of K that measured fastest on this GPU; 0 keeps the cost rule.  One copy
// for the host and one in device memory, installed together, so a captured
// step decides as the host path does.
__device__ int d_sk_table[AT_TILE_BUCKETS * AT_K_BUCKETS];
static int h_sk_table[AT_TILE_BUCKETS * AT_K_BUCKETS];

namespace {

__host__ __device__ inline int prod_tuned(long M, long N, long K, int tri) {
    const long t64 = ((M + 63) / 64) * ((N + 63) / 64);
    if (tri || t64 >= 152) return 0;
    const int tb = floor_log2(t64), kb = floor_log2(K);
    if (tb >= AT_TILE_BUCKETS || kb >= AT_K_BUCKETS) return 0;
#ifdef __CUDA_ARCH__
    return d_sk_table[tb * AT_K_BUCKETS + kb];
#else
    return h_sk_table[tb * AT_K_BUCKETS + kb];
#endif
}
__host__ __device__ inline int prod_final(long K, int ks) {  // splits that hold indices
    const int c = prod_chunk(K, ks);
    return (int)((K + c - 1) / c);
}
int prod_split(long M, long N, long K, int tri) {
    const long tiles = prod_tiles(M, N, tri);
    const int lim = prod_limit(tiles, K), tuned = prod_tuned(M, N, K, tri);
    if (tuned > 0) return prod_final(K, std::min(tuned, lim));
    int best = 1;
    for (int k = 2; k <= lim; ++k)
        if (prod_cost(tiles, K, k) < prod_cost(tiles, K, best)) best = k;
    return prod_final(K, best);
}
// the same choice by one warp (a captured step's sizes are the device's)
__device__ __forceinline__ int prod_split_warp(long M, long N, long K, int tri) {
    const long tiles = prod_tiles(M, N, tri);
    const int lim = prod_limit(tiles, K), tuned = prod_tuned(M, N, K, tri);
    if (tuned > 0) return prod_final(K, min(tuned, lim));
    unsigned key = 0xffffffffu;
    for (int k = (threadIdx.x & 31) + 1; k <= lim; k += 32)
        key = min(key, prod_cost(tiles, K, k) * 64u + (unsigned)(k - 1));
    return prod_final(K, (int)(__reduce_min_sync(0xffffffffu, key) & 63u) + 1);
}

// C = alpha op(A) op(B) (+ beta C), or with tri the symmetric product of which
// only the tiles on and above the diagonal are formed (both halves stored).
// desc (a captured step): M, N, K, lda, ldb, ldc in device memory; tc: sizes
// that digits.cu takes are left to it.  An item is (tile, split); ks > 1:
// partials to P (256 doubles an item), arrivals counted in cnt (zero between
// products: the last arrival resets its tile's).  An 8 x 8 product outside
// M x N or below the diagonal is skipped.
template <bool TA, bool TB>
__global__ void __launch_bounds__(THREADS)
prod_kernel(int M, int N, int K, double alpha, const double* __restrict__ A, long lda, const double* __restrict__ B,
            long ldb, double beta, double* __restrict__ C, long ldc, int ks, double* __restrict__ P, int* cnt, int tri,
            const int* __restrict__ desc, int tc) {
    if (desc) {
        M = desc[0];
        N = desc[1];
        K = desc[2];
        lda = desc[3];
        ldb = desc[4];
        ldc = desc[5];
        if (M <= 0 || N <= 0 || (tc && tc8_wanted(M, N, K))) return;
        ks = prod_split_warp(M, N, K, tri);
    }
    __shared__ double red[4][BT * BT];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int TM = (M + BT - 1) / BT, TN = (N + BT - 1) / BT;
    const int chunk = prod_chunk(K, ks);
    const long items = prod_tiles(M, N, tri) * ks;
    for (long item = blockIdx.x; item < items; item += gridDim.x) {
        const long tile = item / ks;
        const int z = (int)(item % ks);
        int tm, tn;
        if (tri) {
            tm = 0;
            long t = tile;
            while (t >= TM - tm) {  // row tm of the upper triangle holds TM - tm tiles
                t -= TM - tm;
                ++tm;
            }
            tn = tm + (int)t;
        } else {
            tm = (int)(tile / TN);
            tn = (int)(tile % TN);
        }
        const int m0 = tm * BT, n0 = tn * BT;
        const int kbeg = z * chunk, kend = min(K, kbeg + chunk);
        const bool l1 = m0 + 8 < M, c1 = n0 + 8 < N;
        const bool use10 = l1 && !(tri && tm == tn), use11 = l1 && c1;
        double acc[2][2][2] = {};
        // lane: row lane / 4 and index lane % 4 of the operands (rows past the
        // last read the last: their outputs are not stored)
        const int r0 = min(m0 + (lane >> 2), M - 1), r1 = min(m0 + 8 + (lane >> 2), M - 1);
        const int q0 = min(n0 + (lane >> 2), N - 1), q1 = min(n0 + 8 + (lane >> 2), N - 1);
        const double* a0 = TA ? A + r0 : A + (long)r0 * lda;
        const double* a1 = TA ? A + r1 : A + (long)r1 * lda;
        const double* b0 = TB ? B + (long)q0 * ldb : B + q0;
        const double* b1 = TB ? B + (long)q1 * ldb : B + q1;
        const long sa = TA ? lda : 1, sb = TB ? 1 : ldb;
        double x0 = 0.0, x1 = 0.0, y0 = 0.0, y1 = 0.0;
        auto load = [&](int k) {
            const int kk = k + (lane & 3);
            const bool in = kk < kend;
            x0 = in ? a0[kk * sa] : 0.0;
            x1 = in && l1 ? a1[kk * sa] : 0.0;
            y0 = in ? b0[kk * sb] : 0.0;
            y1 = in && c1 ? b1[kk * sb] : 0.0;
        };
        int k = kbeg + 4 * warp;
        if (k < kend) load(k);
        for (; k < kend; k += BK) {
            const double u0 = x0, u1 = x1, v0 = y0, v1 = y1;
            if (k + BK < kend) load(k + BK);
            dmma(acc[0][0], u0, v0);
            if (c1) dmma(acc[0][1], u0, v1);
            if (use10) dmma(acc[1][0], u1, v0);
            if (use11) dmma(acc[1][1], u1, v1);
        }
        __syncthreads();  // the item before has read red
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                *reinterpret_cast<double2*>(&red[warp][(8 * i + (lane >> 2)) * BT + 8 * j + (lane & 3) * 2]) =
                    make_double2(acc[i][j][0], acc[i][j][1]);
        __syncthreads();
        double v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + h * THREADS;
            v[h] = (red[0][e] + red[1][e]) + (red[2][e] + red[3][e]);
        }
        if (ks > 1) {
            double* pt = P + tile * ks * (BT * BT);
            __stcg(pt + (long)z * (BT * BT) + tid, v[0]);
            __stcg(pt + (long)z * (BT * BT) + tid + THREADS, v[1]);
            __threadfence();
            __syncthreads();
            if (tid == 0) s_last = atomicAdd(cnt + tile, 1) == ks - 1;
            __syncthreads();
            if (!s_last) continue;
            __threadfence();
            v[0] = v[1] = 0.0;
#pragma unroll 4
            for (int y = 0; y < ks; ++y) {
                v[0] += __ldcg(pt + (long)y * (BT * BT) + tid);
                v[1] += __ldcg(pt + (long)y * (BT * BT) + tid + THREADS);
            }
            if (tid == 0) cnt[tile] = 0;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + h * THREADS;
            const int gm = m0 + e / BT, gn = n0 + e % BT;
            if (gm >= M || gn >= N || (tri && gm > gn)) continue;
            double* dst = C + (long)gm * ldc + gn;
            const double r = alpha * v[h];
            *dst = beta == 0.0 ? r : r + beta * (*dst);
            if (tri && gm != gn) C[(long)gn * ldc + gm] = r;
        }
    }
}

// out[i][j] = in[i][j] * f(v[i]) with rows, cols, ldi, ldo = desc[0..3]
__global__ void scale_rows_dyn_kernel(const int* __restrict__ desc, const double* in, const double* v, int mode,
                                      double* out) {
    const int rows = desc[0], cols = desc[1];
    const long ldi = desc[2], ldo = desc[3];
    const long total = (long)rows * cols;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int i = (int)(t / cols), j = (int)(t % cols);
        const double x = v[i];
        double f;
        switch (mode) {
            case 0: f = x; break;
            case 1: f = sqrt(x); break;
            case 2: f = 1.0 / sqrt(x); break;
            default: f = 1.0 / x; break;
        }
        out[(long)i * ldo + j] = in[(long)i * ldi + j] * f;
    }
}

__global__ void scale_rows_kernel(int rows, int cols, const double* in, long ldi, const double* v,
                                  int mode, double* out, long ldo) {
    const long total = (long)rows * cols;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int i = (int)(t / cols), j = (int)(t % cols);
        const double x = v[i];
        double f;
        switch (mode) {
            case 0: f = x; break;
            case 1: f = sqrt(x); break;
            case 2: f = 1.0 / sqrt(x); break;
            default: f = 1.0 / x; break;
        }
        out[(long)i * ldo + j] = in[(long)i * ldi + j] * f;
    }
}

__global__ void fill_kernel(double* p, size_t n, double value) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n;
         t += (size_t)gridDim.x * blockDim.x)
        p[t] = value;
}

__global__ void copy2d_kernel(int rows, int cols, const double* in, long ldi, double* out,
                              long ldo) {
    const long total = (long)rows * cols;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total;
         t += (long)gridDim.x * blockDim.x) {
        const int i = (int)(t / cols), j = (int)(t % cols);
        out[(long)i * ldo + j] = in[(long)i * ldi + j];
    }
}

// out[j] = alpha sum_i A[i][j] v[i] for tall A (m x ncols, m >> ncols): block b
// sums its chunk of rows for every column (row groups of the block split the
// chunk and meet in shared memory in a fixed order), a second kernel adds the
// block partials in block order -- deterministic, one pass over A.
constexpr int GEMV_THREADS = 256;
__global__ void __launch_bounds__(GEMV_THREADS)
gemv_t_partial_kernel(long m, int ncols, const double* __restrict__ A, long lda,
                      const double* __restrict__ v, long chunk, double* __restrict__ part) {
    __shared__ double red[GEMV_THREADS];
    const int cw = min(GEMV_THREADS, ((ncols + 31) / 32) * 32);
    const int rg = GEMV_THREADS / cw;
    const int t = threadIdx.x, c0 = t % cw, g = t / cw;
    const long i0 = blockIdx.x * chunk, i1 = min(m, i0 + chunk);
    for (int cb = 0; cb < ncols; cb += cw) {
        const int col = cb + c0;
        double acc = 0.0;
        if (g < rg && col < ncols)
            for (long i = i0 + g; i < i1; i += rg) acc += A[i * lda + col] * v[i];
        red[t] = acc;
        __syncthreads();
        if (g == 0 && col < ncols) {
            double s = red[c0];
            for (int q = 1; q < rg; ++q) s += red[q * cw + c0];
            part[(long)blockIdx.x * ncols + col] = s;
        }
        __syncthreads();
    }
}

__global__ void gemv_t_final_kernel(int nblk, int ncols, double alpha, const double* part,
                                    double* out) {
    for (int col = blockIdx.x * blockDim.x + threadIdx.x; col < ncols; col += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int b = 0; b < nblk; ++b) s += part[(long)b * ncols + col];
        out[col] = alpha * s;
    }
}

}  // namespace

namespace {

inline int grid_for(long total, int threads = 256) {
    long b = (total + threads - 1) / threads;
    return (int)std::max<long>(1, std::min<long>(b, 152L * 32));
}

tt_status launch_prod(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha, const double* A, long lda,
                      const double* B, long ldb, double beta, double* C, long ldc, int ks, double* P, int* cnt, int tri,
                      const int* desc, int tc, long items) {
    // more CTAs than fit at once let the scheduler level uneven tiles
    const unsigned grid = (unsigned)std::max(1L, std::min(items, 152L * 64));
    note_launch();
    if (ta && tb)
        prod_kernel<true, true><<<grid, THREADS, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ks, P, cnt, tri, desc, tc);
    else if (ta)
        prod_kernel<true, false><<<grid, THREADS, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ks, P, cnt, tri, desc, tc);
    else if (tb)
        prod_kernel<false, true><<<grid, THREADS, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ks, P, cnt, tri, desc, tc);
    else
        prod_kernel<false, false><<<grid, THREADS, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, ks, P, cnt, tri, desc, tc);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

// A split product's scratch: the partials, then the arrival counters where
// the caller keeps none (zeroed ahead of the launch).
size_t split_doubles(long tiles, int ks) { return (size_t)tiles * ks * (BT * BT); }
size_t split_scratch(long tiles, int ks) { return ks > 1 ? split_doubles(tiles, ks) + (size_t)(tiles + 1) / 2 : 0; }

tt_status split_prod(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha, const double* A, long lda,
                     const double* B, long ldb, double* C, long ldc, int ks, double* P, int* cnt, int tri) {
    const long tiles = prod_tiles(M, N, tri);
    if (ks > 1 && !cnt) {
        cnt = reinterpret_cast<int*>(P + split_doubles(tiles, ks));
        TT_CUDA_TRY(cudaMemsetAsync(cnt, 0, (size_t)tiles * sizeof(int), s));
    }
    return launch_prod(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc, ks, P, cnt, tri, nullptr, 0, tiles * ks);
}

}  // namespace

tt_status dgemm(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha,
                const double* A, long lda, const double* B, long ldb, double beta, double* C,
                long ldc) {
    if (M < 0 || N < 0 || K < 0) {
        set_error("dgemm: negative size");
        return TT_ERR_ARG;
    }
    if (K == 0) {  // C = beta C
        if (beta == 0.0)
            for (int i = 0; i < M; ++i) fill(s, C + (long)i * ldc, N, 0.0);
        return TT_OK;
    }
    if (M == 0 || N == 0) return TT_OK;
    return launch_prod(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, 1, nullptr, nullptr, 0, nullptr, 0,
                       prod_tiles(M, N, 0));
}

size_t dgemm_sk_scratch_doubles(int M, int N, int K) {
    if (tc8_wanted(M, N, K)) return tc8_scratch_doubles(M, N, K, false);
    if (M <= 0 || N <= 0 || K <= 0) return 0;
    return split_scratch(prod_tiles(M, N, 0), prod_split(M, N, K, 0));
}

tt_status dgemm_sk(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha,
                   const double* A, long lda, const double* B, long ldb, double* C, long ldc,
                   DevBuf& scratch, int* status_dev, int* counters) {
    if (tc8_wanted(M, N, K)) {
        const tt_status st = tc8_gemm(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, C, ldc, scratch, status_dev);
        if (st != TT_ERR_OOM) return st;  // without room for the digits: the FP64 pipe
    }
    const int ks = M > 0 && N > 0 && K > 0 ? prod_split(M, N, K, 0) : 1;
    if (ks == 1) return dgemm(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc);
    TT_TRY(scratch.ensure(split_scratch(prod_tiles(M, N, 0), ks), s));
    return split_prod(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, C, ldc, ks, scratch.p, counters, 0);
}

size_t gram_scratch_doubles(int m, int n) {
    const int K = std::max(m, 1);
    return split_scratch(prod_tiles(n, n, 1), prod_split(n, n, K, 1));
}

tt_status gram_fixed_scratch(cudaStream_t s, int m, int n, const double* A, long lda, double* G,
                             long ldg, double* scratch, size_t scratch_doubles, int* counters) {
    if (m < 0 || n < 0) {
        set_error("gram: negative size");
        return TT_ERR_ARG;
    }
    if (n == 0) return TT_OK;
    if (m == 0) {
        for (int i = 0; i < n; ++i) fill(s, G + (long)i * ldg, n, 0.0);
        return TT_OK;
    }
    const long tiles = prod_tiles(n, n, 1);
    int ks = prod_split(n, n, m, 1);
    while (ks > 1 && split_scratch(tiles, ks) > scratch_doubles) --ks;
    ks = prod_final(m, ks);
    // op(A) = A^T (stored m x n), op(B) = A
    return split_prod(s, true, false, n, n, m, 1.0, A, lda, A, lda, G, ldg, ks, scratch, counters, 1);
}

size_t dyn_partials_need(int mode, int Mcap, int Ncap, int Kcap) {
    // prod_limit: a split product has at most SPLIT_ITEMS items
    return Mcap > 0 && Ncap > 0 && Kcap > BK ? (size_t)SPLIT_ITEMS * BT * BT : 0;
}

tt_status dgemm_dyn(cudaStream_t s, bool ta, bool tb, const int* desc, int Mcap, int Ncap, int Kcap,
                    double alpha, const double* A, const double* B, double* C, double* P, size_t pcap, int mode,
                    DevBuf& tcbuf, int* status_dev, int* counters) {
    if (Mcap <= 0 || Ncap <= 0) return TT_OK;
    const int tri = mode == 2 ? 1 : 0;
    const int tc = tc8_wanted(Mcap, Ncap, Kcap) ? 1 : 0;
    if (tc) TT_TRY(tc8_dyn(s, ta, tb, desc, Mcap, Ncap, Kcap, alpha, A, B, C, tcbuf, status_dev, mode == 2));
    if (dyn_partials_need(mode, Mcap, Ncap, Kcap) > pcap) {
        set_error("dgemm: the partials buffer of a captured product is smaller than its split needs");
        return TT_ERR_TOO_LARGE;
    }
    // four CTAs an SM, or fewer where the capacity has no more items, walk
    // whatever the device's sizes give
    return launch_prod(s, ta, tb, 0, 0, 0, alpha, A, 0, B, 0, 0.0, C, 0, 1, P, counters, tri, desc, tc,
                       std::min(152L * 4, prod_tiles(Mcap, Ncap, tri) * MAX_SPLIT));
}

void scale_rows_dyn(cudaStream_t s, const int* desc, long total_cap, const double* in, const double* v, int mode,
                    double* out) {
    if (total_cap <= 0) return;
    note_launch();
    scale_rows_dyn_kernel<<<grid_for(total_cap), 256, 0, s>>>(desc, in, v, mode, out);
}

tt_status gram(cudaStream_t s, int m, int n, const double* A, long lda, double* G, long ldg,
               DevBuf& partials, int* status_dev, int* counters) {
    if (n <= 0) return TT_OK;
    if (tc8_wanted(n, n, m)) {
        const tt_status st = tc8_gram(s, m, n, A, lda, G, ldg, partials, status_dev);
        if (st != TT_ERR_OOM) return st;
    }
    TT_TRY(partials.ensure(gram_scratch_doubles(m, n), s));
    return gram_fixed_scratch(s, m, n, A, lda, G, ldg, partials.p, partials.cap, counters);
}

void scale_rows(cudaStream_t s, int rows, int cols, const double* in, long ldi, const double* v,
                int mode, double* out, long ldo) {
    if (rows <= 0 || cols <= 0) return;
    note_launch();
    scale_rows_kernel<<<grid_for((long)rows * cols), 256, 0, s>>>(rows, cols, in, ldi, v, mode,
                                                                 out, ldo);
}

tt_status gemv_t(cudaStream_t s, long m, int ncols, double alpha, const double* A, long lda,
                 const double* v, double* out, DevBuf& scratch) {
    if (ncols <= 0) return TT_OK;
    if (m <= 0) {
        fill(s, out, (size_t)ncols, 0.0);
        return TT_OK;
    }
    // about 4 blocks per SM, at least 64 rows each
    const long chunk = std::max<long>(64, (m + 152L * 4 - 1) / (152L * 4));
    const int nblk = (int)((m + chunk - 1) / chunk);
    TT_TRY(scratch.ensure((size_t)nblk * ncols, s));
    note_launch();
    gemv_t_partial_kernel<<<nblk, GEMV_THREADS, 0, s>>>(m, ncols, A, lda, v, chunk, scratch.p);
    note_launch();
    gemv_t_final_kernel<<<std::max(1, std::min(152, (ncols + 127) / 128)), 128, 0, s>>>(
        nblk, ncols, alpha, scratch.p, out);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

void fill(cudaStream_t s, double* p, size_t n, double value) {
    if (n == 0) return;
    note_launch();
    fill_kernel<<<grid_for((long)n), 256, 0, s>>>(p, n, value);
}

void copy2d(cudaStream_t s, int rows, int cols, const double* in, long ldi, double* out,
            long ldo) {
    if (rows <= 0 || cols <= 0) return;
    note_launch();
    copy2d_kernel<<<grid_for((long)rows * cols), 256, 0, s>>>(rows, cols, in, ldi, out, ldo);
}

namespace {
constexpr int PEAK_ITERS = 2048;
__global__ void __launch_bounds__(256) fp64_mma_peak_kernel(double* out, double seed) {
    const double a = seed * (threadIdx.x + 1), b = 1.0 + 1e-3 * threadIdx.x;
    double c[8][2];
#pragma unroll
    for (int j = 0; j < 8; ++j) c[j][0] = c[j][1] = 0.0;
    for (int i = 0; i < PEAK_ITERS; ++i) {
#pragma unroll
        for (int j = 0; j < 8; ++j) dmma(c[j], a, b);
    }
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) s += c[j][0] + c[j][1];
    if (s == 1234.5) out[threadIdx.x] = s;  // keeps the chains live; never true in practice
}
}  // namespace

tt_status autotune_install(const int* table, int n) {
    if (n != AT_TILE_BUCKETS * AT_K_BUCKETS) {
        set_error("autotune: the table has " + std::to_string(AT_TILE_BUCKETS * AT_K_BUCKETS) + " entries");
        return TT_ERR_ARG;
    }
    for (int i = 0; i < n; ++i)
        if (table[i] < 0 || table[i] > 64) {
            set_error("autotune: splits are 0 (the rule) or 1 .. 64");
            return TT_ERR_ARG;
        }
    TT_CUDA_TRY(cudaMemcpyToSymbol(d_sk_table, table, n * sizeof(int)));
    for (int i = 0; i < n; ++i) h_sk_table[i] = table[i];
    return TT_OK;
}

void autotune_read(int* table) {
    for (int i = 0; i < AT_TILE_BUCKETS * AT_K_BUCKETS; ++i) table[i] = h_sk_table[i];
}

// Measure, for every (tile-count, depth) bucket up to 2^14 deep, the products'
// time at each split of K the rule allows (1, 2, 4, ..., 64, capped at K / 32)
// on a representative product of that bucket (M x N tiles of 64, the
// bucket's smallest K), and keep the fastest (best of three runs each).
tt_status autotune(cudaStream_t s, int* table_out) {
    constexpr int KB_MAX = 14;
    const long Mmax = 64L << ((AT_TILE_BUCKETS - 1) / 2), Nmax = 64L << (AT_TILE_BUCKETS - 1 - (AT_TILE_BUCKETS - 1) / 2);
    const long Kmax = 1L << KB_MAX;
    double *A = nullptr, *B = nullptr, *C = nullptr, *P = nullptr;
    const size_t pdbl = (size_t)SPLIT_ITEMS * BT * BT;
    int* cnt = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    tt_status st = TT_OK;
    int table[AT_TILE_BUCKETS * AT_K_BUCKETS] = {0};
    auto cleanup = [&]() {
        if (A) cudaFreeAsync(A, s);
        if (B) cudaFreeAsync(B, s);
        if (C) cudaFreeAsync(C, s);
        if (P) cudaFreeAsync(P, s);
        if (cnt) cudaFreeAsync(cnt, s);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
    };
    if (cudaMallocAsync((void**)&A, Mmax * Kmax * sizeof(double), s) != cudaSuccess ||
        cudaMallocAsync((void**)&B, Kmax * Nmax * sizeof(double), s) != cudaSuccess ||
        cudaMallocAsync((void**)&C, Mmax * Nmax * sizeof(double), s) != cudaSuccess ||
        cudaMallocAsync((void**)&P, pdbl * sizeof(double), s) != cudaSuccess ||
        cudaMallocAsync((void**)&cnt, SPLIT_ITEMS * sizeof(int), s) != cudaSuccess ||
        cudaMemsetAsync(cnt, 0, SPLIT_ITEMS * sizeof(int), s) != cudaSuccess ||
        cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        (void)cudaGetLastError();
        cleanup();
        set_error("autotune: device memory for the trial products");
        return TT_ERR_OOM;
    }
    fill(s, A, (size_t)(Mmax * Kmax), 0.5);
    fill(s, B, (size_t)(Kmax * Nmax), 0.25);
    for (int tb = 0; tb < AT_TILE_BUCKETS && st == TT_OK; ++tb) {
        const int M = 64 << (tb / 2), N = 64 << (tb - tb / 2);
        for (int kb = 6; kb <= KB_MAX && st == TT_OK; ++kb) {
            const int K = 1 << kb;
            float best = 1e30f;
            int best_ks = 0;
            for (int ks = 1; ks <= 64 && ks <= std::max(1, K / (2 * BK)); ks *= 2) {
                const int kk = prod_final(K, std::min(ks, prod_limit(prod_tiles(M, N, 0), K)));
                float t = 1e30f;
                for (int rep = 0; rep < 3; ++rep) {
                    cudaEventRecord(e0, s);
                    st = launch_prod(s, false, false, M, N, K, 1.0, A, K, B, N, 0.0, C, N, kk, P, cnt, 0, nullptr, 0,
                                     prod_tiles(M, N, 0) * kk);
                    cudaEventRecord(e1, s);
                    if (st < 0 || cudaEventSynchronize(e1) != cudaSuccess) {
                        if (st >= 0) st = TT_ERR_CUDA;
                        break;
                    }
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    t = std::min(t, ms);
                }
                if (st < 0) break;
                if (t < best) {
                    best = t;
                    best_ks = ks;
                }
            }
            table[tb * AT_K_BUCKETS + kb] = best_ks;
        }
    }
    // deeper products keep the choice of the deepest measured bucket
    for (int tb = 0; tb < AT_TILE_BUCKETS; ++tb)
        for (int kb = KB_MAX + 1; kb < AT_K_BUCKETS; ++kb) table[tb * AT_K_BUCKETS + kb] = table[tb * AT_K_BUCKETS + KB_MAX];
    cleanup();
    if (st < 0) return st;
    TT_TRY(autotune_install(table, AT_TILE_BUCKETS * AT_K_BUCKETS));
    if (table_out)
        for (int i = 0; i < AT_TILE_BUCKETS * AT_K_BUCKETS; ++i) table_out[i] = table[i];
    return TT_OK;
}

tt_status bench_fp64_mma(cudaStream_t s, double* tflops) {
    int dev = 0, sms = 0;
    TT_CUDA_TRY(cudaGetDevice(&dev));
    TT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    double* out = nullptr;
    TT_CUDA_TRY(cudaMallocAsync((void**)&out, 256 * sizeof(double), s));
    cudaEvent_t e0, e1;
    TT_CUDA_TRY(cudaEventCreate(&e0));
    TT_CUDA_TRY(cudaEventCreate(&e1));
    const int blocks = sms * 8;
    float best = 1e30f;
    for (int rep = 0; rep < 4; ++rep) {
        TT_CUDA_TRY(cudaEventRecord(e0, s));
        note_launch();
        fp64_mma_peak_kernel<<<blocks, 256, 0, s>>>(out, 1e-3);
        TT_CUDA_TRY(cudaEventRecord(e1, s));
        TT_CUDA_TRY(cudaEventSynchronize(e1));
        float ms = 0.f;
        TT_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
        if (rep > 0) best = std::min(best, ms);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFreeAsync(out, s);
    const double flops = 2.0 * 8 * 8 * 4 * 8.0 * PEAK_ITERS * blocks * (256 / 32);
    *tflops = flops / (best * 1e-3) / 1e12;
    return TT_OK;
}

}  // namespace ttsn
