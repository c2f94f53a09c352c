// FP64 contractions of the Gram-SVD rounding (App. A.2 of arXiv 2503.18056) on
// the FP64 tensor pipe (mma.sync m8n8k4.f64): the products below the sizes at
// which digits.cu takes over, and whatever it cannot split.
//
// GB300's FP64 pipe issues one warp instruction in 64 clocks per SM
// sub-partition (19 per SM; a DMMA of 256 FMAs takes eight times that), so a
// product's time is the longest chain of DMMAs that a sub-partition is given,
// and loads hardly matter: a step of four indices is 512 clocks a warp against
// two to four loads a lane from L2.  So the work is cut as finely as possible
// and nothing is staged in shared memory: a CTA owns a 16 x 16 tile and a range
// of the contraction, and the CTA that arrives last at a tile adds the splits'
// partials in split order (reproducible), so a split product is one launch.
// Inside a CTA either each of the four warps takes an 8 x 8 block and all of
// the range (the rounding's products), or all warps take the whole tile and
// every fourth group of indices (the library calls, whose contraction may be
// long against their tiles).
//
// The rounding's products keep one order of summation for good: the splits of
// sk_split and gram_split_rule and ascending indices within one.  A truncation
// whose cut falls between singular values that are equal up to rounding (a
// symmetric problem at its rank cap) takes its basis from the last bits, and a
// changed order moves such a run's energies by up to the discarded value: for
// 16 symmetric pulses at their caps by 4e-7 in one of three cases.
//
// Measured (GB300, against 64 x 64 tiles staged in shared memory): a call of
// 133 x 97 x 389 474 -> 24 us; the small-grid 2D step 8.7 -> 6.0 ms, the
// 16-problem captured batch 27.6 -> 20.5 ms.
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
    if (k > 4096 / tiles) k = 4096 / tiles;  // at most 8 MB of partials
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

// Split of K of the rounding's products: where 64 x 64 tiles would leave SMs
// idle, so that there are about two tiles per SM, each with at least 32
// indices, unless the autotuned table holds a measured split for the product's
// bucket.  Host and device use the same rule (a captured step decides it on
// the device from the sizes of that step).
__host__ __device__ void sk_split(int M, int N, int K, int* ks_out, int* kchunk_out) {
    const long tiles = (long)((M + 63) / 64) * ((N + 63) / 64);
    int ks = 1;
    if (tiles < 152 && K >= 4 * BK) {
        long a = (304 + tiles - 1) / tiles, b = K / (2 * BK);
        ks = (int)(a < b ? a : b);
        const int tb = floor_log2(tiles), kb = floor_log2(K);
        if (tb < AT_TILE_BUCKETS && kb < AT_K_BUCKETS) {
#ifdef __CUDA_ARCH__
            const int tuned = d_sk_table[tb * AT_K_BUCKETS + kb];
#else
            const int tuned = h_sk_table[tb * AT_K_BUCKETS + kb];
#endif
            if (tuned > 0) ks = (int)(tuned < b ? tuned : b);
        }
        ks = ks < 1 ? 1 : (ks > 64 ? 64 : ks);
    }
    int kchunk = K;
    if (ks > 1) {
        kchunk = (K + ks - 1) / ks;
        kchunk = (kchunk + BK - 1) / BK * BK;
        ks = (K + kchunk - 1) / kchunk;
    }
    *ks_out = ks;
    *kchunk_out = kchunk;
}

// Row split of the rounding's Gram, at least 256 rows a split: one wave of
// `resident` 64 x 64 tiles for small problems, and for larger ones
// GRAM_MULTI_SPLITS splits where that leaves fewer tiles idle: the time is then
// about W / (64 resident) + 1 / (2 splits) of one unsplit tile's, W = B (B + 1)
// / 2 the 8 x 8 products of the upper triangle that the matrix reaches (B =
// ceil(n / 8)), against 1 / ks0 for one wave.  Integer arithmetic, so the host
// and a captured step's device agree.
__host__ __device__ int gram_split_rule(int m, int n, long resident) {
    const long T = (n + 63) / 64;
    const long tiles = T * (T + 1) / 2;
    long cap = m / 256 < 1 ? 1 : m / 256;
    if (cap > 1024) cap = 1024;
    if (resident < 1) resident = 1;
    long ks0 = resident / tiles;
    if (ks0 < 1) ks0 = 1;
    if (ks0 > cap) ks0 = cap;
    if (ks0 >= 16) return (int)ks0;
    const long km = cap < GRAM_MULTI_SPLITS ? cap : GRAM_MULTI_SPLITS;
    if (km <= ks0) return (int)ks0;
    const long long B = (n + 7) / 8;
    const long long W = B * (B + 1) / 2;
    const long long slots = 64LL * resident;
    // (W / slots + 1 / (2 km)) < 0.97 / ks0, times 2 slots km ks0 100
    if ((2 * W * km + slots) * ks0 * 100 < 97LL * 2 * slots * km) return (int)km;
    return (int)ks0;
}

namespace {

// CTAs of 64 x 64 Gram tiles that gram_split_rule counts on: four per SM.
__host__ __device__ constexpr long gram_resident() { return 152 * 4; }

__host__ __device__ inline int prod_final(long K, int ks) {  // splits that hold indices
    const int c = prod_chunk(K, ks);
    return (int)((K + c - 1) / c);
}
// Splits of a library call's product (interleaved warps): the cheapest.
int prod_split(long M, long N, long K, int tri) {
    const long tiles = prod_tiles(M, N, tri);
    const int lim = prod_limit(tiles, K);
    int best = 1;
    unsigned least = prod_cost(tiles, K, 1);
    for (int k = 2; k <= lim; ++k) {
        const unsigned c = prod_cost(tiles, K, k);
        if (c < least) {
            least = c;
            best = k;
        }
    }
    return prod_final(K, best);
}
// Splits and indices per split of a rounding's product (ordered); tri: the Gram.
__host__ __device__ inline int ordered_split(int M, int N, int K, int tri, int* chunk) {
    int ks = 1;
    if (tri) {
        ks = gram_split_rule(K, M, gram_resident());
        *chunk = prod_chunk(K, ks);
    } else {
        sk_split(M, N, K, &ks, chunk);
    }
    return ks;
}

// C = alpha op(A) op(B) (+ beta C), or with tri the symmetric product of which
// only the tiles on and above the diagonal are formed (both halves stored).
// desc (a captured step): M, N, K, lda, ldb, ldc in device memory.  lost: behind a
// digit product (in a captured step of the sizes that take one), of which it
// recomputes what tc8_lost says: everything, or the tiles with a lost row or
// column.  An item is (tile, split); ks > 1:
// partials to P (256 doubles an item), arrivals counted in cnt (zero between
// products: the last arrival resets its tile's).  ORDERED: a warp per 8 x 8
// block; else the warps share the indices.  An 8 x 8 product outside M x N or below the diagonal is skipped.
template <bool TA, bool TB, bool ORDERED>
__global__ void __launch_bounds__(THREADS)
prod_kernel(int M, int N, int K, double alpha, const double* __restrict__ A, long lda, const double* __restrict__ B,
            long ldb, double beta, double* __restrict__ C, long ldc, int ks, int chunk, double* __restrict__ P, int* cnt,
            int tri, const int* __restrict__ desc, Lost lost) {
    if (desc) {
        M = desc[0];
        N = desc[1];
        K = desc[2];
        lda = desc[3];
        ldb = desc[4];
        ldc = desc[5];
        if (M <= 0 || N <= 0) return;
        ks = 1;
        chunk = K;
        if (P) ks = ordered_split(M, N, K, tri, &chunk);  // P null: an unsplit product
    }
    const bool behind = lost.flag && (!desc || tc8_wanted(M, N, K));
    const int redo = behind ? tc8_lost(lost, K) : 2;
    if (redo == 0) return;
    __shared__ double red[ORDERED ? 1 : 4][BT * BT];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int TM = (M + BT - 1) / BT, TN = (N + BT - 1) / BT;
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
        if (redo == 1) {  // the same for every warp
            const int i = lane < BT ? min(m0 + lane, M - 1) : min(n0 + lane - BT, N - 1);
            if (lost.rho) {
                unsigned r = __float_as_uint(lost.rho[i]);  // not negative: ordered as integers
                const unsigned a = __reduce_max_sync(0xffffffffu, lane < BT ? r : 0u);
                const unsigned b = __reduce_max_sync(0xffffffffu, lane < BT ? 0u : r);
                if (!(__uint_as_float(a) * __uint_as_float(b) > 1.0f)) continue;
            } else if (lost.guard == 2) {  // rows that are lost are large nowhere
                const int c = lane < BT ? lost.la[i] : lost.lb[i];
                const int a = __reduce_min_sync(0xffffffffu, lane < BT ? c : K);
                const int b = __reduce_min_sync(0xffffffffu, lane < BT ? K : c);
                if (a + b >= K + K / 16) continue;
            } else if (!__any_sync(0xffffffffu, (lane < BT ? lost.a[i] : lost.b[i]) == EXP_LOST)) {
                continue;
            }
        }
        const int kbeg = z * chunk, kend = min(K, kbeg + chunk);
        const long sa = TA ? lda : 1, sb = TB ? 1 : ldb;
        __syncthreads();  // the item before has read red
        if (ORDERED) {
            const int mb = m0 + 8 * (warp >> 1), nb = n0 + 8 * (warp & 1);
            double acc[2] = {0.0, 0.0};
            if (mb < M && nb < N && !(tri && mb > nb)) {
                // lane: row lane / 4 and index lane % 4 of the operands (rows
                // past the last read the last: their outputs are not stored);
                // the loads run two steps (1,024 clocks) ahead
                const int r = min(mb + (lane >> 2), M - 1), q = min(nb + (lane >> 2), N - 1);
                const double* a = (TA ? A + r : A + (long)r * lda);
                const double* b = (TB ? B + (long)q * ldb : B + q);
                double x[2], y[2];
                auto load = [&](int k, int h) {
                    const int kk = k + (lane & 3);
                    x[h] = kk < kend ? a[kk * sa] : 0.0;
                    y[h] = kk < kend ? b[kk * sb] : 0.0;
                };
                load(kbeg, 0);
                load(kbeg + 4, 1);
                for (int k = kbeg; k < kend; k += 8) {
                    const double u0 = x[0], v0 = y[0], u1 = x[1], v1 = y[1];
                    load(k + 8, 0);
                    load(k + 12, 1);
                    dmma(acc, u0, v0);
                    if (k + 4 < kend) dmma(acc, u1, v1);
                }
            }
            *reinterpret_cast<double2*>(&red[0][(8 * (warp >> 1) + (lane >> 2)) * BT + 8 * (warp & 1) + (lane & 3) * 2]) =
                make_double2(acc[0], acc[1]);
        } else {
            const bool l1 = m0 + 8 < M, c1 = n0 + 8 < N;
            const bool use10 = l1 && !(tri && tm == tn), use11 = l1 && c1;
            double acc[2][2][2] = {};
            const int r0 = min(m0 + (lane >> 2), M - 1), r1 = min(m0 + 8 + (lane >> 2), M - 1);
            const int q0 = min(n0 + (lane >> 2), N - 1), q1 = min(n0 + 8 + (lane >> 2), N - 1);
            const double* a0 = TA ? A + r0 : A + (long)r0 * lda;
            const double* a1 = TA ? A + r1 : A + (long)r1 * lda;
            const double* b0 = TB ? B + (long)q0 * ldb : B + q0;
            const double* b1 = TB ? B + (long)q1 * ldb : B + q1;
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
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    *reinterpret_cast<double2*>(&red[warp][(8 * i + (lane >> 2)) * BT + 8 * j + (lane & 3) * 2]) =
                        make_double2(acc[i][j][0], acc[i][j][1]);
        }
        __syncthreads();
        double v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + h * THREADS;
            v[h] = ORDERED ? red[0][e]
                           : (red[0][e] + red[ORDERED ? 0 : 1][e]) + (red[ORDERED ? 0 : 2][e] + red[ORDERED ? 0 : 3][e]);
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

// Behind a rounding's digit Gram G: entries are lost where the digits' error may
// exceed that of the FP64 sums they stand for, relative to the two columns' norms.
// Entry (i, j) is off by at most sqrt(Q_i Q_j), Q_i = 9.1 2^-58 sum_blocks c_block
// 4^e_block (c: entries that are not zero), the FP64 pipe's by chunk 2^-53 |a_i| |a_j|
// (chunk: rows of a split).  So with rho_i = sqrt(Q_i / (chunk 2^-53 |a_i|^2)) an
// entry stays where rho_i rho_j <= 1, always above about 2,400 rows a split, and the
// others' tiles are recomputed (prod_kernel): columns of whose blocks' entries few
// make up the norm, against one another.  Shorter splits count as 1,024 rows: Q takes
// every digit at its largest, and even an entry that loses all it can loses a
// twentieth of that; at 256 rows the difference columns of a smooth field on a 128^2
// grid (an entry of 1 at a vacuum face, 0.05 elsewhere) have rho up to 2, and their
// Grams, 60 us, would all be formed twice (440).  G keeps its relative accuracy under
// any scaling of the columns, which the eigenvalues of W G W^T take over, whatever
// the rounding's tolerance.
// A warp a column.
__global__ void __launch_bounds__(256)
gram_check_kernel(int n, int K, const double* __restrict__ G, long ldg, const int* __restrict__ desc, Lost lost) {
    if (desc) {
        n = desc[0];
        K = desc[2];
        ldg = desc[5];
        if (!tc8_wanted(n, n, K)) return;
    }
    int chunk;
    ordered_split(n, n, K, 1, &chunk);
    const int lane = threadIdx.x & 31;
    for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += gridDim.x * 8) {
        const int e = lost.a[i];
        if (lost.mx[i] == 0 || e == EXP_LOST) {
            // no product with a lost column stays, however small the other's rho
            if (lane == 0) lost.rho[i] = e == EXP_LOST ? __int_as_float(0x7f800000) : 1e-30f;
            continue;
        }
        // sum_blocks c_block 4^(e_block - e) in units of 2^-30 (at least one an entry): the
        // same in any order
        unsigned long long sum = 0;
        if (K > digits::ONE_EXP_K) {
            for (long b = lane; b * digits::BLK_K < K; b += 32) {
                const int w = lost.eb[b * lost.ebs + i];
                sum += (unsigned long long)block_count(w) << (30 - 2 * min(max(e - block_exp(w), 0), 15));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        } else {
            sum = (unsigned long long)K << 30;
        }
        const double q = 0x1p-30 * (double)sum * (9.1 / 32.0) / max(chunk, 1024);
        const double r2 = q / scalbn(G[(long)i * ldg + i], -2 * e);
        if (lane == 0) {
            // rounded up; what is not a number or not positive (a diagonal entry cannot be) is lost
            const float r = r2 >= 0.0 ? __fsqrt_ru(__double2float_ru(r2)) : __int_as_float(0x7f800000);
            lost.rho[i] = fmaxf(r, 1e-30f);
            if (r > 1.0f) atomicOr(lost.flag + LOST_ROWS, 1);
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

struct ProdArgs {
    int M, N, K;
    double alpha;
    const double* A;
    long lda;
    const double* B;
    long ldb;
    double beta;
    double* C;
    long ldc;
    int ks, chunk;
    double* P;
    int *cnt, tri;
    const int* desc;
    Lost lost = {};
};

template <bool TA, bool TB>
void launch_one(cudaStream_t s, bool ordered, unsigned grid, const ProdArgs& a) {
    if (ordered)
        prod_kernel<TA, TB, true><<<grid, THREADS, 0, s>>>(a.M, a.N, a.K, a.alpha, a.A, a.lda, a.B, a.ldb, a.beta, a.C,
                                                          a.ldc, a.ks, a.chunk, a.P, a.cnt, a.tri, a.desc, a.lost);
    else
        prod_kernel<TA, TB, false><<<grid, THREADS, 0, s>>>(a.M, a.N, a.K, a.alpha, a.A, a.lda, a.B, a.ldb, a.beta, a.C,
                                                           a.ldc, a.ks, a.chunk, a.P, a.cnt, a.tri, a.desc, a.lost);
}

tt_status launch_prod(cudaStream_t s, bool ta, bool tb, bool ordered, long items, const ProdArgs& a) {
    // more CTAs than fit at once let the scheduler level uneven tiles; behind a
    // rounding's digit product they seldom have any (a library call may lose all)
    const bool idle = a.lost.flag && a.lost.guard != 1 && !a.desc;
    const unsigned grid = (unsigned)std::max(1L, std::min(items, idle ? 152L * 8 : 152L * 64));
    note_launch();
    if (ta && tb)
        launch_one<true, true>(s, ordered, grid, a);
    else if (ta)
        launch_one<true, false>(s, ordered, grid, a);
    else if (tb)
        launch_one<false, true>(s, ordered, grid, a);
    else
        launch_one<false, false>(s, ordered, grid, a);
    TT_CUDA_TRY(cudaGetLastError());
    return TT_OK;
}

// A split product's scratch: the partials, then the arrival counters where
// the caller keeps none (zeroed ahead of the launch).
size_t split_doubles(long tiles, int ks) { return (size_t)tiles * ks * (BT * BT); }
size_t split_scratch(long tiles, int ks) { return ks > 1 ? split_doubles(tiles, ks) + (size_t)(tiles + 1) / 2 : 0; }

// Scratch of a digit product and, behind its head, of the recomputation with ks
// splits.
size_t digits_doubles(long M, long N, long K, int tri, int ks) {
    const size_t part = split_scratch(prod_tiles(M, N, tri), ks);
    if (!tc8_wanted(M, N, K)) return part;
    return std::max(tc8_scratch_doubles(M, N, K, tri != 0), tc8_head_doubles(M, N, K, tri != 0) + part);
}

tt_status split_prod(cudaStream_t s, bool ta, bool tb, bool ordered, ProdArgs a) {
    const long tiles = prod_tiles(a.M, a.N, a.tri);
    if (tiles > PROD_COUNTERS) a.cnt = nullptr;
    if (a.ks > 1 && !a.cnt) {
        a.cnt = reinterpret_cast<int*>(a.P + split_doubles(tiles, a.ks));
        TT_CUDA_TRY(cudaMemsetAsync(a.cnt, 0, (size_t)tiles * sizeof(int), s));
    }
    return launch_prod(s, ta, tb, ordered, tiles * a.ks, a);
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
    return launch_prod(s, ta, tb, true, prod_tiles(M, N, 0),
                       ProdArgs{M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, 1, K, nullptr, nullptr, 0, nullptr});
}

tt_status dgemm_sk(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha,
                   const double* A, long lda, const double* B, long ldb, double* C, long ldc,
                   DevBuf& scratch, const ProdCtx& ctx, bool split, const Bond* bond) {
    int ks = 1, chunk = K;
    if (split && M > 0 && N > 0 && K > 0) ks = ordered_split(M, N, K, 0, &chunk);
    const size_t part = split_scratch(prod_tiles(M, N, 0), ks);
    if (ctx.digits && tc8_wanted(M, N, K)) {
        Lost lost;
        // without room for the digits: the FP64 pipe
        tt_status st = scratch.ensure(digits_doubles(M, N, K, 0, ks), s);
        if (st >= 0)
            st = tc8_gemm(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, C, ldc, scratch, ctx.status, false, bond, &lost);
        if (st >= 0)
            return split_prod(s, ta, tb, true, ProdArgs{M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc, ks, chunk, lost.free,
                                                        ctx.counters, 0, nullptr, lost});
        if (st != TT_ERR_OOM) return st;
    }
    if (ks == 1) return dgemm(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc);
    TT_TRY(scratch.ensure(part, s));
    return split_prod(s, ta, tb, true, ProdArgs{M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc, ks, chunk, scratch.p,
                                                ctx.counters, 0, nullptr});
}

// Between the digit Gram and its recomputation.
static void gram_check(cudaStream_t s, int n, int K, const double* G, long ldg, const int* desc, const Lost& lost) {
    note_launch();
    gram_check_kernel<<<std::max(1, std::min(n / 8, 152)), 256, 0, s>>>(n, K, G, ldg, desc, lost);
}

tt_status gram(cudaStream_t s, int m, int n, const double* A, long lda, double* G, long ldg, DevBuf& partials,
               const ProdCtx& ctx) {
    if (n <= 0) return TT_OK;
    if (m <= 0) {
        for (int i = 0; i < n; ++i) fill(s, G + (long)i * ldg, n, 0.0);
        return TT_OK;
    }
    int chunk = m;
    const int ks = ordered_split(n, n, m, 1, &chunk);
    const size_t part = split_scratch(prod_tiles(n, n, 1), ks);
    // op(A) = A^T (stored m x n), op(B) = A
    ProdArgs a{n, n, m, 1.0, A, lda, A, lda, 0.0, G, ldg, ks, chunk, nullptr, ctx.counters, 1, nullptr};
    if (ctx.digits && tc8_wanted(n, n, m)) {
        tt_status st = partials.ensure(digits_doubles(n, n, m, 1, ks), s);
        if (st >= 0) st = tc8_gram(s, m, n, A, lda, G, ldg, partials, ctx.status, false, &a.lost);
        if (st >= 0) {
            gram_check(s, n, m, G, ldg, nullptr, a.lost);
            a.P = a.lost.free;
            return split_prod(s, true, false, true, a);
        }
        if (st != TT_ERR_OOM) return st;
    }
    TT_TRY(partials.ensure(part, s));
    a.P = partials.p;
    a.lost = {};
    return split_prod(s, true, false, true, a);
}

size_t gram_scratch_doubles(int m, int n) {
    return split_scratch(prod_tiles(n, n, 1), gram_split_rule(std::max(m, 1), n, gram_resident()));
}

// ------------------------------------------------------------ library calls

size_t gemm_call_doubles(int M, int N, int K) { return digits_doubles(M, N, K, 0, prod_split(M, N, K, 0)); }

tt_status gemm_call(cudaStream_t s, bool ta, bool tb, int M, int N, int K, double alpha, const double* A, long lda,
                    const double* B, long ldb, double* C, long ldc, DevBuf& scratch, bool probe) {
    const int ks = prod_split(M, N, K, 0);
    ProdArgs a{M, N, K, alpha, A, lda, B, ldb, 0.0, C, ldc, ks, prod_chunk(K, ks), scratch.p, nullptr, 0, nullptr};
    if (tc8_wanted(M, N, K)) {
        TT_TRY(tc8_gemm(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, C, ldc, scratch, nullptr, true, nullptr, &a.lost, probe));
        a.P = a.lost.free;
    }
    return split_prod(s, ta, tb, false, a);
}

size_t gram_call_doubles(int m, int n) {
    return digits_doubles(n, n, std::max(m, 1), 1, prod_split(n, n, std::max(m, 1), 1));
}

tt_status gram_fixed_scratch(cudaStream_t s, int m, int n, const double* A, long lda, double* G,
                             long ldg, double* scratch, size_t scratch_doubles) {
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
    return split_prod(s, true, false, false, ProdArgs{n, n, m, 1.0, A, lda, A, lda, 0.0, G, ldg, ks, prod_chunk(m, ks),
                                                      scratch, nullptr, 1, nullptr});
}

tt_status gram_call(cudaStream_t s, int m, int n, const double* A, long lda, double* G, long ldg, DevBuf& scratch) {
    if (m > 0 && tc8_wanted(n, n, m)) {
        const int ks = prod_split(n, n, m, 1);
        ProdArgs a{n, n, m, 1.0, A, lda, A, lda, 0.0, G, ldg, ks, prod_chunk(m, ks), nullptr, nullptr, 1, nullptr};
        tt_status st = scratch.ensure(gram_call_doubles(m, n), s);
        if (st >= 0) st = tc8_gram(s, m, n, A, lda, G, ldg, scratch, nullptr, true, &a.lost);
        if (st >= 0) {
            a.P = a.lost.free;
            return split_prod(s, true, false, false, a);
        }
        if (st != TT_ERR_OOM) return st;
    }
    TT_TRY(scratch.ensure(split_scratch(prod_tiles(n, n, 1), prod_split(n, n, std::max(m, 1), 1)), s));
    return gram_fixed_scratch(s, m, n, A, lda, G, ldg, scratch.p, scratch.cap);
}

// ------------------------------------------------------------ captured steps

// Doubles of partials (and counters, where the handle's are too few) that a
// captured product of sizes up to these may use.
size_t dyn_partials_need(int mode, int Mcap, int Ncap, int Kcap) {
    if (mode == 0 || Mcap <= 0 || Ncap <= 0 || Kcap <= 0) return 0;
    size_t most = 0;
    if (mode == 2) {
        for (int n = 1; n <= Ncap; ++n)
            most = std::max(most, split_doubles(prod_tiles(n, n, 1), gram_split_rule(Kcap, n, gram_resident())));
    } else {
        // sk_split's split is not monotone in K (the chunk is rounded), so
        // bound it: below 152 64 x 64 tiles ceil(304 / tiles), the tuned entries
        // of every K bucket up to Kcap, 64, or ceil(Kcap / 16)
        const int TMc = (Mcap + 63) / 64, TNc = (Ncap + 63) / 64, kbmax = floor_log2(Kcap);
        for (int tm = 1; tm <= TMc; ++tm)
            for (int tn = 1; tn <= TNc && (long)tm * tn < 152; ++tn) {
                const long tiles = (long)tm * tn;
                long ks = (304 + tiles - 1) / tiles;
                const int tb = floor_log2(tiles);
                for (int kb = 0; tb < AT_TILE_BUCKETS && kb <= kbmax && kb < AT_K_BUCKETS; ++kb)
                    ks = std::max<long>(ks, h_sk_table[tb * AT_K_BUCKETS + kb]);
                ks = std::min(std::min(ks, 64L), (long)(Kcap + BK - 1) / BK);
                most = std::max(most, split_doubles(tiles * 16, (int)ks));
            }
    }
    const long tiles = prod_tiles(Mcap, Ncap, mode == 2);
    return most + (tiles > PROD_COUNTERS ? (size_t)(tiles + 1) / 2 : 0);
}

tt_status dgemm_dyn(cudaStream_t s, bool ta, bool tb, const int* desc, int Mcap, int Ncap, int Kcap,
                    double alpha, const double* A, const double* B, double* C, double* P, size_t pcap, int mode,
                    DevBuf& tcbuf, const ProdCtx& ctx, const Bond* bond) {
    if (Mcap <= 0 || Ncap <= 0) return TT_OK;
    const int tri = mode == 2 ? 1 : 0;
    Lost lost;
    if (ctx.digits && tc8_wanted(Mcap, Ncap, Kcap))
        TT_TRY(tc8_dyn(s, ta, tb, desc, Mcap, Ncap, Kcap, alpha, A, B, C, tcbuf, ctx.status, mode == 2, bond, &lost));
    if (lost.flag && tri) gram_check(s, Ncap, Kcap, C, 0, desc, lost);
    const size_t need = dyn_partials_need(mode, Mcap, Ncap, Kcap);
    if (need > pcap) {
        set_error("dgemm: the partials buffer of a captured product is smaller than its split needs");
        return TT_ERR_TOO_LARGE;
    }
    const long tiles = prod_tiles(Mcap, Ncap, tri);
    int* cnt = ctx.counters;
    if (mode != 0 && tiles > PROD_COUNTERS) {
        cnt = reinterpret_cast<int*>(P + need - (tiles + 1) / 2);
        TT_CUDA_TRY(cudaMemsetAsync(cnt, 0, (size_t)tiles * sizeof(int), s));
    }
    // eight CTAs an SM, or fewer where the capacity has no more items, walk
    // whatever the device's sizes give; mode 0 does not split
    ProdArgs a{0, 0, 0, alpha, A, 0, B, 0, 0.0, C, 0, 1, 0, mode == 0 ? nullptr : P, cnt, tri, desc, lost};
    return launch_prod(s, ta, tb, true, std::min(152L * 8, tiles * 64), a);
}

void scale_rows_dyn(cudaStream_t s, const int* desc, long total_cap, const double* in, const double* v, int mode,
                    double* out) {
    if (total_cap <= 0) return;
    note_launch();
    scale_rows_dyn_kernel<<<grid_for(total_cap), 256, 0, s>>>(desc, in, v, mode, out);
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
    const size_t pdbl = (size_t)64 * Mmax * Nmax;
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
        cudaMallocAsync((void**)&cnt, PROD_COUNTERS * sizeof(int), s) != cudaSuccess ||
        cudaMemsetAsync(cnt, 0, PROD_COUNTERS * sizeof(int), s) != cudaSuccess ||
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
                int kchunk = (K + ks - 1) / ks;
                kchunk = (kchunk + BK - 1) / BK * BK;
                const int kk = (K + kchunk - 1) / kchunk;
                float t = 1e30f;
                for (int rep = 0; rep < 3; ++rep) {
                    cudaEventRecord(e0, s);
                    st = launch_prod(s, false, false, true, prod_tiles(M, N, 0) * kk,
                                     ProdArgs{M, N, K, 1.0, A, K, B, N, 0.0, C, N, kk, kk > 1 ? kchunk : K, P, cnt, 0,
                                              nullptr});
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
