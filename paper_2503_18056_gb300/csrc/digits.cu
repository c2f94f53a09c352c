// FP64 products on the 5th-generation tensor cores.  GB300's FP64 pipe does
// about 1 TFLOP/s (a warp's DFMA occupies its SM sub-partition for 64 clocks),
// which bounded every contraction of the rounding; its tensor cores multiply
// small integers exactly at 1.9 PFLOP/s.  C = op(A) op(B) is therefore formed
// from exact integer digit products (the error-free splitting of Ozaki, Ogita,
// Oishi, Rump, Numer. Algorithms 59, 2012, with fixed-point digits):
//
//   Split.  Row i of op(A) and column j of op(B) carry a power of two each (of a
//   contraction above 1024 indices, for every block of 512 of them: an entry is
//   measured against its neighbours, not against the whole row), |a_ik| <
//   2^(e_i - 1); a_ik 2^-e_i is rounded to 56-bit fixed point (an entry within a
//   factor 8 of its row's maximum keeps all its 53 bits) and cut into S = 8
//   balanced base-128 digits, d_0 in [0, 64], the others in [-64, 63], each exact
//   in BF16.
//   Products.  d_s d_t (at most 2^12) of level w = s + t <= 7 are summed by
//   tcgen05.mma over at most 512 contraction indices: 8 pairs * 512 * 2^12 =
//   2^24, so the FP32 accumulators hold exact integers.  The dropped levels
//   are about 2^-56 of the maxima's product a term.
//   Sums.  A block's level sums are added as integers (levels 0-3 and 4-7), and
//   the blocks in fixed point under the rows' largest exponents (E_i, E_j), also
//   across splits and chunks of the contraction: the sum is exact (a block more than
//   2^8 below 2^(E_i + E_j) is cut off at 2^-71 of it) and is rounded once to FP64,
//   so the result does not depend on how the work is cut (up to 16384 indices the
//   cut follows from the sizes, above it lies between blocks).
//
// What is lost, the dropped levels and the rounding to 56 bits, is at most 9.1
// 2^-58 2^(e_i + e_j) an index.
// Against the FP64 pipe's running sum (an error of 2^-53 of the partial sum a
// term) the result is nearer to the exact product from K of a few dozen on;
// the sizes where it is used (tc8_wanted) have K >= 64.
//
// Measured (GB300, CUDA events, against the FP64 pipe's kernels): Gram of
// 500,000 x 449 143 -> 5.87 ms (5.67 with one exponent a column), error against the
// exact product 1.3e-15 -> 1.2e-16 (2.4e-16); 200,000 x 577 times 577 x 96 22.4 ->
// 1.8 ms, 8.0e-16 -> 5.5e-16.
//
// Rows that hold Inf or NaN or whose largest entry is outside 2^+-900 cannot be
// split: their exponent is EXP_LOST, their digits are zero, and gemm.cu's
// prod_kernel behind the product, which otherwise returns at once, recomputes the
// 16 x 16 tiles that they reach (tc8_lost), or everything where a wait ran out.
//
// An entry far below its row's (block's) maximum keeps few digits, which matters
// where small entries meet large ones: the sum |a||b| is then far below K max|a_i|
// max|b_j|, which bounds the error.
// - A rounding's Gram is held to its columns' norms (gram_check_kernel in gemm.cu).
// - A handle's other products contract an index that may carry any scaling, one
//   core's columns times D and the next core's rows over D: the sum does not depend
//   on D, but a power of two a row would see D on one side and 1 / D on the other.
//   So they are formed at a scale of the index: the norms of A's columns where a
//   rounding has their Gram matrix (Bond), else the smaller operand's entries
//   (index_max_kernel).  A D of powers of two then changes no bit of tt_to_full.  Such
//   a scale may still hide one operand's blocks from the other's rows; in tt_to_full,
//   whose entries are the caller's, the entries above 2^-9 of a row's maximum are
//   counted, and the 16 x 16 tiles with a row and a column that share fewer than K / 16
//   such indices are recomputed.
//   What the smaller operand gives is not enough in a rounding: P_A's entries go like
//   1 / sigma_j, and its largest ones would set the scale of A' columns to which they
//   do not belong.
// - A library call (A times the identity, disjoint supports) is held to the sum's
//   scale: the split counts each row's entries above 2^-9 of its maximum, and
//   unless every pair of rows has K / 16 indices where both are (tc8_lost), the
//   product is recomputed on the FP64 pipe (the count and the check: 200,000 x 577
//   times 577 x 96 1.73 -> 1.78 ms, the Gram of 500,000 x 449 5.68 -> 5.70; where it
//   is recomputed, a sparse 500,000 x 449 takes 106 ms and 20,000 x 500 times the
//   identity 9.7, on the FP64 pipe alone 143 and 9.8 before).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "internal.h"

namespace ttsn {

namespace {

using namespace digits;

constexpr int T_STAGES = 2;
constexpr int DIG_BYTES = RB * T_K * 2;        // one digit of one block and stage: 4096
constexpr int BLK_BYTES = S8 * DIG_BYTES;      // 32768
constexpr int A_BYTES = 2 * BLK_BYTES, B_BYTES = BLK_BYTES, STAGE_BYTES = A_BYTES + B_BYTES;
// A stage is refilled in two groups of digit pairs (A's digit s with B's digit
// 7 - s): 0 and 1 (15 of the 36 products), then the others
constexpr int GROUPS = 2;
__host__ __device__ constexpr int group_start(int g) { return g == 0 ? 0 : g == 1 ? 2 : S8; }
constexpr int DRAIN_WARPS = 16;
constexpr int THREADS8 = 32 * (2 + DRAIN_WARPS);
constexpr int DCOLS = T_N / (DRAIN_WARPS / 4);  // columns of a drain thread: 16
constexpr unsigned TMEM_COLS = 512;
constexpr long long SPIN = 1LL << 26;
constexpr size_t SMEM8 = (size_t)T_STAGES * STAGE_BYTES + 1024 /* barriers */ + 1024 /* alignment */;

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(unsigned a, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned a, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned a) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned a, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    return ok != 0;
}
// Where a wait that ran out is reported: the caller's status word (null: none)
// and the product's flag, upon which the product is recomputed.
struct Report {
    int *status, *lost;
    __device__ __forceinline__ void timeout() const {
        if (status) atomicOr(status, DEV_TIMEOUT);
        atomicOr(lost + LOST_ALL, 1);
    }
};
// Bounded wait; false once the limit is reached (reported, the other roles told
// through *abort_flag) or another role has given up.
__device__ __forceinline__ bool bar_wait(unsigned a, unsigned parity, const Report& rep, volatile int* abort_flag,
                                         long long limit = SPIN) {
    for (long long it = 0; it < limit; ++it) {
        if (bar_try(a, parity)) return true;
        if (abort_flag && *abort_flag) return false;
        if (it > 64) __nanosleep(32);
    }
    rep.timeout();
    if (abort_flag) *abort_flag = 1;
    return false;
}
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"((unsigned long long)src), "r"(bytes), "r"(bar)
        : "memory");
}
// K-major operand descriptor: 64-byte rows, 64-byte swizzle, 8-row groups 512 bytes apart
__device__ __forceinline__ unsigned long long opdesc(unsigned addr) {
    return (unsigned long long)((addr & 0x3FFFFu) >> 4) | (unsigned long long)(16u >> 4) << 16 |
           (unsigned long long)(512u >> 4) << 32 | 1ull << 46 | 4ull << 61;
}
// kind::f16, FP32 accumulators, BF16 A and B, K-major, M = 128, N = nn
__device__ __forceinline__ unsigned mmadesc(int nn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(nn >> 3) << 17) | ((unsigned)(T_M >> 4) << 24);
}
__device__ __forceinline__ void mma8(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                     unsigned accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(unsigned addr, unsigned (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}
__device__ __forceinline__ void tmem_ld4(unsigned addr, unsigned (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

typedef unsigned long long u64;

// A product's sizes: by value, or (a captured step) read from desc = M, N, K,
// lda, ldb, ldc, when every kernel returns unless the sizes take this path.
// The kernels of one chunk see the contraction indices [k0, k0 + Kc) and the
// rows [i0, i0 + Mc) of op(A).
struct Prod {
    long M, N, K, lda, ldb, ldc;
    const int* desc;
    long k0, Kc, i0, Mc;
    int gram;
    long Mc0;  // rows of the first chunk (set by resolve): the split is chosen from it
};
__device__ __forceinline__ bool resolve(Prod& p) {
    if (p.desc) {
        p.M = p.desc[0];
        p.N = p.desc[1];
        p.K = p.desc[2];
        p.lda = p.desc[3];
        p.ldb = p.desc[4];
        p.ldc = p.desc[5];
        if (!tc8_wanted(p.M, p.N, p.K)) return false;
    }
    p.Mc0 = p.Mc < p.M ? p.Mc : p.M;
    p.Mc = p.Mc < p.M - p.i0 ? p.Mc : p.M - p.i0;
    return p.Mc > 0 && p.k0 < p.K;
}
// split_stages as one warp makes it
__device__ __forceinline__ int split_stages_warp(long M, long N, long ntiles, int nst, int unit) {
    const int lim = split_limit(M, N, nst, unit), lane = threadIdx.x & 31;
    unsigned key = 0xffffffffu;
    for (int k = lane + 1; k <= lim; k += 32)
        key = min(key, split_cost(k, ntiles, nst, unit) * 128u + (unsigned)(k - 1));
    key = __reduce_min_sync(0xffffffffu, key);
    return stages_of_split((int)(key & 127u) + 1, nst, unit);
}

// ------------------------------------------------------------------ split

// |v| as its bit pattern (ordered as the values; Inf and NaN above all).
__device__ __forceinline__ u64 mag(double v) { return (u64)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull; }
__device__ __forceinline__ u64 umax(u64 a, u64 b) { return a > b ? a : b; }
// e with every |v| <= the maximum of this pattern below 2^(e - 1); EXP_LOST (and
// flag latched) where it is Inf, NaN or outside 2^+-900.
__device__ __forceinline__ int split_exp(int ex, bool zero, int* flag) {
    if (!zero && (ex < 1023 - 900 || ex > 1023 + 900)) {
        atomicOr(flag + LOST_ROWS, 1);
        return EXP_LOST;
    }
    return zero ? 0 : ex - 1023 + 2;
}
__device__ __forceinline__ int split_exp(u64 mx, int* flag) { return split_exp((int)(mx >> 52), mx == 0, flag); }
// The same of a block of a row; its range is the row's matter.
constexpr int EXP_ZERO = -EXP_LOST;  // nothing in it but zeros (and subnormals, which have no digits)
// With it goes the number of the block's entries that have digits at all.
__device__ __forceinline__ int block_word(u64 mx, int count) {
    const int ex = (int)(mx >> 52);
    return ((ex == 0 ? EXP_ZERO : ex - 1023 + 2) << 10) | count;
}

// The biased digits of v 2^-e as one integer: F = round(|v| 2^(56 - e)) < 2^55,
// plus 64 at each of the seven lower digit positions, which makes the plain
// base-128 digits of the sum d_s + 64 (s >= 1) without a carry chain.
__device__ __forceinline__ u64 biased56(double v, int e) {
    const u64 bits = (u64)__double_as_longlong(v);
    const int ex = (int)((bits >> 52) & 0x7FF);
    u64 F = 0;
    if (ex != 0) {
        const u64 M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
        const int d = e - 4 - (ex - 1023);  // >= -2 when e bounds |v|
        if (d <= 0)
            F = M << (d < -2 ? 2 : -d);
        else if (d < 55)
            F = (M + (1ull << (d - 1))) >> d;
    }
    return F + 0x1020408102040ull;  // 64 (1 + 128 + ... + 128^6)
}
// The eight digits of two values as the packed BF16 words of the operand
// images (v0 in the low half): the biased digits u of both go into one word
// as the BF16 pair 128 + u, one packed subtraction of 192 (128 for the
// leading digit) leaves the digits exactly, and the signs are flipped in.
__device__ __forceinline__ unsigned digit_pair(u64 F0, u64 F1, int s) {  // without the signs
    const __nv_bfloat162 lead = __floats2bfloat162_rn(128.0f, 128.0f), rest = __floats2bfloat162_rn(192.0f, 192.0f);
    const unsigned u0 = (unsigned)(F0 >> (7 * (7 - s))) & 0x7Fu;
    const unsigned u1 = (unsigned)(F1 >> (7 * (7 - s))) & 0x7Fu;
    const unsigned p = 0x43004300u | u0 | (u1 << 16);
    __nv_bfloat162 x;
    memcpy(&x, &p, 4);
    const __nv_bfloat162 d = __hsub2(x, s == 0 ? lead : rest);
    unsigned r;
    memcpy(&r, &d, 4);
    return r;
}
__device__ __forceinline__ void digits8x2(double v0, double v1, int e0, int e1, unsigned (&w)[S8]) {
    const u64 F0 = biased56(v0, e0), F1 = biased56(v1, e1);
    const unsigned sg = ((unsigned)((u64)__double_as_longlong(v0) >> 48) & 0x8000u) |
                        ((unsigned)((u64)__double_as_longlong(v1) >> 32) & 0x80000000u);
#pragma unroll
    for (int s = 0; s < S8; ++s) w[s] = digit_pair(F0, F1, s) ^ sg;
}
// Byte offset of (row r, index k) in a swizzled digit tile of 64-byte rows
__device__ __forceinline__ unsigned swz(int r, int k) {
    return (unsigned)(r * 64 + (((k >> 3) ^ ((r >> 1) & 3)) << 4) + (k & 7) * 2);
}
// Operand images: for row block rb (64 rows) and stage st (32 indices) the
// eight 64 x 32 digit tiles, each in the MMA's swizzled K-major layout.
__device__ __forceinline__ unsigned char* tile_at(unsigned char* img, long rb, int nst, int st, int s) {
    return img + ((rb * nst + st) * S8 + s) * (long)DIG_BYTES;
}

// v times 2^s is at least 2^(e - 10)
__device__ __forceinline__ bool is_large(double v, int s, int e) {
    const int ex = (int)(mag(v) >> 52);
    return ex != 0 && ex + s >= e - 10 + 1023;
}
// One operand (A's rows, or B's columns) of a product: rows x K.
struct Side {
    const double* p;
    int isB, strided;  // strided: element (i, k) at k * ld + i, else at i * ld + k
    u64* mx;           // row maxima (where they are found ahead of the split)
    int* e;            // row exponents
    unsigned char* img;
    int* large;  // a guarded product: each row's entries of at least 2^(e - 10)
    int* worst;  // and the most that a row falls short of K (split_rows_kernel; spread_kernel)
    int* eb;     // K > ONE_EXP_K: the words of a row's blocks (block_word), a block after the other
    long ebs;    // rows of eb
    // the contraction index's exponents (Bond; sign 0: the smaller operand's largest
    // entries, index_max_kernel) or null, and op(A)'s sign
    const int* ks;
    int sign;
    // entries at index k count as times 2^scale (an index that one operand does not have,
    // exponent 0, at the limit: the other's entries there must not set its rows' scale)
    __device__ __forceinline__ int scale(const Prod& p, long k) const {
        const int s = min(max(ks[k] - 1023, -400), 400);
        return (sign ? (sign < 0) == (isB == 0) : (isB != 0) == (p.M > p.N)) ? -s : s;
    }
    template <bool SCALE>
    __device__ __forceinline__ u64 mag_at(const Prod& p, double v, long k) const {
        const u64 m = mag(v);
        const int ex = (int)(m >> 52);
        if (!SCALE || ex == 0 || ex == 0x7FF) return m;
        return (m & 0xFFFFFFFFFFFFFull) | (u64)min(max(ex + scale(p, k), 1), 0x7FF) << 52;
    }
    // the exponent for the digits of row i at index k, e the row's
    __device__ __forceinline__ int block(int e, long k, long i) const { return e == EXP_LOST ? e : block_exp(eb[k / BLK_K * ebs + i]); }
};
__device__ __forceinline__ void side_sizes(const Prod& p, const Side& o, long& i0, long& rows, long& rpad, long& ld) {
    i0 = o.isB ? 0 : p.i0;
    rows = o.isB ? p.N : p.Mc;
    rpad = up(rows, o.isB ? RB : T_M);
    ld = o.isB ? p.ldb : p.lda;
}

// The exponents of the contraction index where no Bond gives them: of the smaller
// operand's (by rows) largest entry at each index.
__global__ void __launch_bounds__(256) index_max_kernel(Prod p, Side a, Side b, int* out) {
    p.Mc = p.M;
    if (!resolve(p)) return;
    const bool useB = p.M > p.N;
    const long rows = useB ? p.N : p.M, ld = useB ? p.ldb : p.lda;
    const double* q = useB ? b.p : a.p;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr long SEG = 256;
    const long segs = (rows + SEG - 1) / SEG;
    auto exponent = [](double v) {  // 0 of what has none
        const int ex = (__double2hiint(v) >> 20) & 0x7FF;
        return ex == 0x7FF ? 0 : ex;
    };
    if (useB ? b.strided : a.strided) {  // a warp an index and SEG rows
        for (long t = blockIdx.x * 8L + warp; t < p.K * segs; t += gridDim.x * 8L) {
            const long k = t / segs, i1 = min(rows, (t % segs + 1) * SEG);
            int m = 0;
#pragma unroll 4
            for (long i = t % segs * SEG + lane; i < i1; i += 32) m = max(m, exponent(q[k * ld + i]));
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0 && m) atomicMax(out + k, m);
        }
        return;
    }
    __shared__ int part[8][32];
    const long kbs = (p.K + 31) / 32;
    for (long t = blockIdx.x; t < kbs * segs; t += gridDim.x) {  // a CTA 32 indices and SEG rows
        const long k = t / segs * 32 + lane, i1 = min(rows, (t % segs + 1) * SEG);
        int m = 0;
        if (k < p.K) {
#pragma unroll 4
            for (long i = t % segs * SEG + warp; i < i1; i += 8) m = max(m, exponent(q[i * ld + k]));
        }
        __syncthreads();
        part[warp][lane] = m;
        __syncthreads();
        if (warp == 0 && k < p.K) {
#pragma unroll
            for (int w = 1; w < 8; ++w) m = max(m, part[w][lane]);
            if (m) atomicMax(out + k, m);
        }
    }
}
// The same from the diagonal of the bond's Gram matrix: half its exponent.
__global__ void __launch_bounds__(256) bond_scale_kernel(int n, int rep, const double* __restrict__ G, long ldg,
                                                         const int* __restrict__ desc, int* __restrict__ out) {
    if (desc) {
        n = desc[0];
        ldg = desc[5];
    }
    for (int k = blockIdx.x * 256 + threadIdx.x; k < n; k += gridDim.x * 256) {
        const double g = G[(long)k * ldg + k];
        const int ex = __double2hiint(g) >> 20;  // negative entries: none
        const int x = ex > 0 && ex < 0x7FF ? ((ex - 1023) >> 1) + 1023 : 0;
        for (int q = 0; q < rep; ++q) out[(long)q * n + k] = x;
    }
}

// Rows with a contiguous contraction index, K <= 64 V: a warp reads a row
// once, reduces its maximum (the exponent) and writes its digits.  A lane
// holds the pairs k = 64 t + 2 lane, so a digit store covers two whole
// 64-byte tile rows.  Rows past the last are zero.
template <int V, bool SCALE>
__global__ void __launch_bounds__(256) split_rows_kernel(Prod p, Side o, int* flag) {
    if (!resolve(p)) return;
    long i0, rows, rpad, ld;
    side_sizes(p, o, i0, rows, rpad, ld);
    const int K = (int)p.K, nst = stages(K);
    if (nst > 2 * V || (V > 2 && nst <= V)) return;  // another instance's size (a captured step launches all)
    const double* A = o.p + i0 * ld;
    const int lane = threadIdx.x & 31;
    const long nw = (long)gridDim.x * 8;
    short2 sc[SCALE ? V : 1];  // the scales of this lane's indices, the same in every row
    if (SCALE) {
#pragma unroll
        for (int t = 0; t < V; ++t) {
            const int k = 64 * t + 2 * lane;
            sc[SCALE ? t : 0] = make_short2((short)(k < K ? o.scale(p, k) : 0), (short)(k + 1 < K ? o.scale(p, k + 1) : 0));
        }
    }
    for (long r = (long)blockIdx.x * 8 + (threadIdx.x >> 5); r < rpad; r += nw) {
        double v[V][2];
        u64 mx = 0;
        int top = 0;  // SCALE: the largest exponent, 0 of a zero row
        if (r < rows) {
            const double* row = A + r * ld;
#pragma unroll
            for (int t = 0; t < V; ++t) {
                const int k = 64 * t + 2 * lane;
                v[t][0] = k < K ? row[k] : 0.0;
                v[t][1] = k + 1 < K ? row[k + 1] : 0.0;
            }
            if (SCALE) {
                auto see = [&](double x, int s) {
                    const int hi = __double2hiint(x) & 0x7FFFFFFF, ex = hi >> 20;
                    int y = ex ? max(ex + s, 1) : ((hi | __double2loint(x)) ? 1 : 0);
                    if (ex == 0x7FF) y = 4095;
                    top = max(top, y);
                };
#pragma unroll
                for (int t = 0; t < V; ++t) {
                    see(v[t][0], sc[SCALE ? t : 0].x);
                    see(v[t][1], sc[SCALE ? t : 0].y);
                }
                top = __reduce_max_sync(0xffffffffu, top);
            } else {
#pragma unroll
                for (int t = 0; t < V; ++t) mx = umax(mx, umax(mag(v[t][0]), mag(v[t][1])));
#pragma unroll
                for (int q = 16; q > 0; q >>= 1) mx = umax(mx, __shfl_xor_sync(0xffffffffu, mx, q));
            }
        } else {
#pragma unroll
            for (int t = 0; t < V; ++t) v[t][0] = v[t][1] = 0.0;
        }
        const int e = SCALE ? split_exp(top, top == 0, flag) : split_exp(mx, flag);
        if (lane == 0 && r < rows) o.e[i0 + r] = e;
        if (o.worst && r < rows) {
            int c = 0;
#pragma unroll
            for (int t = 0; t < V; ++t)
                c += is_large(v[t][0], SCALE ? sc[SCALE ? t : 0].x : 0, e) + is_large(v[t][1], SCALE ? sc[SCALE ? t : 0].y : 0, e);
            c = __reduce_add_sync(0xffffffffu, c);
            const bool zero = SCALE ? top == 0 : mx == 0;
            if (lane == 0) {
                o.large[i0 + r] = zero ? K : c;
                if (!zero && e != EXP_LOST && K - c > *(volatile int*)o.worst) atomicMax(o.worst, K - c);
            }
        }
        const unsigned off = swz((int)(r & 63), 2 * (lane & 15));
#pragma unroll
        for (int t = 0; t < V; ++t) {
            const int st = 2 * t + (lane >> 4);
            if (st < nst) {
                unsigned w[S8];
                digits8x2(v[t][0], v[t][1], e - (SCALE ? sc[SCALE ? t : 0].x : 0), e - (SCALE ? sc[SCALE ? t : 0].y : 0),
                          w);
                unsigned char* q = tile_at(o.img, r >> 6, nst, st, 0) + off;
#pragma unroll
                for (int s = 0; s < S8; ++s) *reinterpret_cast<unsigned*>(q + s * DIG_BYTES) = w[s];
            }
        }
    }
}

// Longer rows in two passes: the maxima of their blocks (a warp each), then the
// digits of a chunk.
template <bool SCALE>
__global__ void __launch_bounds__(256) row_max_kernel(Prod p, Side o) {
    p.Mc = p.M;
    if (!resolve(p) || p.K <= ONE_EXP_K) return;
    const long rows = o.isB ? p.N : p.M, ld = o.isB ? p.ldb : p.lda;
    const int lane = threadIdx.x & 31;
    const long nw = (long)gridDim.x * 8;
    const long nblk = (p.K + BLK_K - 1) / BLK_K;
    for (long t = (long)blockIdx.x * 8 + (threadIdx.x >> 5); t < rows * nblk; t += nw) {
        const long r = t / nblk, kb = t % nblk, k1 = min(p.K, (kb + 1) * BLK_K);
        const double* row = o.p + r * ld;
        u64 m0 = 0, m1 = 0, m2 = 0, m3 = 0;
        int c = 0;
        auto see = [&](u64& m, long k) {
            const u64 v = o.mag_at<SCALE>(p, row[k], k);
            m = umax(m, v);
            c += (v >> 52) != 0;
        };
        long k = kb * BLK_K + lane;
        for (; k + 96 < k1; k += 128) {
            see(m0, k);
            see(m1, k + 32);
            see(m2, k + 64);
            see(m3, k + 96);
        }
        for (; k < k1; k += 32) see(m0, k);
        m0 = umax(umax(m0, m1), umax(m2, m3));
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) m0 = umax(m0, __shfl_xor_sync(0xffffffffu, m0, q));
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) {
            o.eb[kb * o.ebs + r] = block_word(m0, c);
            if (m0) atomicMax(o.mx + r, m0);
        }
    }
}
template <bool SCALE>
__global__ void __launch_bounds__(256) split_rows_long_kernel(Prod p, Side o, int* flag) {
    if (!resolve(p) || p.K <= ONE_EXP_K) return;
    long i0, rows, rpad, ld;
    side_sizes(p, o, i0, rows, rpad, ld);
    const long Kc = p.Kc < p.K - p.k0 ? p.Kc : p.K - p.k0;
    const int nst = stages(Kc);
    const double* A = o.p + i0 * ld + p.k0;
    const long total = rpad * nst * (T_K / 2);
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const int kw = (int)(t & 15);
        const long q = t >> 4;
        const int st = (int)(q % nst);
        const long r = q / nst;
        const long k = (long)st * T_K + 2 * kw;
        double v0 = 0.0, v1 = 0.0;
        int e = 0, eb = 0;
        if (r < rows) {
            e = split_exp(o.mx[i0 + r], flag);
            if (k == 0) o.e[i0 + r] = e;
            eb = o.block(e, p.k0 + k, i0 + r);
            if (k < Kc) v0 = A[r * ld + k];
            if (k + 1 < Kc) v1 = A[r * ld + k + 1];
        }
        const int s0 = SCALE && k < Kc ? o.scale(p, p.k0 + k) : 0, s1 = SCALE && k + 1 < Kc ? o.scale(p, p.k0 + k + 1) : 0;
        if (o.large) {  // 16 lanes a row, whole warps (total is a multiple of 32)
            const unsigned b0 = __ballot_sync(0xffffffffu, is_large(v0, s0, e));
            const unsigned b1 = __ballot_sync(0xffffffffu, is_large(v1, s1, e));
            const unsigned half = threadIdx.x & 16 ? 0xffff0000u : 0xffffu;
            if (kw == 0 && r < rows) atomicAdd(o.large + i0 + r, __popc(b0 & half) + __popc(b1 & half));
        }
        unsigned w[S8];
        digits8x2(v0, v1, eb - s0, eb - s1, w);
        unsigned char* d = tile_at(o.img, r >> 6, nst, st, 0) + swz((int)(r & 63), 2 * kw);
#pragma unroll
        for (int s = 0; s < S8; ++s) *reinterpret_cast<unsigned*>(d + s * DIG_BYTES) = w[s];
    }
}

// Rows that are the columns of a stored matrix (the Gram's operand): column
// maxima, then the digits of a chunk of its rows.  A thread splits 8 rows of one
// column, so that a warp reads 32 neighbouring columns of a row at a time, and
// stores 16 bytes a digit.  Bound by the latency of its loads: 8 rows fit 64
// registers, four CTAs an SM (49,152 x 449: 156 us, 3.7 TB/s; with 16 rows a
// thread, 128 registers and two CTAs 251 us, with 48 registers and spills 230).
// Of up to MAX_WARPS warps: where there are fewer CTAs than fit at once, their time is
// that of a warp's loads after one another, and 32 warps read a block of 512 rows in two
// batches of eight loads each (3,000 x 100: 20.8 -> 10.8 us); more CTAs want eight warps
// (500,000 x 449: 0.26 ms against 0.46 with 32).
constexpr int MAX_WARPS = 32;
template <bool SCALE>
__global__ void __launch_bounds__(32 * MAX_WARPS) strided_max_kernel(Prod p, Side o) {
    p.Mc = p.M;
    if (!resolve(p)) return;
    const long n = o.isB ? p.N : p.M, ld = o.isB ? p.ldb : p.lda;
    // a block of indices after the other, or one range a CTA
    const bool blocked = p.K > ONE_EXP_K;
    const long per = blocked ? BLK_K : (p.K + gridDim.y - 1) / gridDim.y;
    const int W = blockDim.x >> 5;
    __shared__ u64 part[MAX_WARPS][32];
    __shared__ int count[MAX_WARPS][32];
    for (long jb = blockIdx.x * 32L; jb < n; jb += gridDim.x * 32L) {
        const long j = jb + (threadIdx.x & 31);
        u64 top = 0;
        for (long kb = blockIdx.y; kb * per < p.K; kb += gridDim.y) {
            const long k1 = min(p.K, (kb + 1) * per);
            u64 m0 = 0, m1 = 0, m2 = 0, m3 = 0;
            int c = 0;
            auto see = [&](u64& m, double x, long k) {
                const u64 v = o.mag_at<SCALE>(p, x, k);
                m = umax(m, v);
                c += (v >> 52) != 0;
            };
            if (j < n) {
                long k = kb * per + (threadIdx.x >> 5);
                for (; k + 7 * W < k1; k += 8 * W) {
                    double x[8];
#pragma unroll
                    for (int t = 0; t < 8; ++t) x[t] = o.p[(k + W * t) * ld + j];
#pragma unroll
                    for (int t = 0; t < 8; t += 4) {
                        see(m0, x[t], k + W * t);
                        see(m1, x[t + 1], k + W * (t + 1));
                        see(m2, x[t + 2], k + W * (t + 2));
                        see(m3, x[t + 3], k + W * (t + 3));
                    }
                }
#pragma unroll 4
                for (; k < k1; k += W) see(m0, o.p[k * ld + j], k);
            }
            __syncthreads();
            part[threadIdx.x >> 5][threadIdx.x & 31] = umax(umax(m0, m1), umax(m2, m3));
            count[threadIdx.x >> 5][threadIdx.x & 31] = c;
            __syncthreads();
            if (threadIdx.x < 32 && j < n) {
                u64 m = part[0][threadIdx.x];
#pragma unroll 8
                for (int w = 1; w < W; ++w) {
                    m = umax(m, part[w][threadIdx.x]);
                    c += count[w][threadIdx.x];
                }
                if (blocked) o.eb[kb * o.ebs + j] = block_word(m, c);
                top = umax(top, m);
            }
        }
        if (threadIdx.x < 32 && j < n && top) atomicMax(o.mx + j, top);
    }
}
template <bool GUARD, bool SCALE>
__global__ void __launch_bounds__(256, 4) split_strided_kernel(Prod p, Side o, int* flag) {
    __shared__ int s_large[GUARD ? 32 : 1];
    if (!resolve(p)) return;
    long i0, rows, rpad, ld;
    side_sizes(p, o, i0, rows, rpad, ld);
    const long Kc = p.Kc < p.K - p.k0 ? p.Kc : p.K - p.k0;
    const int nst = stages(Kc);
    const double* A = o.p + i0 + p.k0 * ld;
    const bool blocked = p.K > ONE_EXP_K;
    for (long jb = blockIdx.x * 32L; jb < rpad; jb += gridDim.x * 32L) {
        const long j = jb + (threadIdx.x & 31);
        int e = 0;
        if (j < rows) {
            e = split_exp(o.mx[i0 + j], flag);
            if (blockIdx.y == 0 && threadIdx.x < 32) o.e[i0 + j] = e;
        }
        if (GUARD) {
            __syncthreads();
            if (threadIdx.x < 32) s_large[threadIdx.x] = 0;
            __syncthreads();
        }
        const long groups = (long)nst * 4;
        for (long g = (long)blockIdx.y * 8 + (threadIdx.x >> 5); g < groups; g += (long)gridDim.y * 8) {
            const long k0 = g * 8;
            u64 F[8];
            unsigned sg[4];
            const int eb = blocked && j < rows ? o.block(e, p.k0 + k0, i0 + j) : e;
#pragma unroll
            for (int r = 0; r < 8; ++r) F[r] = j < rows && k0 + r < Kc ? (u64)__double_as_longlong(__ldcs(A + (k0 + r) * ld + j)) : 0ull;
            if (GUARD) {
                int c = 0;
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    c += is_large(__longlong_as_double((long long)F[r]), SCALE && k0 + r < Kc ? o.scale(p, p.k0 + k0 + r) : 0, e);
                atomicAdd(&s_large[threadIdx.x & 31], c);
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const unsigned sign = ((unsigned)(F[r] >> 48) & 0x8000u) << (16 * (r & 1));
                sg[r >> 1] = r & 1 ? sg[r >> 1] | sign : sign;
                F[r] = biased56(__longlong_as_double((long long)F[r]),
                                eb - (SCALE && k0 + r < Kc ? o.scale(p, p.k0 + k0 + r) : 0));
            }
            unsigned char* d = tile_at(o.img, j >> 6, nst, (int)(g >> 2), 0) + swz((int)(j & 63), (int)(g & 3) * 8);
#pragma unroll
            for (int s = 0; s < S8; ++s)
                *reinterpret_cast<uint4*>(d + s * DIG_BYTES) =
                    make_uint4(digit_pair(F[0], F[1], s) ^ sg[0], digit_pair(F[2], F[3], s) ^ sg[1],
                               digit_pair(F[4], F[5], s) ^ sg[2], digit_pair(F[6], F[7], s) ^ sg[3]);
        }
        if (GUARD) {
            __syncthreads();
            if (threadIdx.x < 32 && j < rows && s_large[threadIdx.x]) atomicAdd(o.large + i0 + j, s_large[threadIdx.x]);
        }
    }
}

// *worst: the most indices of a nonzero row that are not large; zero rows count as
// large everywhere
__global__ void __launch_bounds__(256) spread_kernel(Prod p, Side o) {
    p.Mc = p.M;
    if (!resolve(p) || (!o.strided && p.K <= ONE_EXP_K)) return;  // found by the split
    const long rows = o.isB ? p.N : p.M;
    int w = 0;
    for (long r = blockIdx.x * 256L + threadIdx.x; r < rows; r += gridDim.x * 256L) {
        if (o.mx[r] == 0)
            o.large[r] = (int)p.K;
        else if (o.e[r] != EXP_LOST)
            w = max(w, (int)p.K - o.large[r]);
    }
    w = __reduce_max_sync(0xffffffffu, w);
    if ((threadIdx.x & 31) == 0 && w > *(volatile int*)o.worst) atomicMax(o.worst, w);
}

// ------------------------------------------------------------------ product

// Sums: t stands for t 2^(e - 63 - ROOM), e the sum of the rows' exponents.  |t| is
// below 2^(61 + ROOM) K, so 96 bits hold it; a thread keeps 96, planes 128.
constexpr int ROOM = 8;
__device__ __forceinline__ __int128 whole_sum(long long hi, long long lo) { return (((__int128)hi << 28) + lo) << ROOM; }
struct Sum96 {
    long long hi;
    unsigned lo;
    // + (h 2^28 + l) 2^(ROOM - r), r >= 0, rounded down
    __device__ __forceinline__ void add(long long h, long long l, int r) {
        const long long th = (l >> (32 - ROOM)) + (h << (28 + ROOM - 32));
        const unsigned tl = (unsigned)l << ROOM;
        const unsigned below = r < 32 ? __funnelshift_r(tl, (unsigned)th, r) : (unsigned)(th >> min(r - 32, 63));
        const unsigned s = lo + below;
        hi += (th >> min(r, 63)) + (s < below ? 1 : 0);
        lo = s;
    }
    __device__ __forceinline__ __int128 value() const { return ((__int128)hi << 32) + lo; }
};
__device__ __forceinline__ __int128 join(longlong2 v) { return ((__int128)v.y << 64) + (u64)v.x; }
__device__ __forceinline__ longlong2 parts(__int128 t) { return make_longlong2((long long)(u64)t, (long long)(t >> 64)); }

// t 2^(e - 63 - ROOM) rounded to nearest.
__device__ __forceinline__ double digits_value(__int128 t, int e) {
    const bool neg = t < 0;
    unsigned __int128 u = neg ? (unsigned __int128)(-t) : (unsigned __int128)t;
    u64 uh = (u64)(u >> 64), ul = (u64)u;
    if ((uh | ul) == 0) return 0.0;
    // the leading bit to bit 63 of m, what is cut off as a sticky bit
    const int z = uh ? __clzll((long long)uh) : 64 + __clzll((long long)ul);
    u <<= z;
    u64 m = (u64)(u >> 64);
    const u64 rest = (u64)u;
    int ex = e - 63 - ROOM + 127 - z;  // exponent of the leading bit
    const u64 low = (m & 0x7FF) | (rest ? 1ull : 0ull);
    m >>= 11;  // 53 bits
    if (low > 0x400 || (low == 0x400 && (m & 1))) {
        if (++m == (1ull << 53)) {
            m >>= 1;
            ++ex;
        }
    }
    if (ex < -1022 || ex > 1023) {  // beyond the normal range: ldexp's rounding
        const double v = ldexp((double)m, ex - 52);
        return neg ? -v : v;
    }
    const u64 bits = ((u64)(ex + 1023) << 52) | (m & 0xFFFFFFFFFFFFFull) | (neg ? 1ull << 63 : 0ull);
    return __longlong_as_double((long long)bits);
}

// Output tile of item t: row block (128) and column block (64); the Gram takes
// only the tiles that hold some j <= k.
__device__ __forceinline__ void tile_of(long t, int nb, bool tri, long& mb, int& kb) {
    if (!tri) {
        mb = t / nb;
        kb = (int)(t % nb);
        return;
    }
    int jt = 0;
    while (t >= nb - 2 * jt) {
        t -= nb - 2 * jt;
        ++jt;
    }
    mb = jt;
    kb = 2 * jt + (int)t;
}

// One CTA per SM walks (split of the contraction, output tile) items.  Warp 0
// copies: A's digit s and B's digit 7 - s are the pair that the MMAs of digit s
// use last, so a group of pairs is refilled for the stage after next as soon as
// the MMAs of its last digit are done (a commit per group).  Warp 1 issues: eight
// FP32 accumulators of 128 x 64 (one per level, all 512 TMEM columns); the digit
// tiles of B lie back to back, so A's digit s meets up to four of B's digits in
// one MMA of N <= 256 whose levels are neighbouring column ranges.  Sixteen warps
// drain a block's accumulators into integers (a float-to-int and a wide multiply-add
// a value, with an exponent a block also a shifted 96-bit addition an output) and, at
// an item's end, write the FP64 results while the next item's MMAs run.
//
// What bounds it: the tensor cores (72% of their cycles; 1184 clocks of MMA per
// 16 indices against 937 of operand reads and 375 of arrivals in shared memory),
// then the drains, which the MMAs wait for: TMEM holds one set of accumulators.
// The issuing thread must not be what bounds it: with a rolled loop, descriptors
// computed per MMA and a commit per digit a stage took 4600 clocks even without
// loads (tensor cores at 45%); unrolled, with descriptors that are constants from
// the stage's, about 2900.  196,608 x 512 times 512 x 512: 4.1 -> 2.6 ms; commits
// per stage 8, 4, 3, 2, 1 with the rolled loop: 3.84, 4.02, 3.94, 3.59, 3.55 ms.
template <bool BLOCKED>
__global__ void __launch_bounds__(THREADS8, 1)
tc8_kernel(Prod p, const unsigned char* __restrict__ At, const int* __restrict__ eA, const int* __restrict__ ebA,
           long ebsA, const unsigned char* __restrict__ Bt, const int* __restrict__ eB, const int* __restrict__ ebB,
           long ebsB, double alpha, double* __restrict__ C,
           longlong2* __restrict__ planes, int spc, Report rep, long long limit) {
    // every thread, before any barrier; a captured step launches both forms
    if (!resolve(p) || (p.K > ONE_EXP_K) != BLOCKED) return;
    const long M = p.Mc;
    const int N = (int)p.N;
    const int nst = stages(p.Kc < p.K - p.k0 ? p.Kc : p.K - p.k0);
    const long ntiles = tiles_of(M, N, p.gram);
    // a captured step decides the split here (from the first chunk, as the
    // reduction does)
    if (p.desc)
        spc = planes ? split_stages_warp(p.M, N, tiles_of(p.Mc0, N, p.gram), stages(p.Kc < p.K ? p.Kc : p.K),
                                         split_unit(p.K))
                     : nst;
    const bool accumulate = p.k0 > 0;
    const bool whole = planes == nullptr || (p.desc && !p.gram && p.K <= p.Kc && spc >= nst);
    extern __shared__ unsigned char raw[];
    const unsigned raw_s = smem_addr(raw);
    const unsigned pad = ((raw_s + 1023u) & ~1023u) - raw_s;
    const unsigned sb = raw_s + pad;
    u64* bars = reinterpret_cast<u64*>(raw + pad + T_STAGES * STAGE_BYTES);
    // bars: [0,1] stage full, [2 + 8 st + q] group q empty, [18] accumulators full,
    // [19] accumulators drained, [20] every MMA done
    unsigned* tmem_slot = reinterpret_cast<unsigned*>(bars + 24);
    volatile int* flags = reinterpret_cast<volatile int*>(tmem_slot + 2);  // abort, stages issued, consumed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nb = (N + T_N - 1) / T_N;
    const int ksp = (nst + spc - 1) / spc;
    const long items = ntiles * ksp;
    if ((long)blockIdx.x >= items) return;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 21; ++i)
            bar_init(smem_addr(&bars[i]), i < 2 ? (unsigned)GROUPS : (i == 19 ? (unsigned)DRAIN_WARPS : 1u));
        flags[0] = flags[1] = flags[2] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            long g = 0;
            bool stop = false;
            for (long item = blockIdx.x; item < items && !stop; item += gridDim.x) {
                long mb;
                int kb;
                tile_of(item % ntiles, nb, p.gram != 0, mb, kb);
                const int sp = (int)(item / ntiles);
                const int st1 = min(nst, (sp + 1) * spc);
                for (int it = sp * spc; it < st1 && !stop; ++it, ++g) {
                    const int st = (int)(g % T_STAGES);
                    const unsigned ph = (unsigned)(g / T_STAGES) & 1u;
                    const unsigned full = smem_addr(&bars[st]);
                    const unsigned dst = sb + (unsigned)(st * STAGE_BYTES);
                    const unsigned char* a0 = At + (2 * mb * nst + it) * (long)BLK_BYTES;
                    const unsigned char* a1 = a0 + (long)nst * BLK_BYTES;
                    const unsigned char* b0 = Bt + ((long)kb * nst + it) * BLK_BYTES;
                    for (int q = 0; q < GROUPS; ++q) {
                        if (!stop && !bar_wait(smem_addr(&bars[2 + 8 * st + q]), ph ^ 1u, rep, flags, limit)) stop = true;
                        if (stop) {  // the stage's barrier completes with what was issued
                            bar_arrive(full);
                            continue;
                        }
                        const int s0 = group_start(q), s1 = group_start(q + 1);
                        bar_expect(full, (unsigned)(3 * (s1 - s0) * DIG_BYTES));
                        for (int s = s0; s < s1; ++s) {
                            bulk_g2s(dst + s * 2 * DIG_BYTES, a0 + s * DIG_BYTES, DIG_BYTES, full);
                            bulk_g2s(dst + s * 2 * DIG_BYTES + DIG_BYTES, a1 + s * DIG_BYTES, DIG_BYTES, full);
                        }
                        bulk_g2s(dst + A_BYTES + (S8 - s1) * DIG_BYTES, b0 + (S8 - s1) * DIG_BYTES,
                                 (unsigned)((s1 - s0) * DIG_BYTES), full);
                    }
                    flags[1] = (int)(g + 1);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            long g = 0, gb = 0;
            bool stop = false;
            for (long item = blockIdx.x; item < items && !stop; item += gridDim.x) {
                const int st0 = (int)(item / ntiles) * spc, st1 = min(nst, st0 + spc);
                for (int it = st0; it < st1; ++it, ++g) {
                    const int st = (int)(g % T_STAGES);
                    const unsigned ph = (unsigned)(g / T_STAGES) & 1u;
                    const int at = BLOCKED ? it : it - st0;
                    const bool first = it == st0 || at % T_BLK == 0;
                    if (first && gb > 0) {
                        if (!bar_wait(smem_addr(&bars[19]), (unsigned)(gb - 1) & 1u, rep, flags, limit)) {
                            stop = true;
                            break;
                        }
                        fence_after();
                    }
                    if (!bar_wait(smem_addr(&bars[st]), ph, rep, flags, limit)) {
                        stop = true;
                        break;
                    }
                    flags[2] = (int)(g + 1);
                    fence_after();
                    // every MMA's descriptors are the stage's plus a constant: one
                    // thread issues 24 MMAs a stage, a few instructions each
                    const u64 ad0 = opdesc(sb + (unsigned)(st * STAGE_BYTES));
                    const unsigned acc0 = first ? 0u : 1u;
#pragma unroll
                    for (int s = 0; s < S8; ++s) {
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk) {
                            const u64 ad = ad0 + (u64)((s * 2 * DIG_BYTES + kk * 32) >> 4);
#pragma unroll
                            for (int t0 = 0; t0 < S8 - s; t0 += 4) {
                                const u64 bd = ad0 + (u64)((A_BYTES + t0 * DIG_BYTES + kk * 32) >> 4);
                                mma8(tmem + (unsigned)((s + t0) * T_N), ad, bd,
                                     mmadesc((S8 - s - t0 < 4 ? S8 - s - t0 : 4) * T_N), s == 0 && kk == 0 ? acc0 : 1u);
                            }
                        }
#pragma unroll
                        for (int q = 0; q < GROUPS; ++q)
                            if (s == group_start(q + 1) - 1) mma_commit(smem_addr(&bars[2 + 8 * st + q]));
                    }
                    if (at % T_BLK == T_BLK - 1 || it == st1 - 1) {
                        mma_commit(smem_addr(&bars[18]));
                        ++gb;
                    }
                }
            }
            mma_commit(smem_addr(&bars[20]));
            bar_wait(smem_addr(&bars[20]), 0u, rep, nullptr);
        }
    } else {
        const int q = warp & 3;  // TMEM lanes 32 q .. 32 q + 31
        const int c0 = ((warp - 2) >> 2) * DCOLS;
        long gb = 0;
        bool stop = false;
        for (long item = blockIdx.x; item < items && !stop; item += gridDim.x) {
            long mb;
            int kb;
            tile_of(item % ntiles, nb, p.gram != 0, mb, kb);
            const int sp = (int)(item / ntiles);
            const int st0 = sp * spc, st1 = min(nst, st0 + spc);
            const int b0 = BLOCKED ? st0 / T_BLK : 0, b1 = BLOCKED ? (st1 - 1) / T_BLK + 1 : (st1 - st0 + T_BLK - 1) / T_BLK;
            const long i = mb * T_M + 32 * q + lane;
            const int col0 = kb * T_N + c0;
            long long hi[BLOCKED ? 1 : DCOLS], lo[BLOCKED ? 1 : DCOLS];  // sums of levels 0-3 and 4-7
            Sum96 all[BLOCKED ? DCOLS : 1];
#pragma unroll
            for (int c = 0; c < DCOLS; ++c) {
                if (BLOCKED)
                    all[BLOCKED ? c : 0] = Sum96{0, 0u};
                else
                    hi[BLOCKED ? 0 : c] = lo[BLOCKED ? 0 : c] = 0;
            }
            for (int b = b0; b < b1; ++b, ++gb) {
                int below = 0;              // the block's exponents below the rows': of the row,
                unsigned bcol[DCOLS / 4];  // of the columns, a byte each
                if (BLOCKED) {
                    const long blk = p.k0 / BLK_K + b;
                    if (i < M) below = min(max(eA[p.i0 + i] - block_exp(ebA[blk * ebsA + p.i0 + i]), 0), 127);
#pragma unroll
                    for (int c = 0; c < DCOLS; ++c) {
                        const int v = col0 + c < N ? min(max(eB[col0 + c] - block_exp(ebB[blk * ebsB + col0 + c]), 0), 127) : 0;
                        bcol[c / 4] = c % 4 ? bcol[c / 4] | (unsigned)v << (8 * (c % 4)) : (unsigned)v;
                    }
                }
                if (!__all_sync(0xffffffffu, bar_wait(smem_addr(&bars[18]), (unsigned)gb & 1u, rep, flags, limit))) {
                    stop = true;
                    break;
                }
                fence_after();
                const unsigned ta = tmem + ((unsigned)(32 * q) << 16) + (unsigned)c0;
                if (!BLOCKED) {
#pragma unroll
                    for (int w = 0; w < S8; ++w) {
                        unsigned r[16];
                        tmem_ld16(ta + (unsigned)(w * T_N), r);
                        tmem_wait_ld();
                        const int scale = 1 << (7 * (3 - (w & 3)));
#pragma unroll
                        for (int c = 0; c < DCOLS; ++c) {
                            const long long v = (long long)__float2int_rn(__uint_as_float(r[c])) * scale;
                            if (w < 4)
                                hi[BLOCKED ? 0 : c] += v;
                            else
                                lo[BLOCKED ? 0 : c] += v;
                        }
                    }
                } else {  // a few columns at a time: every block has its shifts
#pragma unroll
                    for (int c = 0; c < DCOLS; c += 4) {
                        unsigned r[S8][4];
#pragma unroll
                        for (int w = 0; w < S8; ++w) tmem_ld4(ta + (unsigned)(w * T_N + c), r[w]);
                        tmem_wait_ld();
                        if (c + 4 == DCOLS) {  // the accumulators are read: the next block may start
                            fence_before();
                            __syncwarp();
                            if (lane == 0) bar_arrive(smem_addr(&bars[19]));
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            long long h = 0, l = 0;
#pragma unroll
                            for (int w = 0; w < S8; ++w) {
                                const long long v =
                                    (long long)__float2int_rn(__uint_as_float(r[w][u])) * (1 << (7 * (3 - (w & 3))));
                                if (w < 4)
                                    h += v;
                                else
                                    l += v;
                            }
                            all[BLOCKED ? c + u : 0].add(h, l, below + (int)((bcol[c / 4] >> (8 * u)) & 0xFFu));
                        }
                    }
                }
                if (!BLOCKED) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0) bar_arrive(smem_addr(&bars[19]));
                }
            }
            if (stop) break;
            auto sum = [&](int c) {
                return BLOCKED ? all[BLOCKED ? c : 0].value() : whole_sum(hi[BLOCKED ? 0 : c], lo[BLOCKED ? 0 : c]);
            };
            if (i < M && !flags[0]) {
                if (whole) {
                    const int ea = eA[p.i0 + i];
                    double* out = C + (p.i0 + i) * p.ldc;
#pragma unroll
                    for (int c = 0; c < DCOLS; ++c)
                        if (col0 + c < N) {
                            const double v = digits_value(sum(c), ea + eB[col0 + c]);
                            out[col0 + c] = alpha == 1.0 ? v : alpha * v;
                        }
                } else {
                    longlong2* out = planes + ((long)sp * p.M + p.i0 + i) * N;
#pragma unroll
                    for (int c = 0; c < DCOLS; ++c)
                        if (col0 + c < N) {
                            const __int128 v = sum(c);
                            out[col0 + c] = parts(accumulate ? v + join(out[col0 + c]) : v);
                        }
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {  // after an abort: copies in flight land before the CTA exits
        for (long g = flags[2]; g < flags[1]; ++g)
            bar_wait(smem_addr(&bars[g % T_STAGES]), (unsigned)(g / T_STAGES) & 1u, rep, nullptr);
    }
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// The splits' integer sums added and rounded once: C (the Gram: both halves
// from the entries j <= k that are held).
__global__ void __launch_bounds__(256)
tc8_reduce_kernel(Prod p, const longlong2* __restrict__ planes, const int* __restrict__ eA,
                  const int* __restrict__ eB, int spc, double alpha, double* __restrict__ C) {
    if (!resolve(p) || !planes) return;  // without planes tc8_kernel has written C
    const int nst = stages(p.Kc < p.K ? p.Kc : p.K);
    if (p.desc) {
        spc = split_stages_warp(p.M, p.N, tiles_of(p.Mc0, p.N, p.gram), nst, split_unit(p.K));
        if (!p.gram && p.K <= p.Kc && spc >= nst) return;  // written whole
    }
    const int ksp = (nst + spc - 1) / spc;
    const long total = p.M * p.N;
    for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
        const long i = t / p.N, j = t % p.N;
        const long src = p.gram && j < i ? j * p.N + i : t;
        // planes are read once, a Gram's twice; the first with the exponents (20,000 x 100
        // x 300, two splits: 157 -> 152 us a call)
        const int e = eA[i] + eB[j];
        __int128 v;
        if (p.gram) {
            v = join(planes[src]);
            for (int z = 1; z < ksp; ++z) v += join(planes[z * total + src]);
        } else {
            v = join(__ldcs(planes + src));
            for (int z = 1; z < ksp; ++z) v += join(__ldcs(planes + z * total + src));
        }
        const double x = digits_value(v, e);
        C[i * p.ldc + j] = alpha == 1.0 ? x : alpha * x;
    }
}

unsigned blocks_for(long work, long cap) { return (unsigned)std::max<long>(1, std::min<long>(work, cap)); }

// desc: a captured product of sizes up to M, N, K (then lda, ldb, ldc are the
// descriptor's).
tt_status run(cudaStream_t s, bool ta, bool tb, long M, long N, long K, double alpha, const double* A, long lda,
              const double* B, long ldb, double* C, long ldc, DevBuf& scratch, int* status_dev, bool gram,
              const int* desc, bool guard, const Bond* bond, Lost* lost, long long limit = SPIN) {
    const Plan q = make_plan(M, N, K, gram, desc != nullptr);
    // slack to bring the base to a 1024-byte boundary (a pool may give 256)
    TT_TRY(scratch.ensure((q.bytes() + 1024 + 7) / 8, s));
    unsigned char* base = reinterpret_cast<unsigned char*>(((uintptr_t)scratch.p + 1023) & ~(uintptr_t)1023);
    int* flag = reinterpret_cast<int*>(base);
    u64* mx = reinterpret_cast<u64*>(base + 256);
    const long nrows = gram ? M : M + N;
    const bool entries = bond && bond->entries;
    const bool scale = !gram && !guard && (!bond || bond->s || entries), find = scale && !(bond && bond->s);
    int* kx = reinterpret_cast<int*>(mx + nrows);  // of its own, found below
    const int* ks = !scale ? nullptr : find ? kx : bond->s;
    const int sign = bond ? bond->sign : 0;
    int* ex = kx + (gram ? 0 : K);
    const bool count = guard || entries;
    int* large = count ? ex + nrows : nullptr;
    int* worst = count ? flag + LOST_WORST : nullptr;
    int* eb = ex + 2 * nrows;  // behind the counts
    Side a{A, 0, ta ? 1 : 0, mx, ex, base + q.head + q.imgB, large, worst, eb, M, ks, sign};
    Side b{B, 1, tb ? 0 : 1, mx + M, ex + M, base + q.head, count ? large + M : nullptr, count ? worst + 1 : nullptr,
           eb + (K + BLK_K - 1) / BLK_K * M, N, ks, sign};
    if (gram) {
        a.img = base + q.head;
        b = a;
    }
    longlong2* planes = q.part ? reinterpret_cast<longlong2*>(base + q.head + q.imgA + q.imgB) : nullptr;
    Prod p{M, N, K, lda, ldb, ldc, desc, 0, q.Kc, 0, q.Mc, gram ? 1 : 0, q.Mc};
    int dev = 0, sms = 152;
    TT_CUDA_TRY(cudaGetDevice(&dev));
    TT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    TT_TRY(ensure_max_dynamic_smem((const void*)tc8_kernel<false>));
    TT_TRY(ensure_max_dynamic_smem((const void*)tc8_kernel<true>));
    // the flag and, where atomics find them, the maxima and counts start at zero
    const size_t maxima_bytes = a.strided || b.strided || K > ONE_EXP_K || find ? 8 * (size_t)nrows : 0;
    TT_CUDA_TRY(cudaMemsetAsync(flag, 0, 256 + maxima_bytes + (find ? 4 * (size_t)K : 0), s));
    if (count) TT_CUDA_TRY(cudaMemsetAsync(large, 0, 4 * (size_t)nrows, s));
    const bool fusable = K <= ONE_EXP_K;  // a captured step launches both forms when K may be longer
    auto maxima = [&](const Side& o) {
        const long rows = o.isB ? N : M;
        if (o.strided) {
            note_launch();
            const dim3 grid(blocks_for((rows + 31) / 32, 4096), blocks_for(K / (fusable ? 256 : BLK_K), 512));
            const int threads = 32 * (grid.x * grid.y < 304 ? MAX_WARPS : 8);
            (scale ? strided_max_kernel<true> : strided_max_kernel<false>)<<<grid, threads, 0, s>>>(p, o);
        } else if (!fusable) {
            note_launch();
            const unsigned grid = blocks_for((rows * ((K + BLK_K - 1) / BLK_K) + 7) / 8, 152L * 64);
            (scale ? row_max_kernel<true> : row_max_kernel<false>)<<<grid, 256, 0, s>>>(p, o);
        }
    };
    auto split = [&](const Side& o) {
        const long rows = o.isB ? N : std::min(q.Mc, M - p.i0), rpad = up(rows, T_M);
        const int nst = stages(q.Kc);
        if (o.strided) {
            const dim3 grid(blocks_for((rpad + 31) / 32, 4096), blocks_for(((long)nst * 2 + 7) / 8, 2048));
            note_launch();
            (entries ? split_strided_kernel<true, true>
             : guard ? split_strided_kernel<true, false>
             : scale ? split_strided_kernel<false, true>
                     : split_strided_kernel<false, false>)<<<grid, 256, 0, s>>>(p, o, flag);
            return;
        }
        if (!fusable) {
            note_launch();
            const unsigned long_grid = blocks_for((rpad * nst * 16 + 255) / 256, 152L * 64);
            (scale ? split_rows_long_kernel<true> : split_rows_long_kernel<false>)<<<long_grid, 256, 0, s>>>(p, o, flag);
            if (!desc) return;
        }
        const unsigned grid = blocks_for((rpad + 7) / 8, 152L * 64);
        const int need = std::min(nst, ONE_EXP_K / T_K);
        // by value one instance, the smallest that holds the row; a captured
        // product launches each that a size up to its capacity may need
        if (desc ? true : need <= 4) {
            note_launch();
            (scale ? split_rows_kernel<2, true> : split_rows_kernel<2, false>)<<<grid, 256, 0, s>>>(p, o, flag);
        }
        if (need > 4 && (desc || need <= 8)) {
            note_launch();
            (scale ? split_rows_kernel<4, true> : split_rows_kernel<4, false>)<<<grid, 256, 0, s>>>(p, o, flag);
        }
        if (need > 8 && (desc || need <= 16)) {
            note_launch();
            (scale ? split_rows_kernel<8, true> : split_rows_kernel<8, false>)<<<grid, 256, 0, s>>>(p, o, flag);
        }
        if (need > 16) {
            note_launch();
            (scale ? split_rows_kernel<16, true> : split_rows_kernel<16, false>)<<<grid, 256, 0, s>>>(p, o, flag);
        }
    };
    const int nst0 = stages(q.Kc);
    const int spc = split_stages(M, N, tiles_of(q.Mc, N, gram), nst0, split_unit(K));
    const bool direct = !desc && !gram && q.Kc >= K && spc >= nst0;
    if (find) {
        const long segs = (std::min(M, N) + 255) / 256;
        note_launch();
        index_max_kernel<<<blocks_for(std::max((K + 31) / 32, K / 8) * segs, 152L * 8), 256, 0, s>>>(p, a, b, kx);
    }
    maxima(a);
    if (!gram) maxima(b);
    for (p.k0 = 0; p.k0 < K; p.k0 += q.Kc) {
        if (!gram) {
            p.i0 = 0;
            p.Mc = M;
            split(b);
        }
        for (p.i0 = 0; p.i0 < M; p.i0 += q.Mc) {
            p.Mc = q.Mc;
            split(a);
            const long items = tiles_of(std::min(q.Mc, M - p.i0), N, gram) * ((nst0 + spc - 1) / spc);
            auto product = [&](auto kernel) {
                note_launch();
                kernel<<<desc ? sms : (int)std::min<long>(items, sms), THREADS8, SMEM8, s>>>(
                    p, a.img, a.e, a.eb, a.ebs, b.img, b.e, b.eb, b.ebs, alpha, C, direct ? nullptr : planes, spc,
                    Report{status_dev, flag}, limit);
            };
            if (fusable || (desc && p.k0 == 0)) product(tc8_kernel<false>);
            if (!fusable) product(tc8_kernel<true>);
            TT_CUDA_TRY(cudaGetLastError());
        }
    }
    p.k0 = p.i0 = 0;
    p.Mc = q.Mc;
    if (!direct) {
        note_launch();
        tc8_reduce_kernel<<<blocks_for((M * N + 255) / 256, 152L * 16), 256, 0, s>>>(p, planes, a.e, b.e, spc, alpha, C);
    }
    if (count) {
        auto spread = [&](const Side& o) {
            const long rows = o.isB ? N : M;
            if (!o.strided && fusable) return;  // found by the split
            note_launch();
            spread_kernel<<<blocks_for((rows + 255) / 256, 152), 256, 0, s>>>(p, o);
        };
        spread(a);
        if (!gram) spread(b);
    }
    TT_CUDA_TRY(cudaGetLastError());
    *lost = Lost{flag, a.e, b.e, guard ? 1 : entries ? 2 : 0, gram ? 1 : 0, reinterpret_cast<double*>(base + q.head), mx, a.eb, a.ebs,
                 gram && !guard ? reinterpret_cast<float*>(ex + nrows) : nullptr, a.large, b.large};
    return TT_OK;
}

}  // namespace

size_t tc8_scratch_doubles(long M, long N, long K, bool gram, bool captured) {
    return (make_plan(M, N, K, gram, captured).bytes() + 1024 + 7) / 8;
}

size_t tc8_reserve_doubles(long M, long N, long K, bool gram) {
    return (reserve_bytes(M, N, K, gram) + 1024 + 7) / 8;
}

void bond_scale(cudaStream_t s, int n, int rep, const double* G, long ldg, int* out, const int* desc) {
    if (n <= 0) return;
    note_launch();
    bond_scale_kernel<<<blocks_for((n + 255) / 256, 152), 256, 0, s>>>(n, rep, G, ldg, desc, out);
}

size_t tc8_head_doubles(long M, long N, long K, bool gram) { return (head_bytes(M, N, K, gram) + 1024 + 7) / 8; }

tt_status tc8_gemm(cudaStream_t s, bool ta, bool tb, long M, long N, long K, double alpha, const double* A, long lda,
                   const double* B, long ldb, double* C, long ldc, DevBuf& scratch, int* status_dev, bool guard,
                   const Bond* bond, Lost* lost, bool probe) {
    return run(s, ta, tb, M, N, K, alpha, A, lda, B, ldb, C, ldc, scratch, status_dev, false, nullptr, guard, bond, lost,
               probe ? 0 : SPIN);
}

tt_status tc8_gram(cudaStream_t s, long m, long n, const double* A, long lda, double* G, long ldg, DevBuf& scratch,
                   int* status_dev, bool guard, Lost* lost) {
    return run(s, true, false, n, n, m, 1.0, A, lda, A, lda, G, ldg, scratch, status_dev, true, nullptr, guard, nullptr, lost);
}

tt_status tc8_dyn(cudaStream_t s, bool ta, bool tb, const int* desc, long Mcap, long Ncap, long Kcap, double alpha,
                  const double* A, const double* B, double* C, DevBuf& scratch, int* status_dev, bool gram,
                  const Bond* bond, Lost* lost) {
    return run(s, ta, tb, Mcap, Ncap, Kcap, alpha, A, 0, B, 0, C, 0, scratch, status_dev, gram, desc, false, bond, lost);
}

}  // namespace ttsn
