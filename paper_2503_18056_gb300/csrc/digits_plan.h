// How a digit product (digits.cu) is cut, and the scratch it takes.  Plain
// integer rules shared by the host, which lays the scratch out, and by the
// kernels of a captured step, which cut a product from sizes that only the
// device knows; the header compiles as host code too.
#pragma once
#include <cstddef>
#include <cstdint>

#ifndef TTSN_HD
#ifdef __CUDACC__
#define TTSN_HD __host__ __device__ __forceinline__
#else
#define TTSN_HD inline
#endif
#endif

namespace ttsn {

// The sizes for which digits.cu is taken: below 16M terms (32 us of the FP64 pipe)
// the five or six launches cost more than they save; a contraction under 64
// would not be rounded less often than the FP64 sum it replaces; the 64-bit
// sums hold 2^26 indices.
TTSN_HD bool tc8_wanted(long M, long N, long K) {
    return K >= 64 && K <= (1L << 26) && M >= 32 && N >= 16 && N <= (1L << 20) && M * N <= (1L << 40) &&
           (N <= 16384 || K <= 16384) && M * N >= (16000000L + K - 1) / K;
}

namespace digits {

constexpr int S8 = 8;
constexpr int T_M = 128, T_N = 64, T_K = 32;  // output tile; contraction indices of a stage
constexpr int T_BLK = 16;                     // stages of an exact block (512 indices)
constexpr int RB = 64;                        // rows of an image block
// A contraction of up to ONE_EXP_K indices has one power of two a row, a longer
// one an own for each BLK_K of them.
constexpr int BLK_K = T_K * T_BLK, ONE_EXP_K = 1024;
// Digit images of one pass over an operand; a longer operand goes in chunks.  A
// chunk costs its launches and a last wave: with images of 2^26, 2^27, 2^28, 2^29
// and 2^30 bytes the Gram of 500,000 x 449 took 10.3, 9.1, 8.5, 8.4 and 8.6 ms and
// 200,000 x 577 times 577 x 96 3.0, 2.6, 2.1, 2.1 and 2.5 (before the present
// issue loop and split), although only the smaller ones stay in the 129 MB L2.
constexpr long IMG_LIMIT = 1L << 28;

TTSN_HD long up(long x, long m) { return (x + m - 1) / m * m; }
TTSN_HD long least(long a, long b) { return a < b ? a : b; }
TTSN_HD long most(long a, long b) { return a > b ? a : b; }
TTSN_HD int stages(long Kc) { return (int)((Kc + T_K - 1) / T_K); }
TTSN_HD long tiles_of(long M, long N, int gram) {
    const long nb = (N + T_N - 1) / T_N;
    if (!gram) return (M + T_M - 1) / T_M * nb;
    const long h = (nb + 1) / 2;  // rows of 128: nb, nb - 2, ... tiles
    return h * nb - h * (h - 1);
}

// Splits of a chunk's contraction: stages per split.  The time of a launch is
// about its waves of one CTA per SM times the stages of a split and one more
// for an item's end; a plane costs its write and its read in the reduction.
// A split has at least four stages, and the planes at most PLANE_ELEMS entries.
// A contraction that may go in chunks is split between exact blocks, so that the
// blocks' sums, and with them the result's bits, do not depend on the chunks
// (unit: stages that stay together).
constexpr long PLANE_ELEMS = 1L << 23;
// Whole blocks go badly into 64 parts: up to 80 of them (a Gram of 100,000 x 100, two
// tiles: 66 splits of three blocks instead of 49 of four; of 30,000 x 60, one tile: 59 of
// one block).
constexpr int MAX_SPLITS = 64, MAX_BLOCK_SPLITS = 80;
constexpr long CHUNK_MIN = 16384;  // no shorter contraction goes in chunks
TTSN_HD int split_unit(long K) { return K > CHUNK_MIN ? T_BLK : 1; }
TTSN_HD long most_splits(int nst, int unit) {
    return unit > 1 ? least((nst + unit - 1) / unit, MAX_BLOCK_SPLITS) : least(nst / 4, MAX_SPLITS);
}
TTSN_HD int split_limit(long M, long N, int nst, int unit) {
    const long k = least(PLANE_ELEMS / (M * N), most_splits(nst, unit));
    return k < 1 ? 1 : (int)k;
}
TTSN_HD int stages_of_split(int k, int nst, int unit) { return (int)up((nst + k - 1) / k, unit); }
TTSN_HD unsigned split_cost(int k, long ntiles, int nst, int unit) {
    const int spc = stages_of_split(k, nst, unit), kk = (nst + spc - 1) / spc;
    const long waves = (ntiles * kk + 151) / 152;
    const long c = waves * (spc + 1) * 64 + kk;
    return c > 0x01ffffffL ? 0x01ffffffu : (unsigned)c;  // 25 bits (split_stages_warp)
}
TTSN_HD int split_stages(long M, long N, long ntiles, int nst, int unit) {
    const int lim = split_limit(M, N, nst, unit);
    int best = 1;
    unsigned cost = split_cost(1, ntiles, nst, unit);
    for (int k = 2; k <= lim; ++k) {
        const unsigned c = split_cost(k, ntiles, nst, unit);
        if (c < cost) {
            cost = c;
            best = k;
        }
    }
    return stages_of_split(best, nst, unit);
}

// Chunks and scratch of a product.  A captured product (captured) has these
// sizes or any smaller ones, and its kernels choose the split from the sizes
// they find: a smaller output may split where the capacity would not, so the
// planes have the entries of every smaller size's splits.
struct Plan {
    long Kc, Mc;
    size_t head, imgA, imgB, part;  // bytes: flags, maxima and exponents; images; planes (0: none)
    size_t bytes() const { return head + imgA + imgB + part; }
};
// Flags; per row its largest entry, exponent and count of large entries, and
// the exponents of its blocks; the exponents of the contraction index.
inline size_t head_bytes(long M, long N, long K, bool gram) {
    const long rows = gram ? M : M + N;
    return (size_t)up(256 + 16 * rows + (gram ? 0 : 4 * K) + (K > ONE_EXP_K ? 4 * rows * ((K + BLK_K - 1) / BLK_K) : 0) + 64, 1024);
}
inline Plan make_plan(long M, long N, long K, bool gram, bool captured) {
    Plan p;
    const long Np = up(N, gram ? T_M : RB);
    // images of about IMG_LIMIT bytes each: a long contraction is cut along K
    // (for an operand of up to 1024 rows), a tall A along its rows
    const long wide = most(up(least(M, 1024L), T_M), Np);
    const long kmax = most(CHUNK_MIN, IMG_LIMIT / (2 * S8 * wide) / (T_K * T_BLK) * (T_K * T_BLK));
    p.Kc = K <= kmax ? K : up((K + (K + kmax - 1) / kmax - 1) / ((K + kmax - 1) / kmax), T_K * T_BLK);
    const int nst = stages(p.Kc);
    p.Mc = gram ? M : least(M, most((long)T_M, IMG_LIMIT / (2L * S8 * nst * T_K) / T_M * T_M));
    const bool sums = gram || p.Kc < K;  // planes although there is one split
    long elems = sums ? M * N : 0;
    if (captured) {
        const long splits = most(most_splits(nst, 1), K > CHUNK_MIN ? most_splits(nst, T_BLK) : 1);
        if (splits > 1) elems = most(elems, least(M * N * splits, PLANE_ELEMS));
    } else {
        const int spc = split_stages(M, N, tiles_of(p.Mc, N, gram), nst, split_unit(K));
        if (spc < nst) elems = M * N * ((nst + spc - 1) / spc);
    }
    p.head = head_bytes(M, N, K, gram);
    p.imgB = (size_t)(Np * nst * T_K * 2 * S8);
    p.imgA = gram ? 0 : (size_t)(up(p.Mc, T_M) * nst * T_K * 2 * S8);
    p.part = 16 * (size_t)elems;
    return p;
}

// Bytes that hold the scratch of every product of sizes up to these: a smaller
// operand goes in fewer or longer chunks and may split more often, so no size's
// own plan bounds the others'.
inline size_t reserve_bytes(long M, long N, long K, bool gram) {
    const long Np = up(N, gram ? T_M : RB), Kp = up(K, T_K), row = 2 * S8;
    const long imgB = least(Np * Kp, most(IMG_LIMIT / row, CHUNK_MIN * Np)) * row;
    const long imgA = gram ? 0 : least(up(M, T_M) * Kp, IMG_LIMIT / row) * row;
    const long splits = most(most_splits(stages(K), 1), K > CHUNK_MIN ? most_splits(stages(K), T_BLK) : 1);
    long elems = gram || K > CHUNK_MIN ? M * N : 0;
    if (splits > 1) elems = most(elems, least(M * N * splits, PLANE_ELEMS));
    return head_bytes(M, N, K, gram) + (size_t)(imgA + imgB + 16 * elems);
}

}  // namespace digits
}  // namespace ttsn
