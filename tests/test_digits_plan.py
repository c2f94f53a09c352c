"""The scratch of a digit product (csrc/digits_plan.h) holds what its kernels write.

A captured product's scratch is laid out from the capacities, but its kernels
choose the split of the contraction from the sizes they find: every smaller
size's images and split planes must fit, and a product without planes must not
split.  The header compiles as host code.
"""

import os
import shutil
import subprocess

import pytest

SRC = r"""
#include "digits_plan.h"
#include <cstdio>
#include <initializer_list>
using namespace ttsn;
using namespace ttsn::digits;
static long bad = 0, split_under_unsplit = 0;
static void fail(const char* what, long Mc, long Nc, long Kc, long M, long N, long K) {
    if (++bad <= 10) std::printf("%s: %ld %ld %ld up to %ld %ld %ld\n", what, M, N, K, Mc, Nc, Kc);
}
// sizes M, N, K in the scratch of `q`, which was laid out for Mc, Nc, Kc
static void check(const Plan& q, bool captured, bool gram, long Mc, long Nc, long Kc, long M, long N, long K) {
    const long chunk = least(q.Kc, K), rows = least(q.Mc, M);
    const int nst = stages(chunk);
    const int spc = split_stages(M, N, tiles_of(rows, N, gram), nst, split_unit(K)), ks = (nst + spc - 1) / spc;
    const bool whole = !gram && K <= q.Kc && ks == 1;
    if (!whole && q.part < 16ull * M * N * ks) fail(q.part ? "planes too small" : "no planes", Mc, Nc, Kc, M, N, K);
    if (q.part && captured && ks > 1 && stages(q.Kc) >= 8 && split_limit(Mc, Nc, stages(q.Kc), split_unit(Kc)) == 1) ++split_under_unsplit;
    const size_t stage = 2ull * S8 * T_K;
    if (up(N, gram ? T_M : RB) * nst * stage > q.imgB) fail("image B", Mc, Nc, Kc, M, N, K);
    if (!gram && up(rows, T_M) * nst * stage > q.imgA) fail("image A", Mc, Nc, Kc, M, N, K);
    const size_t side = gram ? M : M + N;
    if (q.head < 256 + 16 * side + (gram ? 0 : 4 * K) + (K > ONE_EXP_K ? 4 * side * ((K + BLK_K - 1) / BLK_K) : 0)) fail("head", Mc, Nc, Kc, M, N, K);
    // a contraction that goes in chunks is cut between exact blocks
    if (K > q.Kc && (q.Kc % BLK_K || spc % T_BLK)) fail("cut", Mc, Nc, Kc, M, N, K);
    if (q.Kc < Kc && q.Kc % (T_K * T_BLK)) fail("chunk", Mc, Nc, Kc, M, N, K);
}
int main() {
    // captured steps: cells, ordinates and caps; every rank below the cap
    const long grids[][2] = {{32 * 32, 5}, {96 * 90, 5}, {128 * 128, 5}, {200 * 200, 5}, {256 * 256, 5}, {500 * 500, 5},
                             {64 * 64 * 64, 7}, {128 * 128 * 128, 7}};
    const long angles[][2] = {{16, 32}, {32, 64}};
    for (auto& g : grids)
        for (auto& a : angles)
            for (long cap : {24L, 64L, 96L, 128L}) {
                const long nc = g[0], t = g[1], nt = a[0], np = a[1];
                const long c1 = least(cap, nt * np), c2 = least(cap, np), G1 = t * c1 + 1, G2 = t * c2 + 1;
                const Plan gramL = make_plan(G1, G1, nc, true, true), upd = make_plan(nc, c1, G1, false, true);
                const Plan bwd = make_plan(G1 * nt, G2, G2, false, true), gb = make_plan(G1, G1, nt * G2, false, true);
                const Plan next = make_plan(c1, nt * G2, G1, false, true), sq = make_plan(G1, G1, G1, false, true);
                const Plan upd1 = make_plan(c1 * nt, c2, G2, false, true), gram1 = make_plan(G2, G2, c1 * nt, true, true);
                for (long r1 = 1; r1 <= c1; ++r1) {
                    const long R1 = t * r1 + 1;
                    auto one = [&](const Plan& q, bool gram, long Mc, long Nc, long Kc, long M, long N, long K) {
                        if (!tc8_wanted(M, N, K)) return;
                        check(q, true, gram, Mc, Nc, Kc, M, N, K);
                        const Plan own = make_plan(M, N, K, gram, false);
                        check(own, false, gram, M, N, K, M, N, K);
                        if (own.bytes() > reserve_bytes(Mc, Nc, Kc, gram)) fail("reservation", Mc, Nc, Kc, M, N, K);
                    };
                    one(gramL, true, G1, G1, nc, R1, R1, nc);
                    for (long r : {1L, 7L, r1 / 2, r1, (r1 + c1) / 2, c1})
                        if (r > 0) one(upd, false, nc, c1, G1, nc, r, R1);
                    for (long r2 = 1; r2 <= c2; r2 += r1 % 5 == 0 ? 1 : 13) {
                        const long R2 = t * r2 + 1;
                        one(bwd, false, G1 * nt, G2, G2, R1 * nt, R2, R2);
                        one(gb, false, G1, G1, nt * G2, R1, R1, nt * R2);
                        one(next, false, c1, nt * G2, G1, r1, nt * R2, R1);
                        one(upd1, false, c1 * nt, c2, G2, r1 * nt, r2, R2);
                        one(gram1, true, G2, G2, c1 * nt, R2, R2, r1 * nt);
                    }
                    for (long k = 1; k <= R1; k += 37) one(sq, false, G1, G1, G1, R1, k, R1);
                }
            }
    if (split_under_unsplit == 0) ++bad, std::printf("no size splits where its capacity does not\n");
    // long contractions, cut along K, and wide outputs
    const long odd[][3] = {{17, 33, 40000000}, {64, 64, 1 << 26}, {897, 897, 2097152}, {1100, 1100, 500001},
                           {2000000, 400, 600}, {40, 100000, 16384}, {5000, 5000, 5000}, {33, 16, 40001}};
    for (auto& s : odd)
        for (int gram = 0; gram < 2; ++gram) {
            const long M = gram ? s[1] : s[0];
            check(make_plan(M, s[1], s[2], gram, false), false, gram, M, s[1], s[2], M, s[1], s[2]);
            const Plan cap = make_plan(M, s[1], s[2], gram, true);
            for (long f = 1; f <= 64; f *= 2)
                for (long h = 1; h <= 64; h *= 2) {
                    const long n = most(1, s[1] / f), k = most(1, s[2] / h);
                    for (long m : {M, most(1, M / f), most(1, M / 3)}) {
                        check(cap, true, gram, M, s[1], s[2], gram ? n : m, n, k);
                        if (make_plan(gram ? n : m, n, k, gram, false).bytes() > reserve_bytes(M, s[1], s[2], gram))
                            fail("reservation", M, s[1], s[2], m, n, k);
                    }
                }
        }
    // a small problem's products (32^2 cells, 8 x 16 ordinates, cap 128) hold no planes
    // that their contraction cannot be split into
    if (reserve_bytes(641, 641, 1024, true) > (80u << 20)) fail("small Gram", 641, 641, 1024, 641, 641, 1024);
    std::printf("%ld\n", bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_every_smaller_size_fits_the_scratch_of_its_capacity(tmp_path):
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_18056_gb300", "csrc")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", csrc, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
