"""Integer division and square root (csrc/intfp.h) against the hardware's, bit for bit.

The header compiles as host code; its FP32 estimates are shifted by up to two
units in the last place, more than the device's approximations are off.
"""

import os
import shutil
import subprocess

import pytest

SRC = r"""
#include "intfp.h"
#include <cstdio>
#include <random>
using namespace ttsn::intfp;
int main() {
    std::mt19937_64 g(5);
    long bad = 0;
    auto same = [&](double got, double want) { bad += bits(got) != bits(want) && !(got != got && want != want); };
    auto mant = [&](long i) -> uint64_t {  // random, next to 1 and 2, short, and one bit off a power of two
        const uint64_t r = g() & MANT;
        switch (i % 5) {
            case 0: return r;
            case 1: return r & 7;
            case 2: return MANT - (r & 7);
            case 3: return (r >> 40) << 40;
            default: return ((1ull << (r % 52)) + (r >> 51) - 1) & MANT;
        }
    };
    for (long i = 0; i < 2000000; ++i) {
        const int span = i % 3 ? 2000 : 1;
        const uint64_t ea = 1023 + g() % span - span / 2, eb = 1023 + g() % span - span / 2;
        const double a = from_bits((g() & 1) << 63 | ea << 52 | mant(i));
        const double b = from_bits((g() & 1) << 63 | eb << 52 | mant(i / 5));
        same(div(a, b), a / b);
        same(div(a * b, b), a * b / b);
        same(root(std::fabs(a)), std::sqrt(std::fabs(a)));
        same(root(from_bits(bits(b * b) + i % 5 - 2)), std::sqrt(from_bits(bits(b * b) + i % 5 - 2)));
    }
    const double sp[] = {0.0, -0.0, 5e-324, 1e-310, 2.3e-308, 1.0, -1.0, 1.7e308, INFINITY, -INFINITY, NAN};
    for (double a : sp) {
        for (double b : sp) same(div(a, b), a / b);
        same(root(a), std::sqrt(a));
    }
    std::printf("%ld\n", bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
@pytest.mark.parametrize("ulps", [-2, 0, 2])
def test_quotients_and_roots_are_the_hardware_s(tmp_path, ulps):
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_18056_gb300", "csrc")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", csrc, "-DTTSN_INTFP_ULPS=%d" % ulps, "-o", str(exe), str(src)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
