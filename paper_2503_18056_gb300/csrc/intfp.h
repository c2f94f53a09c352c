// FP64 division and square root in 32-bit and 64-bit integer arithmetic, rounded
// to nearest even: the operators' results bit for bit, in the latency of integer
// instructions.
//
// On GB300 an FP64 instruction holds its warp for 64 clocks, and a division or a
// square root is a chain of them (about 580 and 610 clocks); an integer multiply
// takes about 5.  A kernel whose serial chain has divisions in it (one rotation
// angle a pair and round, one pivot a column) takes its quotients here.
//
// Both are digit recurrences with an exact remainder: an FP32 estimate of the
// reciprocal (of the divisor, of the root), scaled down so that it never exceeds
// the true one, gives 12 to 20 bits of the result a step from the remainder's
// leading 32 bits; the remainder is then formed exactly (it is small and known to
// be nonnegative, so its low 64 bits say it all).  The last step leaves the floor of
// the result with two or three bits below the last place, after at most one
// correction; no quotient or root of normal numbers lies halfway between two
// doubles, so those bits decide the rounding.  Zeros, subnormals, infinities,
// NaN and results near the ends of the range go to the operators.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define TTSN_HD __host__ __device__ __forceinline__
#else
#define TTSN_HD inline
#endif

namespace ttsn {
namespace intfp {

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ uint64_t bits(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double from_bits(uint64_t u) { return __longlong_as_double((long long)u); }
__device__ __forceinline__ uint32_t fbits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ float from_fbits(uint32_t u) { return __uint_as_float(u); }
__device__ __forceinline__ uint32_t mulhi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
// relative errors at most 2^-23 (one ulp) and 2^-22.9
__device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
#else
inline uint64_t bits(double x) { uint64_t u; std::memcpy(&u, &x, 8); return u; }
inline double from_bits(uint64_t u) { double x; std::memcpy(&x, &u, 8); return x; }
inline uint32_t fbits(float x) { uint32_t u; std::memcpy(&u, &x, 4); return u; }
inline float from_fbits(uint32_t u) { float x; std::memcpy(&x, &u, 4); return x; }
inline uint32_t mulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
#ifndef TTSN_INTFP_ULPS
#define TTSN_INTFP_ULPS 0  // a host build may shift the estimates, to show that their error does not matter
#endif
inline float rcp(float x) { return from_fbits(fbits(1.0f / x) + (uint32_t)(TTSN_INTFP_ULPS)); }
inline float rsqrt(float x) { return from_fbits(fbits((float)(1.0 / std::sqrt((double)x))) + (uint32_t)(TTSN_INTFP_ULPS)); }
#endif

constexpr uint64_t MANT = (1ull << 52) - 1, ONE = 1ull << 52;

// a / b
TTSN_HD double div(double a, double b) {
    const uint64_t ua = bits(a), ub = bits(b);
    const int ea = (int)(ua >> 52) & 0x7FF, eb = (int)(ub >> 52) & 0x7FF;
    const int e = ea - eb + 1023;
    if ((unsigned)(ea - 1) >= 2046u || (unsigned)(eb - 1) >= 2046u || (unsigned)(e - 2) >= 2044u) return a / b;
    const uint64_t ma = (ua & MANT) | ONE, mb = (ub & MANT) | ONE;
    // x in (1, 2], not below the divisor's significand: t in [0.5, 1) is below
    // its reciprocal by at most 2^-20 of it
    const float x = from_fbits(0x3F800001u + ((uint32_t)(ub >> 29) & 0x7FFFFFu));
    float t = rcp(x) * (1.0f - 0x1p-21f);
    t = t > 0.5f ? t : 0.5f;
    const uint32_t u = fbits(t) << 8 | 0x80000000u;  // 2^32 t
    // quotient in (1/2, 2): 20, 20 and 15 bits below the point
    const uint32_t q1 = mulhi((uint32_t)(ma >> 21), u) >> 11;
    const uint64_t r1 = (ma << 20) - q1 * mb;  // [0, 4 mb), as r2
    const uint32_t q2 = mulhi((uint32_t)(r1 >> 23), u) >> 9;
    const uint64_t r2 = (r1 << 20) - q2 * mb;
    const uint32_t q3 = mulhi((uint32_t)(r2 >> 23), u) >> 14;
    const uint64_t r3 = (r2 << 15) - q3 * mb;  // [0, 2 mb)
    const uint64_t q = ((uint64_t)q1 << 35) + ((uint64_t)q2 << 15) + q3 + (r3 >= mb ? 1 : 0);
    const int hi = (int)(q >> 55);  // quotient at least 1
    const uint64_t m = (q + (hi ? 4 : 2)) >> (2 + hi);
    return from_bits(((ua ^ ub) & (1ull << 63)) | (((uint64_t)(e - 2 + hi) << 52) + m));
}

// sqrt(a)
TTSN_HD double root(double a) {
    const uint64_t ua = bits(a);
    if (ua - ONE >= (0x7FFull << 52) - ONE) return std::sqrt(a);  // not a positive normal number
    const int e = (int)(ua >> 52) - 1023, odd = e & 1;
    const uint64_t m = ((ua & MANT) | ONE) << odd;  // [2^52, 2^54)
    const float x = from_fbits((uint32_t)(127 + odd) << 23 | ((uint32_t)(ua >> 29) & 0x7FFFFFu));
    const float r = rsqrt(x);
    // s in [1, 2), below the root by at most 2^-20 of it
    float s = x * r * (1.0f - 0x1p-21f);
    s = s > 1.0f ? s : 1.0f;
    // 2^31 / root, low by 2^-20 to 2^-18.7 of it: a step's second-order term (2^-21) stays covered
    const uint32_t u = (fbits(fmaf(r, 0.5f - 0x1p-20f, 1.0f)) & 0x7FFFFFu) << 9;
    // integer part of the root of 4^j m: 26 bits, then 16 and 12 more
    const uint32_t s0 = ((fbits(s) & 0x7FFFFFu) | 0x800000u) << 3;
    const uint64_t r0 = m - (uint64_t)s0 * s0;  // [0, 2^35)
    const uint32_t d1 = mulhi((uint32_t)(r0 >> 3), u) >> 7;
    const uint64_t s1 = ((uint64_t)s0 << 16) + d1;
    const uint64_t r1 = (r0 << 32) - d1 * (((uint64_t)s0 << 17) + d1);  // [0, 2^48.5)
    const uint32_t d2 = mulhi((uint32_t)(r1 >> 17), u) >> 13;
    uint64_t s2 = (s1 << 12) + d2;
    const uint64_t r2 = (r1 << 24) - d2 * ((s1 << 13) + d2);  // [0, 4 s2)
    s2 += r2 > 2 * s2 ? 1 : 0;
    return from_bits(((uint64_t)((e >> 1) + 1022) << 52) + ((s2 + 2) >> 2));
}

}  // namespace intfp
}  // namespace ttsn
