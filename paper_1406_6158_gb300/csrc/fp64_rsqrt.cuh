// fp64_rsqrt.cuh -- x^-1/2, x^-3/2 and x^1/2 of FP64 numbers in fixed point.
//
// The FP64 pipe of this GPU retires 2 lanes per SM and clock (one warp
// instruction per 16 clocks) against 64 and more of integer work, so a pair's
// time is its count of FP64 instructions: sqrt() and a division cost about 20,
// an FP32 seed with a third-order FP64 step 6 (x^-1/2) or 8 (x^-3/2), this none.
// x = f 4^k with f in [1, 4); the seed y (25 bits) is the FP32 rsqrt of f, and
// with e = 1 - f y^2 (|e| < 1.4 2^-21 as rsqrtf errs by at most 2 units),
//   f^-1/2 = y (1 + e/2 + 3 e^2/8 + ..),  f^-3/2 = y^3 (1 + 3 e/2 + 15 e^2/8 + ..);
// the dropped terms are below 2^-60. Every product is the high half of a 64-bit
// one, and the result is rounded once: at most 0.52 units in the last place
// (against an exact root, over seeds off by 2 units either way), where the
// FP64 step rounded 3 times.
// Energy of 65536 particles: 51.3 ms with the FP64 step (13 instructions a
// pair), 27.0 with this one (7). One kick-drift-kick step at N = 30011: far
// forces 2.36 ms (16 instructions a pair), 1.46 (10).
#pragma once

#include <cstdint>

namespace hy {

struct RsqrtSeed {
    uint64_t A;      // f 2^62
    uint64_t Q;      // y^2 2^63
    uint32_t Y;      // y 2^31
    int64_t e, e2;   // e 2^61, e^2 2^82
    int k;
};

// For x between 2^-640 and 2^640, where none of the results leaves the range of normal numbers; false for the rest
// (0, tiny, huge, negative, infinity, NaN), for which the callers below take sqrt and division.
__device__ __forceinline__ bool rsqrt_seed(double x, RsqrtSeed &s)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int E = (int)hi >> 20;
    if ((unsigned)(E - 383) > 1280u) return false;
    const int p = (E + 1) & 1;
    s.k = (E - 1023 - p) >> 1;
    const float f = __uint_as_float(((127u + p) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const uint32_t y = (uint32_t)(rsqrtf(f) * 16777216.0f);   // exact
    s.A = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << (10 + p);
    s.Q = ((uint64_t)y * y) << 15;
    s.Y = y << 7;
    s.e = (int64_t)((1ull << 61) - __umul64hi(s.A, s.Q));
    const int e = (int)(s.e >> 20);
    s.e2 = (int64_t)e * e;
    return true;
}

// high half of (a 2^32) b
__device__ __forceinline__ uint64_t mul_hi(uint32_t a, uint64_t b)
{
    return (uint64_t)a * (uint32_t)(b >> 32) + (((uint64_t)a * (uint32_t)b) >> 32);
}

// f^-1/2 2^62, in [2^61, 2^62]
__device__ __forceinline__ uint64_t rsqrt_fixed(const RsqrtSeed &s)
{
    return mul_hi(s.Y, (uint64_t)((1ll << 61) + (s.e >> 1) + ((3 * s.e2) >> 24)) << 2);
}

// v 2^-61 in [1, 2] times 2^E, rounded (a carry moves into the exponent)
__device__ __forceinline__ double from_fixed(uint64_t v, int E)
{
    return __longlong_as_double(((int64_t)(1023 + E) << 52) + (int64_t)((v - (1ull << 61) + 256) >> 9));
}

// m x^-3/2; 0 for x = 0 (a sink met by itself without softening)
__device__ __forceinline__ double mass_over_r3(double m, double x)
{
    RsqrtSeed s;
    if (!rsqrt_seed(x, s)) {
        const double ri = x > 0.0 ? 1.0 / sqrt(x) : 0.0;
        return m * ri * ri * ri;
    }
    const uint64_t c = (uint64_t)((1ll << 61) + s.e + (s.e >> 1) + ((15 * s.e2) >> 24)) << 2;
    const uint64_t v = __umul64hi(mul_hi(s.Y, s.Q) << 1, c);   // f^-3/2 2^62, in [2^59, 2^62]
    const int z = __clzll((long long)v);
    const int64_t b = (int64_t)((((v << z) >> 10) + 1) >> 1);   // 53 bits with the leading one
    return __dmul_rn(m, __longlong_as_double(((int64_t)(1023 - z - 3 * s.k) << 52) + b));
}

// sqrt(x) = x x^-1/2 for x >= 0
__device__ __forceinline__ double sqrt_seeded(double x)
{
    RsqrtSeed s;
    if (!rsqrt_seed(x, s)) return x == 0.0 ? 0.0 : sqrt(x);
    return from_fixed(__umul64hi(s.A, rsqrt_fixed(s) << 1), s.k);
}

// w + m x^-1/2
__device__ __forceinline__ double add_mass_over_r(double w, double m, double x)
{
    RsqrtSeed s;
    if (!rsqrt_seed(x, s)) return w + m / sqrt(x);
    return __fma_rn(m, from_fixed(rsqrt_fixed(s), -1 - s.k), w);
}

}  // namespace hy
