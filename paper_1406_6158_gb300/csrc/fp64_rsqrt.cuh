// fp64_rsqrt.cuh -- r^2 + eps^2 and x^-1/2, x^-3/2 and x^1/2 of FP64 numbers in
// fixed point.
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
// pair), 27.0 with this one (7), 16.2 with r^2 + eps^2 in fixed point too (4).
// One kick-drift-kick step at N = 30011: far forces 2.36 ms (16 instructions a
// pair), 1.46 (10), 1.07 (7); near forces 0.68, 0.48, 0.46, and 0.37 ms with the
// K argument's r^2 and its comparison with R2^2 in fixed point too.
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

__device__ __forceinline__ RsqrtSeed seed_of(uint64_t A, int k)
{
    RsqrtSeed s;
    s.A = A;
    s.k = k;
    const uint32_t y = (uint32_t)(rsqrtf((float)(uint32_t)(A >> 32)) * 549755813888.0f);   // 2^39; exact
    s.Q = ((uint64_t)y * y) << 15;
    s.Y = y << 7;
    s.e = (int64_t)((1ull << 61) - __umul64hi(s.A, s.Q));
    const int e = (int)(s.e >> 20);
    s.e2 = (int64_t)e * e;
    return s;
}

__device__ __forceinline__ uint64_t significand(double x)
{
    return (uint64_t)(((uint32_t)__double2hiint(x) & 0xfffffu) | 0x100000u) << 32 | (uint32_t)__double2loint(x);
}

// eps^2 = S 2^-60 4^(E - 1023), S 2^-60 in [1, 4) (S = E = 0: none)
struct Eps2Fixed {
    uint64_t S;
    int E;
    double eps2;
};

__device__ __forceinline__ Eps2Fixed eps2_fixed(double eps2)
{
    const int E = __double2hiint(eps2) >> 20, p = (E + 1) & 1;
    if (E == 0) return Eps2Fixed{0ull, 0, eps2};
    return Eps2Fixed{significand(eps2) << (8 + p), ((E - 1023 - p) >> 1) + 1023, eps2};
}

// v^2 2^60 / 4^(Em - 1023), for v of exponent E <= Em (0, and what is below 2^-63 of the largest, give 0)
__device__ __forceinline__ uint64_t square_fixed(double v, int E, int Em)
{
    const uint64_t m = (significand(v) << 11) >> min(Em - E, 63);
    const uint32_t h = (uint32_t)(m >> 32), l = (uint32_t)m;
    return ((uint64_t)h * h + (((uint64_t)h * l) >> 31)) >> 2;
}

// A number as A 2^-62 4^k, A 2^-62 in [1, 4); larger numbers have a larger k, or the same k and a larger A.
struct Fixed {
    uint64_t A;
    int k;
};

// x >= 0, below everything for zero and subnormals, above everything for infinity
__device__ __forceinline__ Fixed to_fixed(double x)
{
    const int E = __double2hiint(x) >> 20, p = (E + 1) & 1;
    if (E == 0) return Fixed{0ull, -2000};
    return Fixed{significand(x) << (10 + p), (E - 1023 - p) >> 1};
}

// dx^2 + dy^2 + dz^2 + eps^2, summed in units of 2^-60 of the largest term's power of four (4 units of truncation at
// most, 2^-58 of the sum, where three multiply-adds in FP64 round by up to 2^-53 each). False outside 2^-640 to 2^640,
// where a result could leave the range of normal numbers (and for NaN and all zero): the callers take sqrt and division.
__device__ __forceinline__ bool r2_fixed(double dx, double dy, double dz, const Eps2Fixed &eps, Fixed &r2)
{
    const int Ex = (__double2hiint(dx) >> 20) & 0x7ff, Ey = (__double2hiint(dy) >> 20) & 0x7ff,
              Ez = (__double2hiint(dz) >> 20) & 0x7ff;
    const int Em = max(max(Ex, Ey), max(Ez, eps.E));
    if ((unsigned)(Em - 703) > 638u) return false;   // the largest from 2^-320 to below 2^319
    const uint64_t S = square_fixed(dx, Ex, Em) + square_fixed(dy, Ey, Em) + square_fixed(dz, Ez, Em) +
                       (eps.S >> min(2 * (Em - eps.E), 63));   // in [2^60, 2^64)
    const bool up = S >> 62;
    r2 = Fixed{up ? S : S << 2, Em - (up ? 1022 : 1023)};
    return true;
}
__device__ __forceinline__ bool r2_seed(double dx, double dy, double dz, const Eps2Fixed &eps, RsqrtSeed &s)
{
    Fixed r2;
    if (!r2_fixed(dx, dy, dz, eps, r2)) return false;
    s = seed_of(r2.A, r2.k);
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

// m (r^2 + eps^2)^-3/2; 0 for r = eps = 0 (a sink met by itself without softening)
__device__ __forceinline__ double mass_over_r3(double m, double dx, double dy, double dz, const Eps2Fixed &eps)
{
    RsqrtSeed s;
    if (!r2_seed(dx, dy, dz, eps, s)) {
        const double x = __fma_rn(dx, dx, __fma_rn(dy, dy, __fma_rn(dz, dz, eps.eps2)));
        const double ri = x > 0.0 ? 1.0 / sqrt(x) : 0.0;
        return m * ri * ri * ri;
    }
    const uint64_t c = (uint64_t)((1ll << 61) + s.e + (s.e >> 1) + ((15 * s.e2) >> 24)) << 2;
    const uint64_t v = __umul64hi(mul_hi(s.Y, s.Q) << 1, c);   // f^-3/2 2^62, in [2^59, 2^62]
    const int z = __clzll((long long)v);
    const int64_t b = (int64_t)((((v << z) >> 10) + 1) >> 1);   // 53 bits with the leading one
    return __dmul_rn(m, __longlong_as_double(((int64_t)(1023 - z - 3 * s.k) << 52) + b));
}

// sqrt(x) = x x^-1/2
__device__ __forceinline__ double sqrt_fixed(const Fixed &x)
{
    const RsqrtSeed s = seed_of(x.A, x.k);
    return from_fixed(__umul64hi(s.A, rsqrt_fixed(s) << 1), s.k);
}

// w + m (r^2 + eps^2)^-1/2
__device__ __forceinline__ double add_mass_over_r(double w, double m, double dx, double dy, double dz,
                                                  const Eps2Fixed &eps)
{
    RsqrtSeed s;
    if (!r2_seed(dx, dy, dz, eps, s))
        return w + m / sqrt(__fma_rn(dx, dx, __fma_rn(dy, dy, __fma_rn(dz, dz, eps.eps2))));
    return __fma_rn(m, from_fixed(rsqrt_fixed(s), -1 - s.k), w);
}

}  // namespace hy
