// fp64_rsqrt.cuh -- 1/sqrt of FP64 numbers with few FP64 instructions.
//
// The FP64 pipe of this GPU retires 2 lanes per SM and clock (one warp
// instruction per 16 clocks) against 128 lanes of FP32 and integer work, and
// sqrt() followed by a division costs about 20 FP64 instructions. Here the
// seed y0 comes from an FP32 rsqrt of the argument scaled to [1, 4) (integer
// moves only), and one third-order step in FP64 finishes it: with
// e = 1 - x y0^2 (y0 has 24 bits, so y0^2 is exact and e is rounded once),
//   x^-1/2 = y0 (1 + e/2 + 3 e^2/8 + ..),  x^-3/2 = y0^3 (1 + 3 e/2 + 15 e^2/8 + ..);
// |e| < 2^-21, so the dropped terms are below 2^-60.
#pragma once

#include <cstdint>

namespace hy {

// Seed for x >= 0: true with y0 and e when x lies between 2^-640 and 2^640, where
// neither y0^2 nor y0^3 leaves the range of normal numbers; the callers below
// take sqrt and division for the rest.
__device__ __forceinline__ bool rsqrt_seed(double x, double &y0, double &q, double &e)
{
    const int hi = __double2hiint(x);
    const int E = hi >> 20;
    if ((unsigned)(E - 383) > 1280u) return false;   // 0, tiny, huge, negative, infinity, NaN
    const int p = (E - 1023) & 1;                    // x = f 4^k with f in [1, 4), k = (E - 1023 - p) / 2
    const int k = (E - 1023 - p) >> 1;
    const float f = __int_as_float(((127 + p) << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)__double2loint(x) >> 29));
    const int b = __float_as_int(rsqrtf(f));         // in (1/2, 1]
    y0 = __hiloint2double((((b >> 23) + 896 - k) << 20) | ((b & 0x7fffff) >> 3), b << 29);
    q = __dmul_rn(y0, y0);
    e = __fma_rn(-x, q, 1.0);
    return true;
}

// m x^-3/2; 0 for x = 0 (a sink met by itself without softening)
__device__ __forceinline__ double mass_over_r3(double m, double x)
{
    double y0, q, e;
    if (!rsqrt_seed(x, y0, q, e)) {
        const double ri = x > 0.0 ? 1.0 / sqrt(x) : 0.0;
        return m * ri * ri * ri;
    }
    const double c = __dmul_rn(__dmul_rn(m, y0), q);
    const double s = __dmul_rn(e, __fma_rn(e, 1.875, 1.5));
    return __fma_rn(c, s, c);
}

// sqrt(x) = x x^-1/2 for x >= 0
__device__ __forceinline__ double sqrt_seeded(double x)
{
    double y0, q, e;
    if (!rsqrt_seed(x, y0, q, e)) return x == 0.0 ? 0.0 : sqrt(x);
    const double r = __dmul_rn(x, y0);
    const double s = __dmul_rn(e, __fma_rn(e, 0.375, 0.5));
    return __fma_rn(r, s, r);
}

// w + m x^-1/2
__device__ __forceinline__ double add_mass_over_r(double w, double m, double x)
{
    double y0, q, e;
    if (!rsqrt_seed(x, y0, q, e)) return w + m / sqrt(x);
    const double t = __dmul_rn(m, y0);
    const double s = __dmul_rn(e, __fma_rn(e, 0.375, 0.5));
    return __dadd_rn(w, __fma_rn(t, s, t));
}

}  // namespace hy
