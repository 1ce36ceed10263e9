// energy_pairs.cuh -- softened energies of one system by direct FP64 summation
// (the total-energy check of Sec. IV-A), shared by the context call and the
// allocation-free call.
//
// The FP64 pipe bounds it (2 lanes per SM and clock), so each pair is taken
// once (W = -G sum_{j < i} m_i m_j / sqrt(r^2 + eps^2)) with 4 FP64
// instructions (r^2 and rsqrt in fixed point, fp64_rsqrt.cuh). Work item = EN_ROW sinks (one
// per thread) against EN_COL sources in shared memory, from the lower triangle
// of the pair matrix; items go round robin to the blocks, which keep their
// sums in registers and write one partial each, so the result does not depend
// on timing. At n = 65536: 16.2 ms (13.6 ms at the full FP64 rate), against 239
// ms with every pair taken from both sides by sqrt and division.
#pragma once

#include <cstdint>

#include "fp64_rsqrt.cuh"

namespace hy {

constexpr int EN_ROW = 256, EN_COL = 64;
constexpr int EN_BLOCKS_PER_SM = 8;
constexpr int EN_PER_ROW = EN_ROW / EN_COL;

struct alignas(32) EnergySrc {
    double x, y, z, m;
};

struct EnergyArgs {
    int64_t n;
    const double *x, *y, *z, *vx, *vy, *vz, *m;
    double G, eps2;
};

__host__ __device__ __forceinline__ int64_t energy_items(int64_t n)
{
    const int64_t rows = (n + EN_ROW - 1) / EN_ROW;
    return EN_PER_ROW * (rows * (rows + 1) / 2);
}

// The sums of this block (EN_ROW threads) to out[0] (kinetic), out[1] (potential).
__device__ __forceinline__ void energy_block(const EnergyArgs &a, double *out)
{
    __shared__ EnergySrc tile[EN_COL];
    __shared__ double red[2][EN_ROW / 32];
    const int64_t items = energy_items(a.n);
    const Eps2Fixed eps = eps2_fixed(a.eps2);
    double T = 0.0, W = 0.0;
    for (int64_t t = blockIdx.x; t < items; t += gridDim.x) {
        // row I: the largest with EN_PER_ROW I (I + 1) / 2 <= t (FP32 estimate, then exact)
        const int64_t p = t / EN_PER_ROW;
        int64_t I = (int64_t)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
        while (I * (I + 1) / 2 > p) --I;
        while ((I + 1) * (I + 2) / 2 <= p) ++I;
        const int64_t i0 = I * EN_ROW, j0 = (t - EN_PER_ROW * (I * (I + 1) / 2)) * EN_COL;
        const int64_t i = i0 + threadIdx.x;
        const bool ok = i < a.n;
        __syncthreads();   // the last item's sources are used
        if (threadIdx.x < EN_COL && j0 + threadIdx.x < a.n) {
            const int64_t j = j0 + threadIdx.x;
            tile[threadIdx.x] = EnergySrc{a.x[j], a.y[j], a.z[j], a.m[j]};
        }
        __syncthreads();
        const int64_t ii = ok ? i : 0;
        const double xi = a.x[ii], yi = a.y[ii], zi = a.z[ii], mi = a.m[ii];
        if (j0 == 0 && ok) {
            const double v0 = a.vx[i], v1 = a.vy[i], v2 = a.vz[i];
            T = __fma_rn(__dmul_rn(0.5, mi), __fma_rn(v0, v0, __fma_rn(v1, v1, __dmul_rn(v2, v2))), T);
        }
        // sources j < i of this thread's sink: all of them away from the diagonal
        const int64_t left = i - j0;
        const int lim = !ok || left <= 0 ? 0 : (int)(left < EN_COL ? left : EN_COL);
        const int nt = (int)(a.n - j0 < EN_COL ? a.n - j0 : EN_COL);
        double Wi = 0.0;
        for (int k = 0; k < nt; ++k) {
            if (k >= lim) continue;
            const EnergySrc q = tile[k];
            const double dx = __dsub_rn(q.x, xi), dy = __dsub_rn(q.y, yi), dz = __dsub_rn(q.z, zi);
            Wi = add_mass_over_r(Wi, q.m, dx, dy, dz, eps);
        }
        if (lim > 0) W = __fma_rn(mi, Wi, W);
    }
    W *= -a.G;
    for (int o = 16; o > 0; o >>= 1) {
        T += __shfl_xor_sync(0xffffffffu, T, o);
        W += __shfl_xor_sync(0xffffffffu, W, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = T;
        red[1][threadIdx.x >> 5] = W;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double tT = 0.0, tW = 0.0;
        for (int k = 0; k < EN_ROW / 32; ++k) {
            tT += red[0][k];
            tW += red[1][k];
        }
        out[0] = tT;
        out[1] = tW;
    }
}

// One block of EN_ROW threads: the totals of nb block sums, in a fixed order.
__device__ __forceinline__ void energy_total(int nb, const double *part, double *out)
{
    __shared__ double red[2][EN_ROW];
    double T = 0.0, W = 0.0;
    for (int b = threadIdx.x; b < nb; b += EN_ROW) {
        T += part[2 * b];
        W += part[2 * b + 1];
    }
    red[0][threadIdx.x] = T;
    red[1][threadIdx.x] = W;
    __syncthreads();
    for (int s = EN_ROW / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = red[0][0];
        out[1] = red[1][0];
    }
}

}  // namespace hy
