// root_box.cuh -- root cubes of the systems and the start of the sample sort,
// run by whichever kernel last touches the positions before a build: the drift
// of a single system, else k_box.
#pragma once

#include "hy_internal.cuh"

namespace hy {

// order-preserving map of doubles to unsigned integers (for atomic min/max)
__device__ __forceinline__ unsigned long long ord_dbl(double v)
{
    unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double unord_dbl(unsigned long long u)
{
    return __longlong_as_double((long long)((u >> 63) ? (u & 0x7fffffffffffffffull) : ~u));
}

struct BoxArgs {
    unsigned long long *bmin, *bmax;   // per system and axis, as ord_dbl images; empty before the first block
    int nbk, S;                        // buckets of the sample sort (0: radix sort), systems
    const int64_t *off;
    const SSys *ss;
    const uint64_t *key;               // the last build's sorted keys
    uint32_t *cnt, *bsys, *flag;
    unsigned *ticket;                  // 0 between launches
    unsigned *trip;                    // 0 between launches: a particle of a list-reusing drift has moved too far
    SysBox *box;
};

inline BoxArgs box_args(hybrid_ctx *c)
{
    BoxArgs b;
    b.bmin = (unsigned long long *)c->boxmin.p;
    b.bmax = (unsigned long long *)c->boxmax.p;
    b.nbk = c->sort_fallback ? 0 : c->nbk;
    b.S = c->S;
    b.off = (const int64_t *)c->off_dev.p;
    b.ss = (const SSys *)c->ss_sys.p;
    b.key = (const uint64_t *)c->keys[0].p;
    b.cnt = (uint32_t *)c->ss_cnt.p;
    b.bsys = (uint32_t *)c->ss_bsys.p;
    b.flag = (uint32_t *)c->ss_flag.p;
    b.ticket = (unsigned *)((unsigned long long *)c->counter.p + 14);
    b.trip = b.ticket + 1;
    b.box = (SysBox *)c->box.p;
    return b;
}

// The sample sort's bucket counts cleared, the buckets' systems (of a batch), its overflow flag reset, and whether its
// splitters (the last build's keys at every SS_BUCKET-th position) are in order. Every thread of the grid.
__device__ __forceinline__ void begin_sort(const BoxArgs &a)
{
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gtid == 0) {
        a.flag[0] = 0u;
        a.cnt[a.nbk] = 0u;
    }
    for (int b = gtid; b < a.nbk; b += gridDim.x * blockDim.x) {
        a.cnt[b] = 0u;
        int s = 0;
        if (a.S > 1) {   // system of bucket b
            int hi = a.S;
            while (hi - s > 1) {
                const int mid = (s + hi) >> 1;
                if (a.ss[mid].bbase <= b) s = mid;
                else hi = mid;
            }
            a.bsys[b] = (uint32_t)s;
        }
        const SSys y = a.ss[s];
        const int j = b - y.bbase;
        const uint64_t *k = a.key + a.off[s] + (int64_t)j * SS_BUCKET;
        if (j >= 1 && j + 1 < y.nb && k[SS_BUCKET] < k[0]) a.flag[1] = 1u;
    }
}

// Bounds of a thread's particles: exact, and no FP64 instruction.
struct Bounds {
    unsigned long long v[6] = {~0ull, ~0ull, ~0ull, 0ull, 0ull, 0ull};

    __device__ __forceinline__ void add(double x, double y, double z)
    {
        const unsigned long long p0 = ord_dbl(x), p1 = ord_dbl(y), p2 = ord_dbl(z);
        v[0] = min(v[0], p0);
        v[1] = min(v[1], p1);
        v[2] = min(v[2], p2);
        v[3] = max(v[3], p0);
        v[4] = max(v[4], p1);
        v[5] = max(v[5], p2);
    }
    // the block's bounds (256 threads, all of one system) into the system's
    __device__ __forceinline__ void reduce_block(const BoxArgs &b, int sys)
    {
        __shared__ unsigned long long sh[6][8];
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int j = 0; j < 3; ++j) v[j] = min(v[j], __shfl_xor_sync(0xffffffffu, v[j], o));
#pragma unroll
            for (int j = 3; j < 6; ++j) v[j] = max(v[j], __shfl_xor_sync(0xffffffffu, v[j], o));
        }
        if (lane == 0)
#pragma unroll
            for (int j = 0; j < 6; ++j) sh[j][w] = v[j];
        __syncthreads();
        if (threadIdx.x < 6) {
            const int j = threadIdx.x;
            unsigned long long r = sh[j][0];
            for (int k = 1; k < 8; ++k) r = (j < 3) ? min(r, sh[j][k]) : max(r, sh[j][k]);
            if (j < 3) atomicMin(&b.bmin[3 * sys + j], r);
            else atomicMax(&b.bmax[3 * sys + j - 3], r);
        }
        __syncthreads();
    }
};

// Root cube: per-axis minimum lo; side L = smallest power of two >= the
// largest extent (1 when all particles coincide); scale = 2^21 / L.
__device__ __forceinline__ SysBox make_box(const BoxArgs &a, int s)
{
    double lo[3], ext = 0.0;
    for (int d = 0; d < 3; ++d) {   // values other blocks made
        lo[d] = unord_dbl(__ldcg(a.bmin + 3 * s + d));
        const double e = __dsub_rn(unord_dbl(__ldcg(a.bmax + 3 * s + d)), lo[d]);
        if (e > ext) ext = e;
    }
    double L = 1.0;
    if (ext > 0.0) {
        int e2;
        const double f = frexp(ext, &e2);
        L = (f == 0.5) ? ext : ldexp(1.0, e2);
    }
    SysBox b;
    b.lo[0] = lo[0];
    b.lo[1] = lo[1];
    b.lo[2] = lo[2];
    b.L = L;
    b.scale = ldexp(1.0, LEVELS) / L;   // ratio of powers of two: exact
    b.u = ldexp(L, -20);
    b.inv_u = ldexp(1.0, 20) / L;
    b.uf = (float)b.u;
    b.inv_uf = (float)b.inv_u;
    return b;
}

// The last block to get here (a ticket, no waiting) makes the cubes.
__device__ __forceinline__ void finish_boxes(const BoxArgs &a)
{
    __shared__ bool last;
    __threadfence();   // this block's bounds are visible before its ticket
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int s = threadIdx.x; s < a.S; s += blockDim.x) a.box[s] = make_box(a, s);
    if (threadIdx.x == 0) *a.ticket = 0u;
}

}  // namespace hy
