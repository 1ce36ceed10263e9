// pair.cu -- pair kernels of the soft and hard forces (Eq. 2 split by Eq. 7-10).
//
// The walk gives every sink group three lists:
//   cells and far particles: K = 0 for every pair (the walk's R2 + b_max
//     test), so they only add F to the soft force ("far" kernel);
//   near particles: the only pairs where K can be non-zero; one pass adds
//     F (1 - K) to the soft force and F K to the hard force ("near" kernel,
//     k_near).
//
// FP32 form. Work item = (group, run of at most item_len consecutive entries
// of one of the group's lists), written by the walk and pulled from a global
// counter. Near kernel: one block per work item, see k_near and, for the items
// of groups well inside R2, near_dense. Far kernel: one
// warp per work item; sources are staged, 64 at a time, into the
// warp's shared-memory tile relative to the group's reference point (the hi
// part of its first sink: on the hi grid, so hi - c is exact), as {x, y, z, m}
// or in the expanded form of body_exp2; the gathers run
// ahead of their use (see the staging ring). A group of n sinks uses
// lpc = ceil(n / KS) lanes per copy with KS sinks per lane in registers, and
// copies = 32 / lpc copies of the group split the sources (source j goes to
// copy j mod copies) and are added at the end. When that
// leaves many lanes idle (e.g. 72 sinks, KS = 4: 18 lanes, one copy), the
// sinks are taken in rounds whose lanes per copy are a power of two (64
// sinks on 2 copies of 16 lanes, then 8 sinks on 16 copies of 2 lanes):
// each round streams the item's sources again, but no lane idles. A group
// with one chunk stores its sums; a group with several adds them atomically
// into zeroed outputs.
// rsqrtf runs on the CUDA cores: the pair sum is not a dense contraction.
//
// FP64 form (the plain form): plain FP64 differences; see k_pair_f64.
#include "hy_internal.cuh"

#include "fp64_rsqrt.cuh"

namespace hy {

namespace {

constexpr int PAIR_THREADS = 128;
constexpr int FAR_SPLIT_PCT = 75;   // far kernel: a round below this fill of its sink slots is split (see below)
constexpr int PAIR_WARPS = PAIR_THREADS / 32;
constexpr int NEAR_MIN_BLOCKS = 8;  // near kernel: resident blocks of PAIR_THREADS per SM (64 registers, see k_near)
constexpr int TILE = 64;

struct PairArgs {
    const int64_t *ngroups;
    const uint32_t *gfirst, *gsys;
    const SysParams *sp;
    const uint64_t *off;    // [3 * ng + 1] list offsets: cells, far particles, near particles
    const uint32_t *list;
    const float4 *phi, *plo, *nA, *nB;
    const double4_32a *pd, *nD;
    void *as[3], *ah[3];    // soft / hard accelerations (float or double)
    unsigned long long *counter;
    unsigned long long *inter_soft, *inter_hard;   // pairs of the far kernel / of the near kernel
    const Status *st;
    // FP32 work items (see WorkItem) and their number
    const WorkItem *items;
    const uint64_t *nwork;
    const WorkItem *dense_items;          // the end of the near items' array: the dense ones lie before it
    unsigned long long *dense_counter;
    int want_soft, want_hard;
};

struct HardC {
    float eps2, R2, R2sq, R2sqlo, invdR;
};

// ---- FP32 bodies ----------------------------------------------------------
// Eq. (10) with Y from D = R2^2 - r^2: Y = D / ((R2 + r)(R2 - R1)), clamped
// to [0, 1]; K = Y^6 (10 + Y^2 (-15 + 6 Y^2)), exactly 1 at Y = 1 and 0 at Y = 0.
// D is rebuilt in double-float arithmetic from the grid-aligned hi parts
// (whose differences are exact) and the lo parts: near R2, K ~ 10 Y^6
// magnifies any error of R2 - r.
__device__ __forceinline__ float dll_K_precise(float r2u, float hx, float hy, float hz, float lx, float ly, float lz,
                                               const HardC &H)
{
    const float px = __fmul_rn(hx, hx), py = __fmul_rn(hy, hy), pz = __fmul_rn(hz, hz);
    const float ex = __fmaf_rn(hx, hx, -px), ey = __fmaf_rn(hy, hy, -py), ez = __fmaf_rn(hz, hz, -pz);
    // R2^2 - px - py - pz keeping every rounding error (|R2^2| >= px, d1 >= py, d2 >= pz inside R2)
    const float d1 = __fsub_rn(H.R2sq, px), e1 = __fsub_rn(__fsub_rn(H.R2sq, d1), px);
    const float d2 = __fsub_rn(d1, py), e2 = __fsub_rn(__fsub_rn(d1, d2), py);
    const float d3 = __fsub_rn(d2, pz), e3 = __fsub_rn(__fsub_rn(d2, d3), pz);
    // (h + l)^2 = h^2 + (2h + l) l: the lo parts are up to half a grid step, so l^2 counts too
    const float cross = fmaf(2.0f * hx + lx, lx, fmaf(2.0f * hy + ly, ly, (2.0f * hz + lz) * lz));
    const float corr = ((e1 + e2) + e3) + (H.R2sqlo - ((ex + ey) + ez)) - cross;
    const float D = d3 + corr;
    const float r = sqrtf(r2u);
    const float Y = __saturatef(D * H.invdR / (H.R2 + r));
    const float Y2 = Y * Y;
    return (Y2 * Y2 * Y2) * fmaf(Y2, fmaf(6.0f, Y2, -15.0f), 10.0f);
}

__device__ __forceinline__ int64_t next_item(unsigned long long *counter, int lane)
{
    unsigned long long g = 0;
    if (lane == 0) g = atomicAdd(counter, 1ull);
    return (int64_t)__shfl_sync(0xffffffffu, g, 0);
}

// ---------------------------------------------------------------------------
// FP32 work items and source staging
// ---------------------------------------------------------------------------
constexpr uint32_t MULTI = ITEM_MULTI;

// Raw sources (hi, lo float4 pairs of cells or particles) are gathered into a
// ring of NST shared-memory stages (the staging depth, 2 to 4) with 16-byte cp.async copies issued NST - 1 tiles ahead,
// from list indices loaded one tile before that; only the rebasing to the
// group's reference point (one pass per staged entry, by the lane that copied
// it) stands between a landed stage and its use.
constexpr int PER = TILE / 32;

// Rebased sources of the far kernel: each source twice over, {x, x, y, y} {z, z,
// m, m}, for the packed two-sink arithmetic, or in the expanded form of
// exp_tile, two float4 per entry, in tile[0, 2 PADT): entries from nt up to
// PADT = TILE + 32 are zero-mass sources (all zero in either form).
constexpr int PADT = TILE + 32;
template <int NST, int TILE4>
struct WarpStage {
    float4 tile[TILE4];
    float4 rh[NST][TILE];     // raw hi parts (cells: nA, particles: phi)
    float4 rl[NST][TILE];     // raw lo parts (cells: nB, particles: plo)
};

__device__ __forceinline__ void cp16(void *dst, const void *src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

struct ItemSrc {
    uint64_t cbase, pbase;
    uint32_t Lc, e0, e1;

    __device__ __forceinline__ void load_idx(const PairArgs &a, int t, int lane, uint32_t (&idx)[PER]) const
    {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const uint32_t e = e0 + (uint32_t)(t * TILE + u * 32 + lane);
            idx[u] = e < e1 ? a.list[(e < Lc ? cbase : pbase) + e] : 0u;
        }
    }
    // gathers of tile t into stage t % NST; always closes one cp.async group
    template <int NST, typename Stage>
    __device__ __forceinline__ void issue(const PairArgs &a, Stage &S, int t, int lane,
                                          const uint32_t (&idx)[PER]) const
    {
        const int st = t % NST;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const uint32_t e = e0 + (uint32_t)(t * TILE + u * 32 + lane);
            if (e < e1) {
                const bool cell = e < Lc;
                cp16(&S.rh[st][u * 32 + lane], (cell ? a.nA : a.phi) + idx[u]);
                cp16(&S.rl[st][u * 32 + lane], (cell ? a.nB : a.plo) + idx[u]);
            }
        }
        cp_commit();
    }
};

// Runs the staging pipeline over the item's entries and calls body(stage, nt)
// once per tile: the tile's nt raw entries have landed in rh / rl[stage], entry
// e from lane e % 32, which alone may read it before a __syncwarp.
template <int NST, typename Stage, typename Body>
__device__ __forceinline__ void pipeline(const PairArgs &a, const ItemSrc &src, Stage &S, int lane, Body &&body)
{
    static_assert(NST >= 2 && NST <= 4, "staging depth");
    const uint32_t ne = src.e1 - src.e0;
    const int ntile = (int)((ne + TILE - 1) / TILE);
    if (ntile == 0) return;
    {   // prologue: the indices of tiles 0 .. NST-2 are loaded together, then their gathers issued
        uint32_t ip[NST - 1][PER];
#pragma unroll
        for (int t = 0; t < NST - 1; ++t) src.load_idx(a, t, lane, ip[t]);
#pragma unroll
        for (int t = 0; t < NST - 1; ++t) src.issue<NST>(a, S, t, lane, ip[t]);
    }
    uint32_t i0[PER];
    src.load_idx(a, NST - 1, lane, i0);
    for (int t = 0; t < ntile; ++t) {
        src.issue<NST>(a, S, t + NST - 1, lane, i0);   // no copies past the end, but one group per tile
        if (t + NST < ntile) src.load_idx(a, t + NST, lane, i0);
        cp_wait<NST - 1>();                       // this lane's copies of tile t have landed
        body(t % NST, (int)min((uint32_t)TILE, ne - (uint32_t)(t * TILE)));
        __syncwarp();
    }
}

// The far kernel's tile from a stage: every source twice over, or expanded (EXP).
template <bool EXP, typename Stage>
__device__ __forceinline__ void stage_far(Stage &S, int st, int nt, int lane, float crx, float cry, float crz)
{
#pragma unroll
    for (int u = 0; u < PER; ++u) {   // entries past nt become zero-mass sources
        const int el = u * 32 + lane;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (el < nt) {
            const float4 h = S.rh[st][el], l = S.rl[st][el];
            v = make_float4((h.x - crx) + l.x, (h.y - cry) + l.y, (h.z - crz) + l.z, h.w);
        }
        if (!EXP) {
            S.tile[2 * el] = make_float4(v.x, v.x, v.y, v.y);
            S.tile[2 * el + 1] = make_float4(v.z, v.z, v.w, v.w);
        } else {
            const float c = fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z));
            S.tile[2 * el] = make_float4(-2.0f * v.x, -2.0f * v.y, -2.0f * v.z, c);
            S.tile[2 * el + 1] = make_float4(v.w * v.x, v.w * v.y, v.w * v.z, v.w);
        }
    }
    __syncwarp();
}

// sums of the copies into copy 0: a butterfly over the copies when they fill the warp (lpc a power of
// two), else in copy order
template <int KS>
__device__ __forceinline__ void reduce_copies(int lane, int copy, int copies, int lpc, float (&x)[KS], float (&y)[KS],
                                              float (&z)[KS])
{
    if (copies > 1 && copies * lpc == 32) {
        for (int o = lpc; o < 32; o <<= 1) {
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                x[k] += __shfl_xor_sync(0xffffffffu, x[k], o);
                y[k] += __shfl_xor_sync(0xffffffffu, y[k], o);
                z[k] += __shfl_xor_sync(0xffffffffu, z[k], o);
            }
        }
        return;
    }
    for (int cc = 1; cc < copies; ++cc) {
        const int src = (copy == 0) ? lane + cc * lpc : lane;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const float vx = __shfl_sync(0xffffffffu, x[k], src);
            const float vy = __shfl_sync(0xffffffffu, y[k], src);
            const float vz = __shfl_sync(0xffffffffu, z[k], src);
            if (copy == 0) {
                x[k] += vx;
                y[k] += vy;
                z[k] += vz;
            }
        }
    }
}

// ---- packed two-sink arithmetic (f32x2: one instruction, two FP32 lanes) ----
__device__ __forceinline__ uint64_t pk2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Weight 1 (cells, far particles): two sinks (S*) against one source given
// twice over (X2 = {x, x}, ..). GUARD: r^2 + eps^2 may be 0 (eps = 0 and a self
// pair, only possible without a hard part).
template <bool GUARD>
__device__ __forceinline__ void body_far2(uint64_t X2, uint64_t Y2, uint64_t Z2, uint64_t M2, uint64_t SX, uint64_t SY,
                                          uint64_t SZ, uint64_t E2, uint64_t &AX, uint64_t &AY, uint64_t &AZ)
{
    const uint64_t dx = sub2(X2, SX), dy = sub2(Y2, SY), dz = sub2(Z2, SZ);
    const uint64_t r2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, E2)));
    float ra, rb;
    upk2(r2, ra, rb);
    float ia = rsqrtf(ra), ib = rsqrtf(rb);
    if (GUARD) {
        ia = ra > 0.0f ? ia : 0.0f;
        ib = rb > 0.0f ? ib : 0.0f;
    }
    const uint64_t ri = pk2(ia, ib);
    const uint64_t f = mul2(mul2(M2, ri), mul2(ri, ri));
    AX = fma2(dx, f, AX);
    AY = fma2(dy, f, AY);
    AZ = fma2(dz, f, AZ);
}

// The far sweep of one tile: copy c takes sources c, c + copies, ... Every
// lane runs the same number of rounds of two sources (entries from nt to
// PADT are zero-mass sources), so the loop has no divergence; lanes outside
// the copies compute sums that are never used. KP sink pairs per lane.
template <int KP, bool GUARD, typename Stage>
__device__ __forceinline__ void far_tile(const Stage &S, int nt, int copy, int copies, uint64_t E2,
                                         const uint64_t (&SX)[KP], const uint64_t (&SY)[KP], const uint64_t (&SZ)[KP],
                                         uint64_t (&AX)[KP], uint64_t (&AY)[KP], uint64_t (&AZ)[KP])
{
    const int rounds = (nt + 2 * copies - 1) / (2 * copies);
    uint32_t q = (uint32_t)__cvta_generic_to_shared(S.tile) + 32u * (uint32_t)copy;
    const uint32_t step = 32u * (uint32_t)copies;
    for (int m = 0; m < rounds; ++m, q += 2 * step) {
        uint64_t X0, Y0, Z0, M0, X1, Y1, Z1, M1;
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(X0), "=l"(Y0) : "r"(q));
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(Z0), "=l"(M0) : "r"(q + 16));
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(X1), "=l"(Y1) : "r"(q + step));
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(Z1), "=l"(M1) : "r"(q + step + 16));
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            body_far2<GUARD>(X0, Y0, Z0, M0, SX[k], SY[k], SZ[k], E2, AX[k], AY[k], AZ[k]);
            body_far2<GUARD>(X1, Y1, Z1, M1, SX[k], SY[k], SZ[k], E2, AX[k], AY[k], AZ[k]);
        }
    }
}

// Far sources in expanded form. With the source at s and a sink at k
// (both group-relative), r^2 = |s|^2 + (|k|^2 + eps^2) - 2 s.k and
// sum_j m_j r_j^-3 (s_j - k) = sum_j r_j^-3 (m_j s_j) - k sum_j r_j^-3 m_j, so
// a source stages {-2s, |s|^2, m s, m} and a pair costs the sum c + Q, three
// fma for r^2, rsqrt, two mul for r^-3 and four fma: 10 FP32 lane operations
// against 12 for body_far2. The rounding of r^2 is at most about
// 4 u (|s| + |k|)^2 <= 4 u (r + 2 |k|)^2 (u = 2^-24). With a hard part the walk
// takes a cell only beyond R2 + b_max (and beyond its opening radius) and a far
// particle only beyond R2 of the sinks' box, so r >= R2, and with every sink
// within 64 R2 of the reference point the rounding stays below ~4e-3 of r^2
// (r^2 cannot change sign; typical pairs sit far from that bound). Other items
// keep body_far: without a hard part a cell of one or a few particles can be
// taken right next to the sinks, and a very large group in sparse outskirts
// can have far sources at R2 from its edge.
// Q = |k|^2 + eps^2 per sink; the caller subtracts k FM from A at the end.
__device__ __forceinline__ void body_exp2(uint64_t NX, uint64_t NY, uint64_t NZ, uint64_t C2, uint64_t MX, uint64_t MY,
                                           uint64_t MZ, uint64_t M2, uint64_t SX, uint64_t SY, uint64_t SZ, uint64_t Q,
                                           uint64_t &AX, uint64_t &AY, uint64_t &AZ, uint64_t &FM)
{
    const uint64_t r2 = fma2(NX, SX, fma2(NY, SY, fma2(NZ, SZ, add2(C2, Q))));
    float ra, rb;
    upk2(r2, ra, rb);
    const uint64_t ri = pk2(rsqrtf(ra), rsqrtf(rb));
    const uint64_t t = mul2(mul2(ri, ri), ri);
    AX = fma2(MX, t, AX);
    AY = fma2(MY, t, AY);
    AZ = fma2(MZ, t, AZ);
    FM = fma2(M2, t, FM);
}

// The expanded sweep of one tile (same rounds and copies as far_tile); each
// source is stored once, {-2s, |s|^2} {m s, m}, and every value is paired
// with itself in registers for the packed arithmetic.
template <int KP, typename Stage>
__device__ __forceinline__ void exp_tile(const Stage &S, int nt, int copy, int copies, const uint64_t (&SX)[KP],
                                          const uint64_t (&SY)[KP], const uint64_t (&SZ)[KP], const uint64_t (&Q)[KP],
                                          uint64_t (&AX)[KP], uint64_t (&AY)[KP], uint64_t (&AZ)[KP],
                                          uint64_t (&FM)[KP])
{
    const int rounds = (nt + 2 * copies - 1) / (2 * copies);
    uint32_t q = (uint32_t)__cvta_generic_to_shared(S.tile) + 32u * (uint32_t)copy;
    const uint32_t step = 32u * (uint32_t)copies;
    for (int m = 0; m < rounds; ++m, q += 2 * step) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t qa = q + (h ? step : 0u);
            float nx, ny, nz, c, mx, my, mz, ms;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(nx), "=f"(ny), "=f"(nz), "=f"(c) : "r"(qa));
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(mx), "=f"(my), "=f"(mz), "=f"(ms) : "r"(qa + 16));
            const uint64_t NX = pk2(nx, nx), NY = pk2(ny, ny), NZ = pk2(nz, nz), C2 = pk2(c, c);
            const uint64_t MX = pk2(mx, mx), MY = pk2(my, my), MZ = pk2(mz, mz), M2 = pk2(ms, ms);
#pragma unroll
            for (int k = 0; k < KP; ++k)
                body_exp2(NX, NY, NZ, C2, MX, MY, MZ, M2, SX[k], SY[k], SZ[k], Q[k], AX[k], AY[k], AZ[k], FM[k]);
        }
    }
}

// Sums of a round to the outputs, by copy 0: one item of a group stores, several add.
template <int KS>
__device__ __forceinline__ void put_sums(void *const *acc, bool add, float Gf, uint32_t first, int n, int r0, int lpc,
                                         int slot, const float (&x)[KS], const float (&y)[KS], const float (&z)[KS])
{
    float *ox = (float *)acc[0], *oy = (float *)acc[1], *oz = (float *)acc[2];
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
        const int si = r0 + kk * lpc + slot;
        if (si < n) {
            const uint32_t i = first + si;
            if (!add) {
                ox[i] = Gf * x[kk];
                oy[i] = Gf * y[kk];
                oz[i] = Gf * z[kk];
            } else {
                atomicAdd(ox + i, Gf * x[kk]);
                atomicAdd(oy + i, Gf * y[kk]);
                atomicAdd(oz + i, Gf * z[kk]);
            }
        }
    }
}

// Cells and far particles -> soft accelerations.
template <int KS, int NST>
__global__ void __launch_bounds__(PAIR_THREADS, 0) k_far(PairArgs a)
{
    using Stage = WarpStage<NST, 2 * PADT>;
    __shared__ Stage stages[PAIR_WARPS];
    if (a.st->code) return;
    const int lane = threadIdx.x & 31;
    Stage &S = stages[threadIdx.x >> 5];
    for (int e = 2 * TILE + lane; e < 2 * PADT; e += 32) S.tile[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const int64_t W = (int64_t)*a.nwork;
    unsigned long long inter = 0;
    int64_t w = next_item(a.counter, lane);
    while (w < W) {
        const int64_t wn = next_item(a.counter, lane);   // the next item's number arrives while this one runs
        const WorkItem d = a.items[w];
        const SysParams &P = a.sp[d.sys];
        const float eps2 = P.eps2f;
        const ItemSrc src = {d.cbase, d.pbase, d.Lc, d.e0, d.e1};
        const uint32_t first = d.first;
        const int n = (int)(d.n & ~MULTI);
        const bool multi = (d.n & MULTI) != 0;
        const float4 cref = a.phi[first];
        const float crx = cref.x, cry = cref.y, crz = cref.z;
        inter += (unsigned long long)n * (d.e1 - d.e0);
        for (int r0 = 0, per_round = 0; r0 < n; r0 += per_round) {
            const int rem = n - r0;
            int lpc = rem <= 32 * KS ? (rem + KS - 1) / KS : 32;
            // when the copies would leave many sink slots idle (rem * copies below FAR_SPLIT_PCT % of 32 KS), this
            // round takes a power of two of lanes per copy, which keeps every slot busy, and leaves the other sinks
            // to the next round
            if (rem * (32 / lpc) * 100 < FAR_SPLIT_PCT * 32 * KS) lpc = 1 << (31 - __clz(lpc));
            const int copies = 32 / lpc;
            const int copy = lane / lpc, slot = lane - copy * lpc;
            per_round = lpc * KS;
            float sx[KS], sy[KS], sz[KS], ax[KS], ay[KS], az[KS];
#pragma unroll
            for (int kk = 0; kk < KS; ++kk) {
                int si = r0 + kk * lpc + slot;
                si = si < n ? si : n - 1;
                const float4 h = a.phi[first + si], l = a.plo[first + si];
                sx[kk] = (h.x - crx) + l.x;
                sy[kk] = (h.y - cry) + l.y;
                sz[kk] = (h.z - crz) + l.z;
            }
            constexpr int KP = (KS + 1) / 2;
            uint64_t SX[KP], SY[KP], SZ[KP], AX[KP], AY[KP], AZ[KP];
#pragma unroll
            for (int p = 0; p < KP; ++p) {
                const int k1 = 2 * p + 1 < KS ? 2 * p + 1 : 2 * p;
                SX[p] = pk2(sx[2 * p], sx[k1]);
                SY[p] = pk2(sy[2 * p], sy[k1]);
                SZ[p] = pk2(sz[2 * p], sz[k1]);
                AX[p] = AY[p] = AZ[p] = 0ull;
            }
            const uint64_t E2 = pk2(eps2, eps2);
            // the expanded form only with a hard part (then every far source is at least R2 from the sinks'
            // box; without one, cells and particles can sit next to the sinks) and for sinks within 64 R2
            // of the reference point: the rounding of r^2 stays below 4 u (1 + 2 * 64)^2 ~ 4e-3 of r^2
            float k2 = 0.0f;
#pragma unroll
            for (int kk = 0; kk < KS; ++kk) k2 = fmaxf(k2, fmaf(sx[kk], sx[kk], fmaf(sy[kk], sy[kk], sz[kk] * sz[kk])));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) k2 = fmaxf(k2, __shfl_xor_sync(0xffffffffu, k2, o));
            if (eps2 > 0.0f && P.has_hard && k2 <= 4096.0f * P.R2sqf) {
                uint64_t Q[KP], FM[KP];
#pragma unroll
                for (int p = 0; p < KP; ++p) {
                    const int k1 = 2 * p + 1 < KS ? 2 * p + 1 : 2 * p;
                    Q[p] = pk2(fmaf(sx[2 * p], sx[2 * p], fmaf(sy[2 * p], sy[2 * p], fmaf(sz[2 * p], sz[2 * p], eps2))),
                               fmaf(sx[k1], sx[k1], fmaf(sy[k1], sy[k1], fmaf(sz[k1], sz[k1], eps2))));
                    FM[p] = 0ull;
                }
                pipeline<NST>(a, src, S, lane, [&](int st, int nt) {
                    stage_far<true>(S, st, nt, lane, crx, cry, crz);
                    exp_tile<KP>(S, nt, copy, copies, SX, SY, SZ, Q, AX, AY, AZ, FM);
                });
#pragma unroll
                for (int p = 0; p < KP; ++p) {   // A - k FM
                    const int k1 = 2 * p + 1 < KS ? 2 * p + 1 : 2 * p;
                    AX[p] = fma2(pk2(-sx[2 * p], -sx[k1]), FM[p], AX[p]);
                    AY[p] = fma2(pk2(-sy[2 * p], -sy[k1]), FM[p], AY[p]);
                    AZ[p] = fma2(pk2(-sz[2 * p], -sz[k1]), FM[p], AZ[p]);
                }
            } else if (eps2 > 0.0f) {
                pipeline<NST>(a, src, S, lane, [&](int st, int nt) {
                    stage_far<false>(S, st, nt, lane, crx, cry, crz);
                    far_tile<KP, false>(S, nt, copy, copies, E2, SX, SY, SZ, AX, AY, AZ);
                });
            } else {   // eps = 0 without a hard part: a sink meets itself in its far particles
                pipeline<NST>(a, src, S, lane, [&](int st, int nt) {
                    stage_far<false>(S, st, nt, lane, crx, cry, crz);
                    far_tile<KP, true>(S, nt, copy, copies, E2, SX, SY, SZ, AX, AY, AZ);
                });
            }
#pragma unroll
            for (int p = 0; p < KP; ++p) {
                float t0, t1;
                upk2(AX[p], t0, t1);
                ax[2 * p] = t0;
                if (2 * p + 1 < KS) ax[2 * p + 1] = t1;
                upk2(AY[p], t0, t1);
                ay[2 * p] = t0;
                if (2 * p + 1 < KS) ay[2 * p + 1] = t1;
                upk2(AZ[p], t0, t1);
                az[2 * p] = t0;
                if (2 * p + 1 < KS) az[2 * p + 1] = t1;
            }
            reduce_copies<KS>(lane, copy, copies, lpc, ax, ay, az);
            if (copy == 0) put_sums<KS>(a.as, multi, P.Gf, first, n, r0, lpc, slot, ax, ay, az);
        }
        w = wn;
    }
    cp_wait<0>();   // nothing may stay in flight into shared memory at exit
    if (lane == 0) atomicAdd(a.inter_soft, inter);
}

// ---------------------------------------------------------------------------
// Near particles -> F (1 - K) into the soft and F K into the hard accelerations.
//
// Few near pairs lie within R2 (1.4 % at N = 2^24), but only they need K, some
// 60 instructions, so each tile of sources takes two steps. The distance step
// touches every pair that has to be touched, two sources per instruction and
// without branches, and marks the pairs within R2 in a bit mask per lane; the K
// step then walks the masks, every lane with its own next pair, so a warp runs
// as many K evaluations as its fullest lane has, not one for every source that
// some lane is close to.
//  - HARD alone: pairs beyond R2 contribute nothing, so a warp first packs
//    together the sources within R2 of the box of its sinks (computed with the
//    pair distance's roundings: none is missed).
//  - SOFT: every pair adds F at weight 1 unless it is marked.
// Groups with many pairs within R2 take the loop of near_dense instead.
//
// One block per work item: its warps take blocks of at most 32 consecutive
// sinks (compact in key order), one sink per lane, and share the tiles of
// NEAR_TILE sources, one gathered by each thread while the last tile is worked
// on; with one or two blocks of sinks the warps split the sources. One sink a
// lane keeps the kernel at 64 registers, 32 warps per SM: with 4 sinks a lane
// (124 registers, 16 warps) it was bound by latency at 38-50 % of the issue
// slots, whatever the instruction count; 6 blocks per SM are slower too (2^24
// 39.1 against 35.7 ms). Near time per step against the form before (one warp
// per item, 4 sinks a lane, a divergent K for every source within R2 of some
// lane): N = 2^12 0.139 -> 0.071 ms, 2^17 0.337 -> 0.256, 2^20 (absolute MAC)
// 1.60 -> 1.09, 2^24 40.2 -> 35.2 ms.
// ---------------------------------------------------------------------------
constexpr int NEAR_TILE = PAIR_THREADS;
constexpr float FAR_AWAY = 1e18f;   // padding sources: r^2 is finite; massless, so R2 may be larger (SI or cgs units)

struct NearTile {
    float4 hi[NEAR_TILE];   // rebased hi parts and mass (differences with the sinks' hi parts are exact)
    float4 lo[NEAR_TILE];
};

// the sources a distance step runs over, two by two
struct NearPacked {
    float x[NEAR_TILE], y[NEAR_TILE], z[NEAR_TILE];
    uint8_t j[NEAR_TILE];   // their entries in the tile
};

struct NearSink {
    float hx, hy, hz, lx, ly, lz;   // rebased hi parts and lo parts
};

// One marked pair per lane (on: whether this lane has one), entry j of the tile: r^2 and K as the FP32 form defines them.
template <bool SOFT, bool HARD>
__device__ __forceinline__ void near_pair(const NearTile &T, int j, bool on, const NearSink &s, const HardC &H, float &sax,
                                          float &say, float &saz, float &hax, float &hay, float &haz)
{
    const float4 h = T.hi[j], l = T.lo[j];
    const float dx = (h.x + l.x) - (s.hx + s.lx), dy = (h.y + l.y) - (s.hy + s.ly), dz = (h.z + l.z) - (s.hz + s.lz);
    const float r2u = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float r2 = r2u + H.eps2;
    const float ri = r2 > 0.0f ? rsqrtf(r2) : 0.0f;
    const float f = on ? h.w * ri * (ri * ri) : 0.0f;
    float K = dll_K_precise(r2u, __fsub_rn(h.x, s.hx), __fsub_rn(h.y, s.hy), __fsub_rn(h.z, s.hz), __fsub_rn(l.x, s.lx),
                            __fsub_rn(l.y, s.ly), __fsub_rn(l.z, s.lz), H);
    if (SOFT) {
        K = r2u < H.R2sq ? K : 0.0f;   // the mark of the soft form is a little generous
        const float fs = f * (1.0f - K);
        sax = fmaf(dx, fs, sax);
        say = fmaf(dy, fs, say);
        saz = fmaf(dz, fs, saz);
    }
    if (HARD) {
        const float fh = f * K;
        hax = fmaf(dx, fh, hax);
        hay = fmaf(dy, fh, hay);
        haz = fmaf(dz, fh, haz);
    }
}

// order-preserving integer image of a float (and back)
__device__ __forceinline__ int ord_f(float v)
{
    const int i = __float_as_int(v);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unord_f(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// ---- dense items ----------------------------------------------------------
// Where many of the listed pairs lie within R2 (a clump inside one R2, an R2 of many leaves), marking them and walking
// the marks costs more than it saves: the K step is bound by the issue rate (89 %), at some 95 instructions a pair, and
// with one sink a lane half the lanes idle on groups of about 20. The walk tells such groups by their boxes (NEAR_DENSE),
// and their items, at the other end of the near items' array, are worked on by the loop below: no distance step, two
// sources per packed instruction, and the lanes that a block of sinks leaves over hold further copies of it, each with
// its own source pairs (lanes busy on the groups of a Plummer sphere of 2^17: 86 % against 52 %).
// Near time per step, marks alone -> with this: 2^17 with R2 = 32, 64, 128 eps 1.07 -> .81, 4.37 -> 2.78, 21.9 -> 12.2 ms
// (R2 = 8 eps .176 -> .178, 10^6 1.019 -> 1.034: the registers of the two loops together); a tenth of 2^17 particles in a
// clump of half an R2 4.70 -> 2.25 (bound by the FMA pipe then: its throttle is the top stall; the form before the marks
// took 2.31); N = 30000 with 64 eps 1.27 -> .76. NEAR_DENSE = 0.7: with 0.4 .93 and 2.89 ms for 32
// and 64 eps, with 1 as with 0.7. Counting the near leaves close to the group in the walk chose no better and cost it 4 %.
// A kernel of its own for these items (80 registers, beside k_near on the second stream) was 2 to 4 % faster on them, but
// its launch cost steps of 2^13 particles 2 %.

struct NearSink2 {   // a sink's rebased hi parts and lo parts, twice over
    uint64_t hx, hy, hz, lx, ly, lz;
};

// Two sources (rebased hi parts, masses, lo parts) against one sink, K evaluated if one of them is within R2 (it is 0
// beyond): r^2 from the parts' differences, K term by term as dll_K_precise has it.
template <bool SOFT, bool HARD>
__device__ __forceinline__ void near_both(uint64_t HX, uint64_t HY, uint64_t HZ, uint64_t M, uint64_t LX, uint64_t LY,
                                          uint64_t LZ, const NearSink2 &S, const HardC &H, uint64_t &AX, uint64_t &AY,
                                          uint64_t &AZ, uint64_t &BX, uint64_t &BY, uint64_t &BZ)
{
    const uint64_t hx = sub2(HX, S.hx), hy = sub2(HY, S.hy), hz = sub2(HZ, S.hz);
    const uint64_t lx = sub2(LX, S.lx), ly = sub2(LY, S.ly), lz = sub2(LZ, S.lz);
    const uint64_t dx = add2(hx, lx), dy = add2(hy, ly), dz = add2(hz, lz);
    const uint64_t r2u = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
    float u0, u1, m0, m1;
    upk2(r2u, u0, u1);
    upk2(M, m0, m1);
    const float r0 = u0 + H.eps2, r1 = u1 + H.eps2;
    const float i0 = r0 > 0.0f ? rsqrtf(r0) : 0.0f, i1 = r1 > 0.0f ? rsqrtf(r1) : 0.0f;
    uint64_t f = 0ull;
    if (SOFT) f = mul2(mul2(M, pk2(i0, i1)), mul2(pk2(i0, i1), pk2(i0, i1)));
    if (u0 < H.R2sq || u1 < H.R2sq) {
        const uint64_t nx = mul2(hx, sub2(S.hx, HX)), ny = mul2(hy, sub2(S.hy, HY)), nz = mul2(hz, sub2(S.hz, HZ));   // -h^2
        const uint64_t R = pk2(H.R2sq, H.R2sq);
        const uint64_t d1 = add2(R, nx), d2 = add2(d1, ny), d3 = add2(d2, nz);
        const uint64_t e = add2(add2(add2(sub2(R, d1), nx), add2(sub2(d1, d2), ny)), add2(sub2(d2, d3), nz));
        const uint64_t q = add2(add2(fma2(hx, hx, nx), fma2(hy, hy, ny)), fma2(hz, hz, nz));
        const uint64_t cross = fma2(add2(add2(hx, hx), lx), lx, fma2(add2(add2(hy, hy), ly), ly, mul2(add2(add2(hz, hz), lz), lz)));
        const uint64_t D = add2(d3, sub2(add2(e, sub2(pk2(H.R2sqlo, H.R2sqlo), q)), cross));
        float D0, D1;
        upk2(D, D0, D1);
        auto K_of = [&](float u, float Dk) -> float {
            const float Y = __saturatef(__fdividef(Dk * H.invdR, H.R2 + sqrtf(u)));
            const float Y2 = Y * Y;
            return (Y2 * Y2 * Y2) * fmaf(Y2, fmaf(6.0f, Y2, -15.0f), 10.0f);
        };
        const uint64_t K = pk2(K_of(u0, D0), K_of(u1, D1));
        if (!SOFT) f = mul2(mul2(M, pk2(i0, i1)), mul2(pk2(i0, i1), pk2(i0, i1)));
        if (HARD) {
            const uint64_t fh = mul2(f, K);
            BX = fma2(dx, fh, BX);
            BY = fma2(dy, fh, BY);
            BZ = fma2(dz, fh, BZ);
        }
        if (SOFT) f = mul2(f, sub2(pk2(1.0f, 1.0f), K));
    }
    if (SOFT) {
        AX = fma2(dx, f, AX);
        AY = fma2(dy, f, AY);
        AZ = fma2(dz, f, AZ);
    }
}

// A dense item's tile, its sources two by two: {hx hx' hy hy'} {hz hz' m m'} {lx lx' ly ly'} {lz lz'}.
struct NearPairs {
    float4 a[NEAR_TILE / 2], b[NEAR_TILE / 2], c[NEAR_TILE / 2];
    float2 d[NEAR_TILE / 2];
};
static_assert(sizeof(NearPairs) <= sizeof(NearTile), "either form of a tile");

// Blocks of sinks that a group of up to 64 is cut into: the fewest that keep the most lanes busy, a warp holding 32 / per
// copies of a block of per sinks.
constexpr int near_cut(int n)
{
    int best = n <= 32 ? 1 : 2;
    for (int nb = 2 * best; nb <= 4; nb *= 2) {
        const int c0 = 32 / ((n + best - 1) / best), c1 = 32 / ((n + nb - 1) / nb);   // slots per sink: 32 nb / copies
        if (nb * c0 < best * c1) best = nb;
    }
    return best;
}
constexpr uint64_t near_cuts(int nb)   // bit n - 1: groups of n are cut into nb blocks
{
    uint64_t m = 0;
    for (int n = 1; n <= 64; ++n) m |= near_cut(n) == nb ? 1ull << (n - 1) : 0ull;
    return m;
}
constexpr uint64_t NEAR_CUT2 = near_cuts(2), NEAR_CUT4 = near_cuts(4);

// The dense items, W of them, by the blocks in turn. Returns the number of pairs of this block's.
template <bool SOFT, bool HARD>
__device__ __forceinline__ unsigned long long near_dense(const PairArgs &a, uint32_t W, NearTile *tiles, uint32_t &sh_item)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long inter = 0;
    uint32_t next = 0;
    for (uint32_t it = blockIdx.x; it < W;) {   // a block's first item by its place in the grid
        if (threadIdx.x == 0) next = gridDim.x + (uint32_t)atomicAdd(a.dense_counter, 1ull);   // arrives while this one runs
        const WorkItem d = a.dense_items[-1 - (int64_t)it];   // from the end of the array down
        const SysParams &P = a.sp[d.sys];
        const HardC H = {P.eps2f, P.R2f, P.R2sqf, P.R2sqlo, P.invdRf};
        const uint32_t *list = a.list + d.pbase + d.e0;
        const int ne = (int)(d.e1 - d.e0), n = (int)(d.n & ~MULTI);
        inter += (unsigned long long)n * (unsigned long long)ne;
        const bool multi = (d.n & MULTI) != 0;
        const float4 cref = a.phi[d.first];
        const int nblk = n > 64 ? (n + 31) / 32 : (((NEAR_CUT4 >> (n - 1)) & 1ull) ? 4 : (((NEAR_CUT2 >> (n - 1)) & 1ull) ? 2 : 1));
        const int per = (n + nblk - 1) / nblk, ntile = (ne + NEAR_TILE - 1) / NEAR_TILE;
        for (int b0 = 0; b0 < nblk; b0 += PAIR_WARPS) {
            const int here = min(nblk - b0, PAIR_WARPS);
            const int splits = here == 1 ? 4 : (here == 2 ? 2 : 1);   // warps per block of sinks, each a part of every tile
            const int blk = b0 + w / splits, part = w - (w / splits) * splits;
            const int s0 = blk * per, sn = blk < nblk ? min(per, n - s0) : 0;
            const bool busy = sn > 0;
            // a lane is sink `slot` of copy `copy`, which takes every copies-th pair of sources (the lanes left over: none)
            const uint32_t inv = busy ? (65536u + sn - 1) / sn : 0u;   // lane / sn = (lane inv) >> 16
            const int copies = (int)((32u * inv) >> 16), own = (int)((lane * inv) >> 16), slot = lane - own * sn;
            const int copy = own < copies ? own : NEAR_TILE;
            NearSink2 S = {0, 0, 0, 0, 0, 0};
            if (busy) {
                const float4 h = a.phi[d.first + s0 + slot], l = a.plo[d.first + s0 + slot];
                const float x = h.x - cref.x, y = h.y - cref.y, z = h.z - cref.z;
                S = NearSink2{pk2(x, x), pk2(y, y), pk2(z, z), pk2(l.x, l.x), pk2(l.y, l.y), pk2(l.z, l.z)};
            }
            uint64_t AX = 0ull, AY = 0ull, AZ = 0ull, BX = 0ull, BY = 0ull, BZ = 0ull;
            auto index = [&](int t) -> uint32_t {
                const int e = t * NEAR_TILE + (int)threadIdx.x;
                return e < ne ? list[e] : NONE;
            };
            float4 gh = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, 0.0f), gl = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            auto gather = [&](uint32_t i) {
                if (i != NONE) {
                    gh = a.phi[i];
                    gl = a.plo[i];
                } else {
                    gh = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, 0.0f);
                }
            };
            uint32_t i1 = index(0);
            gather(i1);
            i1 = ntile > 1 ? index(1) : NONE;
            for (int t = 0; t < ntile; ++t) {
                NearPairs &T = *(NearPairs *)&tiles[t & 1];
                {
                    const int k = threadIdx.x >> 1, b = threadIdx.x & 1;
                    float *u = (float *)&T.a[k] + b;
                    u[0] = gh.x - cref.x;
                    u[2] = gh.y - cref.y;
                    u = (float *)&T.b[k] + b;
                    u[0] = gh.z - cref.z;
                    u[2] = gh.w;
                    u = (float *)&T.c[k] + b;
                    u[0] = gl.x;
                    u[2] = gl.y;
                    ((float *)&T.d[k])[b] = gl.z;
                }
                if (t + 1 < ntile) {
                    gather(i1);
                    i1 = t + 2 < ntile ? index(t + 2) : NONE;
                }
                __syncthreads();
                if (!busy) continue;
                const int nt = min(NEAR_TILE, ne - t * NEAR_TILE);
                const int q0 = part * (NEAR_TILE / 2 / splits), q1 = min((nt + 1) / 2, q0 + NEAR_TILE / 2 / splits);
#pragma unroll 1
                for (int q = q0 + copy; q < q1; q += copies) {
                    const uint32_t u = (uint32_t)__cvta_generic_to_shared(&T) + 16u * (uint32_t)q;
                    uint64_t HX, HY, HZ, M, LX, LY, LZ;
                    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(HX), "=l"(HY) : "r"(u));
                    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(HZ), "=l"(M) : "r"(u + 8u * NEAR_TILE));
                    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(LX), "=l"(LY) : "r"(u + 16u * NEAR_TILE));
                    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(LZ) : "r"(u - 8u * (uint32_t)q + 24u * NEAR_TILE));
                    near_both<SOFT, HARD>(HX, HY, HZ, M, LX, LY, LZ, S, H, AX, AY, AZ, BX, BY, BZ);
                }
            }
            if (busy) {   // the copies' sums into the first
                float v[6], t0, t1;
                upk2(SOFT ? AX : BX, t0, t1);
                v[0] = t0 + t1;
                upk2(SOFT ? AY : BY, t0, t1);
                v[1] = t0 + t1;
                upk2(SOFT ? AZ : BZ, t0, t1);
                v[2] = t0 + t1;
                if (SOFT && HARD) {
                    upk2(BX, t0, t1);
                    v[3] = t0 + t1;
                    upk2(BY, t0, t1);
                    v[4] = t0 + t1;
                    upk2(BZ, t0, t1);
                    v[5] = t0 + t1;
                }
                constexpr int NV = SOFT && HARD ? 6 : 3;
                for (int k = 1; k < copies; ++k) {
                    const int src = min(lane + k * sn, 31);
#pragma unroll
                    for (int j = 0; j < NV; ++j) {
                        const float y = __shfl_sync(0xffffffffu, v[j], src);
                        if (copy == 0) v[j] += y;
                    }
                }
                if (copy == 0) {
                    const uint32_t i = d.first + s0 + slot;
#pragma unroll
                    for (int j = 0; j < NV; ++j) {
                        float *o = (float *)(SOFT && j < 3 ? a.as[j] : a.ah[j % 3]) + i;
                        if (!(SOFT && j < 3) && !multi && splits == 1) *o = P.Gf * v[j];
                        else atomicAdd(o, P.Gf * v[j]);   // the near part of the soft force is added to the far part
                    }
                }
            }
            if (b0 + PAIR_WARPS < nblk) __syncthreads();   // the next blocks of sinks write tile 0 again
        }
        if (threadIdx.x == 0) sh_item = next;
        __syncthreads();   // and this item's tiles are used
        it = sh_item;
    }
    return inter;
}

template <bool SOFT, bool HARD>
__global__ void __launch_bounds__(PAIR_THREADS, NEAR_MIN_BLOCKS) k_near(PairArgs a)
{
    __shared__ __align__(16) NearTile tiles[2];
    __shared__ __align__(16) float packed_mem[SOFT ? 2 * 4 * NEAR_TILE : PAIR_WARPS * (sizeof(NearPacked) + 3) / 4];
    __shared__ int64_t sh_item;
    __shared__ uint32_t sh_dense;
    const uint64_t nwork = *a.nwork;   // on its way with the status
    if (a.st->code) return;
    unsigned long long inter = 0;
    const uint32_t ndense = (uint32_t)(nwork >> 32);   // these first: they take longer
    if (blockIdx.x < ndense) inter = near_dense<SOFT, HARD>(a, ndense, tiles, sh_dense);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned ltm = (1u << lane) - 1u;
    const int64_t W = (uint32_t)nwork;
    unsigned long long next = 0;
    if (threadIdx.x == 0) next = atomicAdd(a.counter, 1ull);
    for (;;) {
        __syncthreads();   // the last item's tiles are used
        if (threadIdx.x == 0) {
            sh_item = (int64_t)next;
            next = atomicAdd(a.counter, 1ull);   // arrives while this item runs
        }
        __syncthreads();
        const int64_t it = sh_item;
        if (it >= W) break;
        // items from the last written to the first, which shortens the end of the launch
        const WorkItem d = a.items[W - 1 - it];
        const SysParams &P = a.sp[d.sys];
        HardC H;
        H.eps2 = P.eps2f;
        H.R2 = P.R2f;
        H.R2sq = P.R2sqf;
        H.R2sqlo = P.R2sqlo;
        H.invdR = P.invdRf;
        const uint32_t *list = a.list + d.pbase;   // entries [e0, e1): particles
        const int ne = (int)(d.e1 - d.e0);
        const int n = (int)(d.n & ~MULTI);
        const bool multi = (d.n & MULTI) != 0;
        const float4 cref = a.phi[d.first];
        inter += (unsigned long long)n * (unsigned long long)ne;
        const int nblk = (n + 31) / 32, per = (n + nblk - 1) / nblk;   // blocks of at most 32 sinks, about equal
        const int ntile = (ne + NEAR_TILE - 1) / NEAR_TILE;
        for (int b0 = 0; b0 < nblk; b0 += PAIR_WARPS) {
            const int here = min(nblk - b0, PAIR_WARPS);
            const int splits = here == 1 ? 4 : (here == 2 ? 2 : 1);   // warps per block of sinks, each a part of every tile
            const int blk = b0 + w / splits, part = w - (w / splits) * splits;
            const bool busy = blk < nblk;
            const int s0 = blk * per, sn = busy ? min(per, n - s0) : 0;
            NearSink s = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            if (busy) {
                const uint32_t i = d.first + s0 + min(lane, sn - 1);
                const float4 h = a.phi[i], l = a.plo[i];
                s = NearSink{h.x - cref.x, h.y - cref.y, h.z - cref.z, l.x, l.y, l.z};
            }
            const float sx = s.hx + s.lx, sy = s.hy + s.ly, sz = s.hz + s.lz;
            const uint64_t SX = pk2(sx, sx), SY = pk2(sy, sy), SZ = pk2(sz, sz);
            float lo[3], hi[3];
            if (!SOFT) {   // the box of the warp's sinks
                lo[0] = unord_f(__reduce_min_sync(0xffffffffu, ord_f(sx)));
                lo[1] = unord_f(__reduce_min_sync(0xffffffffu, ord_f(sy)));
                lo[2] = unord_f(__reduce_min_sync(0xffffffffu, ord_f(sz)));
                hi[0] = unord_f(__reduce_max_sync(0xffffffffu, ord_f(sx)));
                hi[1] = unord_f(__reduce_max_sync(0xffffffffu, ord_f(sy)));
                hi[2] = unord_f(__reduce_max_sync(0xffffffffu, ord_f(sz)));
            }
            float ax = 0.0f, ay = 0.0f, az = 0.0f, bx = 0.0f, by = 0.0f, bz = 0.0f;
            uint64_t AX = 0ull, AY = 0ull, AZ = 0ull;
            const uint64_t E2 = pk2(H.eps2, H.eps2);
            // this thread's source of a tile; past the end a far-away massless one
            auto index = [&](int t) -> uint32_t {
                const int e = t * NEAR_TILE + (int)threadIdx.x;
                return e < ne ? list[d.e0 + (uint32_t)e] : NONE;
            };
            float4 gh = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, 0.0f), gl = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            auto gather = [&](uint32_t i) {
                if (i != NONE) {
                    gh = a.phi[i];
                    gl = a.plo[i];
                } else {
                    gh = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, 0.0f);
                }
            };
            uint32_t i1 = index(0);
            gather(i1);
            i1 = ntile > 1 ? index(1) : NONE;
            for (int t = 0; t < ntile; ++t) {
                // double-buffered: a tile is written again only after a barrier that follows its use
                NearTile &T = tiles[t & 1];
                const float4 h = make_float4(gh.x - cref.x, gh.y - cref.y, gh.z - cref.z, gh.w);
                T.hi[threadIdx.x] = h;
                T.lo[threadIdx.x] = gl;
                if (SOFT) {   // source pairs {x x' y y'} {z z' m m'}
                    float *q = packed_mem + (t & 1) * 4 * NEAR_TILE + (threadIdx.x >> 1) * 8 + (threadIdx.x & 1);
                    q[0] = h.x + gl.x;
                    q[2] = h.y + gl.y;
                    q[4] = h.z + gl.z;
                    q[6] = h.w;
                }
                if (t + 1 < ntile) {   // the next tile's sources, and the indices of the one after
                    gather(i1);
                    i1 = t + 2 < ntile ? index(t + 2) : NONE;
                }
                __syncthreads();
                if (!busy) continue;
                const int nt = min(NEAR_TILE, ne - t * NEAR_TILE);
                if constexpr (SOFT) {
                    const float near2 = (H.R2sq + H.eps2) * 1.000001f;   // marks every pair within R2, a few beyond
                    const int q0 = part * (NEAR_TILE / 2 / splits), q1 = min((nt + 1) / 2, q0 + NEAR_TILE / 2 / splits);
                    const float4 *pk = (const float4 *)(packed_mem + (t & 1) * 4 * NEAR_TILE);
                    for (int m0 = q0; m0 < q1; m0 += 16) {   // 16 source pairs: one mask word
                        uint32_t mark = 0u, bit = 1u;
                        const int m1 = min(q1, m0 + 16);
#pragma unroll 2
                        for (int m = m0; m < m1; ++m, bit <<= 2) {
                            const float4 u = pk[2 * m], v = pk[2 * m + 1];
                            const uint64_t dx = sub2(pk2(u.x, u.y), SX), dy = sub2(pk2(u.z, u.w), SY), dz = sub2(pk2(v.x, v.y), SZ);
                            const uint64_t r2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, E2)));
                            float ra, rb, fa, fb;
                            upk2(r2, ra, rb);
                            const uint64_t ri = pk2(rsqrtf(ra), rsqrtf(rb));
                            upk2(mul2(mul2(pk2(v.z, v.w), ri), mul2(ri, ri)), fa, fb);
                            const bool ia = ra < near2, ib = rb < near2;
                            const uint64_t f = pk2(ia ? 0.0f : fa, ib ? 0.0f : fb);
                            mark |= ia ? bit : 0u;
                            mark |= ib ? 2u * bit : 0u;
                            AX = fma2(dx, f, AX);
                            AY = fma2(dy, f, AY);
                            AZ = fma2(dz, f, AZ);
                        }
                        while (__any_sync(0xffffffffu, mark != 0u)) {
                            const bool on = mark != 0u;
                            const int j = on ? 2 * m0 + __ffs(mark) - 1 : 0;
                            near_pair<SOFT, HARD>(T, j, on, s, H, ax, ay, az, bx, by, bz);
                            mark &= mark - 1u;
                        }
                    }
                } else {
                    NearPacked &p = *(NearPacked *)((char *)packed_mem + w * ((sizeof(NearPacked) + 3) / 4 * 4));
                    int nin = 0;
#pragma unroll
                    for (int u = 0; u < NEAR_TILE / 32; ++u) {
                        const int el = u * 32 + lane;
                        if (u / (4 / splits) != part) continue;   // this warp's part of the tile
                        if (u * 32 >= nt) break;
                        const float4 qh = T.hi[el], ql = T.lo[el];
                        const float x = qh.x + ql.x, y = qh.y + ql.y, z = qh.z + ql.z;
                        const float gx = fmaxf(fmaxf(lo[0] - x, x - hi[0]), 0.0f);
                        const float gy = fmaxf(fmaxf(lo[1] - y, y - hi[1]), 0.0f);
                        const float gz = fmaxf(fmaxf(lo[2] - z, z - hi[2]), 0.0f);
                        const bool keep = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < H.R2sq;
                        const unsigned km = __ballot_sync(0xffffffffu, keep);
                        if (keep) {
                            const int q = nin + __popc(km & ltm);
                            p.x[q] = x;
                            p.y[q] = y;
                            p.z[q] = z;
                            p.j[q] = (uint8_t)el;
                        }
                        nin += __popc(km);
                    }
                    if (nin == 0) continue;
                    __syncwarp();
                    const int rounds = (nin + 1) / 2;
                    for (int m0 = 0; m0 < rounds; m0 += 16) {   // 16 source pairs: one mask word
                        uint32_t mark = 0u, bit = 1u;
                        const int m1 = min(rounds, m0 + 16);
#pragma unroll 4
                        for (int m = m0; m < m1; ++m, bit <<= 2) {
                            const float2 x = *(const float2 *)&p.x[2 * m], y = *(const float2 *)&p.y[2 * m],
                                         z = *(const float2 *)&p.z[2 * m];
                            const uint64_t dx = sub2(pk2(x.x, x.y), SX), dy = sub2(pk2(y.x, y.y), SY), dz = sub2(pk2(z.x, z.y), SZ);
                            float ra, rb;
                            upk2(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), ra, rb);
                            mark |= ra < H.R2sq ? bit : 0u;
                            mark |= rb < H.R2sq ? 2u * bit : 0u;
                        }
                        // with an odd number of sources the last pair's other half is none of them
                        if (2 * m1 > nin) mark &= ~(2u << 2 * (m1 - 1 - m0));
                        while (__any_sync(0xffffffffu, mark != 0u)) {
                            const bool on = mark != 0u;
                            const int j = on ? p.j[2 * m0 + __ffs(mark) - 1] : 0;
                            near_pair<SOFT, HARD>(T, j, on, s, H, ax, ay, az, bx, by, bz);
                            mark &= mark - 1u;
                        }
                    }
                    __syncwarp();   // the packed sources are used
                }
            }
            if (busy && lane < sn) {
                const uint32_t i = d.first + s0 + lane;
                const float Gf = P.Gf;
                if (SOFT) {   // the near part is added to the far part
                    float t0, t1;
                    upk2(AX, t0, t1);
                    atomicAdd((float *)a.as[0] + i, Gf * (ax + (t0 + t1)));
                    upk2(AY, t0, t1);
                    atomicAdd((float *)a.as[1] + i, Gf * (ay + (t0 + t1)));
                    upk2(AZ, t0, t1);
                    atomicAdd((float *)a.as[2] + i, Gf * (az + (t0 + t1)));
                }
                if (HARD) {
                    if (!multi && splits == 1) {
                        ((float *)a.ah[0])[i] = Gf * bx;
                        ((float *)a.ah[1])[i] = Gf * by;
                        ((float *)a.ah[2])[i] = Gf * bz;
                    } else {
                        atomicAdd((float *)a.ah[0] + i, Gf * bx);
                        atomicAdd((float *)a.ah[1] + i, Gf * by);
                        atomicAdd((float *)a.ah[2] + i, Gf * bz);
                    }
                }
            }
            if (b0 + PAIR_WARPS < nblk) __syncthreads();   // the next blocks of sinks write tile 0 again
        }
    }
    if (threadIdx.x == 0) atomicAdd(a.inter_hard, inter);
}

// ---------------------------------------------------------------------------
// FP64 kernel. The FP64 pipe (2 lanes per SM and clock) bounds it, so what
// counts is that every SM has work and every lane holds a pair. Work unit =
// (group, slice of at most F64_SINKS sinks), one block of F64_WARPS warps
// each: a warp's lanes are lpc sinks (a power of two) times 32 / lpc copies,
// and the unit's sources go round robin to the F64_WARPS x copies lanes of a
// sink, straight from global memory (a source is 32 B against 4 sinks x 7
// FP64 instructions of 16 clocks: loads are nowhere near the limit). The
// partial sums are added in a fixed order (butterfly over the copies, then the
// warps), and the split depends on the group alone, so a system's forces are
// the same bit for bit alone and in any batch.
// Before, one warp per group with sqrt and division: the far launch of a system
// of 4096 particles took 4.1 ms, its ~100 groups leaving most SMs idle. A soft
// step of 4 hard sub-steps went from 11.9 to 2.07 ms at N = 4096, one
// kick-drift-kick step at N = 30011 from 30.3 to 4.8 ms (8 sinks a slice).
// Slices of 4 sinks make twice the units, so the last ones leave fewer SMs
// idle: far and near .374 + .244 -> .229 + .184 ms of that soft step, 2.51 +
// .71 -> 2.36 + .68 ms at N = 30011. With x^-3/2 and x^1/2 in fixed point
// (fp64_rsqrt.cuh) .149 + .159 and 1.46 + .48 ms; slices of 2 then .128 + .173
// and 1.44 + .55, of 8 .237 + .202 and 1.55 + .50, 8 warps a unit .134 + .182
// and 1.45 + .56. With r^2 + eps^2 in fixed point too .123 + .155 and 1.07 + .46
// ms; slices of 2 .096 + .171 and 1.05 + .53. With the near pairs' r^2 too .121 +
// .132 and 1.07 + .366.
// ---------------------------------------------------------------------------
constexpr int F64_SINKS = 4, F64_WARPS = 4;

template <bool NEAR, bool SOFT, bool HARD>
__global__ void __launch_bounds__(32 * F64_WARPS) k_pair_f64(PairArgs a, int slices)
{
    constexpr int NS = (SOFT ? 3 : 0) + (HARD ? 3 : 0);
    __shared__ double part[F64_WARPS][F64_SINKS][NS];
    __shared__ int64_t unit;
    if (a.st->code) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t ng = *a.ngroups;
    unsigned long long inter = 0;
    for (;;) {
        __syncthreads();   // the last unit's sums are read
        if (threadIdx.x == 0) unit = (int64_t)atomicAdd(a.counter, 1ull);
        __syncthreads();
        const int64_t g = unit / slices;
        if (g >= ng) break;
        const int slice = (int)(unit - g * slices);
        const uint32_t first = a.gfirst[g];
        const int n = (int)(a.gfirst[g + 1] - first);
        if (slice * F64_SINKS >= n) continue;
        const SysParams &P = a.sp[a.gsys[g]];
        const Eps2Fixed eps = eps2_fixed(P.eps2);
        const double R2 = P.R2, R2sq = P.R2sq, invdR = P.invdR;
        const Fixed R2f = to_fixed(R2sq);
        uint64_t c0 = 0, p0;
        int64_t Lc = 0, L;   // entries: cells [0, Lc), then particles [Lc, L)
        if (!NEAR) {
            c0 = a.off[g];
            Lc = (int64_t)(a.off[g + 1] - c0);
            p0 = a.off[ng + g];
            L = Lc + (int64_t)(a.off[ng + g + 1] - p0);
        } else {
            p0 = a.off[2 * ng + g];
            L = (int64_t)(a.off[2 * ng + g + 1] - p0);
        }
        if (slice == 0) inter += (unsigned long long)n * (unsigned long long)L;
        for (int r0 = slice * F64_SINKS; r0 < n; r0 += slices * F64_SINKS) {   // more than one round: leaves above n_crit
            const int rem = min(n - r0, F64_SINKS);
            const int lpc = rem <= 1 ? 1 : 1 << (32 - __clz(rem - 1));   // power of two >= rem
            const int copies = 32 / lpc, copy = lane / lpc, slot = lane & (lpc - 1);
            const double4_32a s = a.pd[first + r0 + min(slot, rem - 1)];
            double ax = 0.0, ay = 0.0, az = 0.0, bx = 0.0, by = 0.0, bz = 0.0;
            const int64_t step = F64_WARPS * copies;
            auto index = [&](int64_t e) -> uint32_t {
                return e < L ? (!NEAR && e < Lc ? a.list[c0 + e] : a.list[p0 + (uint64_t)(e - Lc)]) : 0u;
            };
            auto source = [&](int64_t e, uint32_t i) -> double4_32a {   // a massless copy of the sink past the end
                return e < L ? (!NEAR && e < Lc ? a.nD[i] : a.pd[i]) : make_double4_32a(s.x, s.y, s.z, 0.0);
            };
            int64_t e = w * copies + copy;
            // the source of the next pair and the index of the one after it are on their way during a pair
            uint32_t i1 = index(e + step);
            double4_32a q1 = source(e, index(e));
            for (int64_t k = w * copies; k < L; k += step, e += step) {   // k: the same trip count on every lane
                const double4_32a q = q1;
                q1 = source(e + step, i1);
                i1 = index(e + 2 * step);
                const double dx = __dsub_rn(q.x, s.x), dy = __dsub_rn(q.y, s.y), dz = __dsub_rn(q.z, s.z);
                if (!NEAR) {
                    const double f = mass_over_r3(q.w, dx, dy, dz, eps);
                    ax = __fma_rn(f, dx, ax);
                    ay = __fma_rn(f, dy, ay);
                    az = __fma_rn(f, dz, az);
                } else {
                    Fixed r2f;
                    double r2u = 0.0;
                    const bool fixed = r2_fixed(dx, dy, dz, Eps2Fixed{0ull, 0, 0.0}, r2f);
                    bool in;   // r^2 < R2^2
                    if (fixed) {
                        in = r2f.k < R2f.k || (r2f.k == R2f.k && r2f.A < R2f.A);
                    } else {   // compared as integers (both are >= 0; NaN compares above)
                        r2u = __fma_rn(dx, dx, __fma_rn(dy, dy, __dmul_rn(dz, dz)));
                        in = __double_as_longlong(r2u) < __double_as_longlong(R2sq);
                    }
                    in = in && e < L;
                    const bool any_in = __any_sync(0xffffffffu, in);
                    if (!SOFT && !any_in) continue;
                    const double f = mass_over_r3(q.w, dx, dy, dz, eps);
                    double K = 0.0;
                    if (any_in) {   // Eq. (10); 0 outside R2
                        const double r = fixed ? sqrt_fixed(r2f) : (r2u == 0.0 ? 0.0 : sqrt(r2u));
                        const double Y = __dmul_rn(__dsub_rn(R2, r), invdR);
                        const double Y2 = __dmul_rn(Y, Y);
                        K = __dmul_rn(__dmul_rn(Y2, __dmul_rn(Y2, Y2)),
                                      __fma_rn(Y2, __fma_rn(Y2, 6.0, -15.0), 10.0));
                        K = __double2hiint(Y) >= 0x3ff00000 ? 1.0 : K;   // Y >= 1
                        K = in && __double2hiint(Y) >= 0 ? K : 0.0;      // Y >= 0
                    }
                    if (SOFT) {
                        const double fs = any_in ? __dmul_rn(f, __dsub_rn(1.0, K)) : f;
                        ax = __fma_rn(fs, dx, ax);
                        ay = __fma_rn(fs, dy, ay);
                        az = __fma_rn(fs, dz, az);
                    }
                    if (HARD && any_in) {
                        const double fh = __dmul_rn(f, K);
                        bx = __fma_rn(fh, dx, bx);
                        by = __fma_rn(fh, dy, by);
                        bz = __fma_rn(fh, dz, bz);
                    }
                }
            }
            for (int o = lpc; o < 32; o <<= 1) {
                if (SOFT) {
                    ax += __shfl_xor_sync(0xffffffffu, ax, o);
                    ay += __shfl_xor_sync(0xffffffffu, ay, o);
                    az += __shfl_xor_sync(0xffffffffu, az, o);
                }
                if (HARD) {
                    bx += __shfl_xor_sync(0xffffffffu, bx, o);
                    by += __shfl_xor_sync(0xffffffffu, by, o);
                    bz += __shfl_xor_sync(0xffffffffu, bz, o);
                }
            }
            if (r0 != slice * F64_SINKS) __syncthreads();   // the last round's sums are read
            if (copy == 0) {
                double *o = part[w][slot];
                if (SOFT) {
                    o[0] = ax;
                    o[1] = ay;
                    o[2] = az;
                }
                if (HARD) {
                    o[NS - 3] = bx;
                    o[NS - 2] = by;
                    o[NS - 1] = bz;
                }
            }
            __syncthreads();
            if (threadIdx.x < rem * NS) {
                const int k = threadIdx.x / NS, d = threadIdx.x - k * NS;
                double v = part[0][k][d];
                for (int u = 1; u < F64_WARPS; ++u) v += part[u][k][d];
                v *= P.G;
                const uint32_t i = first + r0 + k;
                if (SOFT && d < 3) {
                    double *o = (double *)a.as[d];
                    o[i] = NEAR ? o[i] + v : v;   // near: the far kernel ran first on the same stream
                } else {
                    ((double *)a.ah[HARD && SOFT ? d - 3 : d])[i] = v;
                }
            }
        }
    }
    if (threadIdx.x == 0) atomicAdd(NEAR ? a.inter_hard : a.inter_soft, inter);
}

void fill_args(hybrid_ctx *c, PairArgs &a)
{
    a.ngroups = (const int64_t *)c->ngroups_dev.p;
    a.gfirst = (const uint32_t *)c->gfirst.p;
    a.gsys = (const uint32_t *)c->gsys.p;
    a.sp = (const SysParams *)c->sp_dev.p;
    a.off = (const uint64_t *)c->lcnt.p;
    a.list = (const uint32_t *)c->list.p;
    a.phi = (const float4 *)c->phi.p;
    a.plo = (const float4 *)c->plo.p;
    a.nA = (const float4 *)c->nA.p;
    a.nB = (const float4 *)c->nB.p;
    a.pd = (const double4_32a *)c->pd.p;
    a.nD = (const double4_32a *)c->nD.p;
    for (int d = 0; d < 3; ++d) {
        a.as[d] = c->acc_s[d].p;
        a.ah[d] = c->acc_h[d].p;
    }
    unsigned long long *ctr = (unsigned long long *)c->counter.p;
    a.counter = ctr + 2;   // + 1 for the near kernels
    a.inter_soft = ctr + 6;
    a.inter_hard = ctr + 7;
    a.st = status_dev(c);
    a.items = nullptr;
    a.nwork = nullptr;
    a.dense_items = nullptr;
    a.dense_counter = nullptr;
    a.want_soft = a.want_hard = 0;
}

// Far kernel: sinks per lane KS = ceil(n_crit / threads_per_group): 1, 2, 4 or
// 8; the default is 4 (one shared-memory read feeds 4 interactions). Staging
// depth: tile_depth (2, 3 or 4; 0 = 3).
int sinks_per_lane(const hybrid_ctx *c)
{
    const int ks = c->p.threads_per_group > 0 ? (c->p.n_crit + c->p.threads_per_group - 1) / c->p.threads_per_group : 4;
    return ks <= 1 ? 1 : (ks <= 2 ? 2 : (ks <= 4 ? 4 : 8));
}

template <int KS>
void go_far(hybrid_ctx *c, const PairArgs &a)
{
    const int depth = c->p.tile_depth == 0 ? 3 : c->p.tile_depth;
    if (depth == 2) k_far<KS, 2><<<c->nsm * 16, PAIR_THREADS, 0, c->st>>>(a);
    else if (depth == 4) k_far<KS, 4><<<c->nsm * 16, PAIR_THREADS, 0, c->st>>>(a);
    else k_far<KS, 3><<<c->nsm * 16, PAIR_THREADS, 0, c->st>>>(a);
}

// Counters and FP32 sums of the next far (soft sums) or near (hard sums) launch to zero.
__global__ void __launch_bounds__(256) k_clear_pairs(PairArgs a, bool near, int bits, int64_t N, int prec)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.counter = 0ull;
        if (near) a.counter[5] = 0ull;   // the dense near kernel's
        *(near ? a.inter_hard : a.inter_soft) = 0ull;
    }
    void *const *acc = near ? a.ah : a.as;
    if (prec == 1 && (!near || (bits & 2)))
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
            for (int d = 0; d < 3; ++d) ((float *)acc[d])[i] = 0.0f;
}

// near = false: cells and far particles (soft); near = true: near particles
// (soft and/or hard per mode bits)
void launch_pairs(hybrid_ctx *c, bool near, int mode)
{
    PairArgs a;
    fill_args(c, a);
    a.want_soft = mode & 1;
    a.want_hard = (mode >> 1) & 1;
    if (near) a.counter += 1;
    // the walk clears the counters and sums of the pair kernels after it; a near launch without a walk of its own
    // (reused lists) clears them here
    const int bits = near ? mode & 3 : 1;
    const bool clean = (c->pairs_clean & bits) == bits;
    c->pairs_clean &= near ? 0 : ~0;
    if (!clean) {
        k_clear_pairs<<<(int)std::min<int64_t>((c->N + 255) / 256, (int64_t)c->nsm * 8), 256, 0, c->st>>>(
            a, near, bits, c->N, c->p.precision);
        c->launches++;
    }
    const int kind = near ? PROF_HARD : PROF_SOFT;
    cudaEvent_t e0 = nullptr;
    prof_begin(c, kind, &e0);
    if (c->p.precision == 0) {
        // a unit for each slice of F64_SINKS sinks a group of n_crit can have (32 slices at most: larger groups take
        // rounds); units past a group's size are passed over
        // (no sum that overflows: n_crit may be anything up to 2^31 - 1, and 0 or fewer slices would never end)
        const int slices = std::min(32, (c->p.n_crit - 1) / F64_SINKS + 1);
        const int grid = c->nsm * 16;
        if (!near) k_pair_f64<false, true, false><<<grid, 32 * F64_WARPS, 0, c->st>>>(a, slices);
        else if (a.want_soft && a.want_hard) k_pair_f64<true, true, true><<<grid, 32 * F64_WARPS, 0, c->st>>>(a, slices);
        else if (a.want_soft) k_pair_f64<true, true, false><<<grid, 32 * F64_WARPS, 0, c->st>>>(a, slices);
        else k_pair_f64<true, false, true><<<grid, 32 * F64_WARPS, 0, c->st>>>(a, slices);
        c->launches++;
    } else {
        // work items written by the one-pass walk: far ones in wmap, near ones in wnear
        a.items = (const WorkItem *)(near ? c->wnear.p : c->wmap.p);
        a.nwork = (const uint64_t *)c->counter.p + (near ? 12 : 11);
        if (!near) {
            const int ks = sinks_per_lane(c);
            if (ks == 1) go_far<1>(c, a);
            else if (ks == 2) go_far<2>(c, a);
            else if (ks == 4) go_far<4>(c, a);
            else go_far<8>(c, a);
        } else {
            a.dense_counter = a.counter + 5;
            a.dense_items = a.items + c->capWork;
            const int grid = c->nsm * NEAR_MIN_BLOCKS;
            if (a.want_soft && a.want_hard) k_near<true, true><<<grid, PAIR_THREADS, 0, c->st>>>(a);
            else if (a.want_soft) k_near<true, false><<<grid, PAIR_THREADS, 0, c->st>>>(a);
            else k_near<false, true><<<grid, PAIR_THREADS, 0, c->st>>>(a);
        }
        c->launches += 1;
    }
    prof_end(c, kind, e0);
}

}  // namespace

void launch_pair_far(hybrid_ctx *c) { launch_pairs(c, false, 1); }

namespace {
template <typename K>
cudaError_t prefer_shared(K *kernel)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
}
}  // namespace

// The pair kernels are limited by registers and by shared memory per block:
// the whole carveout goes to shared memory (they read nothing through L1
// twice), so shared memory never limits their blocks per SM below registers.
cudaError_t init_pair_kernels()
{
    cudaError_t e = cudaSuccess;
    for (cudaError_t r : {prefer_shared(k_far<1, 2>), prefer_shared(k_far<1, 3>), prefer_shared(k_far<1, 4>),
                          prefer_shared(k_far<2, 2>), prefer_shared(k_far<2, 3>), prefer_shared(k_far<2, 4>),
                          prefer_shared(k_far<4, 2>), prefer_shared(k_far<4, 3>), prefer_shared(k_far<4, 4>),
                          prefer_shared(k_far<8, 2>), prefer_shared(k_far<8, 3>), prefer_shared(k_far<8, 4>),
                          prefer_shared(k_near<true, true>), prefer_shared(k_near<true, false>),
                          prefer_shared(k_near<false, true>)})
        if (e == cudaSuccess) e = r;
    return e;
}
void launch_pair_near(hybrid_ctx *c, int mode) { launch_pairs(c, true, mode); }

}  // namespace hy
