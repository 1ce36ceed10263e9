// tree.cu -- octree construction on the device (Sec. III-A1 of the paper,
// done on the GPU instead of the host): root cube, Morton keys, their stable
// order (a sample sort with the last build's keys as splitters, or an LSD radix
// sort) with the particle data gathered into it, the octree of all levels at
// once (a cell with more than n_leaf particles splits into its non-empty
// octants) with the sink groups, and cell moments (Sec. II-B: mass, centre of
// mass; Eq. 5-6: b_max, B2, MAC radius).
//
// All systems of a batch are processed by the same launches; every node,
// particle range, bucket and radix tile stays inside one system.
#include "hy_internal.cuh"
#include "root_box.cuh"

#include <cuda/atomic>
#include <cstdio>
#include <type_traits>

namespace hy {

namespace {

__device__ __forceinline__ void fail(Status *st, int code, int where)
{
    // the first failure wins and keeps its op index: later kernels of the same sequence may fail too (a build
    // after an unsorted one), and the sequence resumes at the first
    if (atomicCAS(&st->code, 0, code) == 0) st->where = where;
}

// Root cubes and the sample sort's start (see root_box.cuh) of a state that no drift of this sequence has moved.
__global__ void __launch_bounds__(256) k_box(const double *__restrict__ x, const double *__restrict__ y,
                                             const double *__restrict__ z, const Chunk *__restrict__ chunks,
                                             int nchunks, BoxArgs b)
{
    // the sort always runs, whatever the status: later kernels rely on a consistent permutation
    begin_sort(b);
    for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
        const Chunk ch = chunks[c];
        Bounds v;
        for (int i = threadIdx.x; i < ch.len; i += blockDim.x) {
            const int64_t k = ch.start + i;
            v.add(x[k], y[k], z[k]);
        }
        v.reduce_block(b, ch.sys);
    }
    finish_boxes(b);
}

// ---------------------------------------------------------------------------
// Morton keys: q = clamp(floor((x - lo) * scale), 0, 2^21 - 1) per axis, bits
// interleaved from the top, x first. Only the subtraction rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t spread3(uint32_t v)
{
    uint64_t x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x1f00000000ffffull;
    x = (x | (x << 16)) & 0x1f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// d = p - lo rounds once (FP64); the scale is a power of two 2^s, so
// floor(d 2^s) is taken from the bits of d (d = m 2^e with an integer m):
// m shifted by e + s, which keeps the FP64 pipe to one operation per axis.
__device__ __forceinline__ uint32_t cell_coord(double p, double lo, int s)
{
    const double d = __dsub_rn(p, lo);
    if (!(d > 0.0)) return 0u;   // zero, or below the root corner
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
    const int E = (int)((bits >> 52) & 0x7ffu);
    const unsigned long long frac = bits & ((1ull << 52) - 1ull);
    const unsigned long long m = E ? (frac | (1ull << 52)) : frac;
    const int sh = (E ? E : 1) - 1075 + s;   // d 2^s = m 2^sh
    constexpr unsigned long long QMAX = (1ull << LEVELS) - 1ull;
    unsigned long long q;
    if (sh >= 0) q = sh >= 11 ? QMAX : min(m << sh, QMAX);   // m >= 2^52 when normal: past the clamp
    else q = -sh >= 64 ? 0ull : (m >> -sh);
    return (uint32_t)min(q, QMAX);
}

// exponent s of a scale that is an exact power of two (normal)
__device__ __forceinline__ int pow2_exponent(double scale)
{
    return (int)(((unsigned long long)__double_as_longlong(scale) >> 52) & 0x7ffu) - 1023;
}

__global__ void __launch_bounds__(256) k_keys(int64_t N, const double *__restrict__ x, const double *__restrict__ y,
                                              const double *__restrict__ z, const int32_t *__restrict__ psys, int S,
                                              const SysBox *__restrict__ box, uint64_t *__restrict__ key,
                                              uint32_t *__restrict__ val)
{
    // the sort always runs, whatever the status: later kernels rely on a consistent permutation
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const SysBox &b = box[S == 1 ? 0 : psys[i]];
        const int es = pow2_exponent(b.scale);
        const uint32_t qx = cell_coord(x[i], b.lo[0], es);
        const uint32_t qy = cell_coord(y[i], b.lo[1], es);
        const uint32_t qz = cell_coord(z[i], b.lo[2], es);
        key[i] = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
        val[i] = (uint32_t)i;
    }
}

// ---------------------------------------------------------------------------
// Stable LSD radix sort, 8-bit digits, one launch per digit.
// k_digit_counts counts, per system, the digits of all eight passes. Pass p
// runs k_onesweep: tiles (chunks of at most ctx->tile keys inside one system)
// are claimed in order from a ticket counter; a tile ranks its keys (stable:
// warp-striped input order), publishes its per-digit counts, then adds up
// the counts of the earlier tiles of its system by reading their published
// words backwards until it meets an inclusive prefix (a chained scan with
// look-back), and publishes its own inclusive prefix. A key's destination is
// the system's start + the system's count of smaller digits + the earlier
// tiles' count of its digit + its rank in the tile; the tile is reordered in
// shared memory by (digit, rank) first, so that consecutive threads write
// consecutive addresses of one digit's run. Tiles only wait on tiles
// with smaller tickets, which were claimed by running blocks and publish
// their counts before they wait on anything; every wait is bounded.
// ---------------------------------------------------------------------------
constexpr uint32_t LB_AGG = 1u << 30, LB_INC = 2u << 30, LB_CNT = (1u << 30) - 1u;
constexpr int LB_SPIN_MAX = 1 << 22;
// sort scratch layout (u32): [0, 64) tickets, then counts[S][8][256], then look[8][nchunks][256]
constexpr int RS_HDR = 64;

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u32(uint32_t *p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Polls *q until one of the flag bits is set, at most max_polls times with a
// short sleep in between; when the polls run out it records HYBRID_ETIMEOUT in
// the status block and returns dflt, so the caller finishes without waiting.
__device__ __forceinline__ uint32_t wait_flagged(const uint32_t *q, uint32_t flags, int max_polls, Status *st,
                                                 uint32_t dflt)
{
    uint32_t v = ld_relaxed_u32(q);
    for (int spins = 0; (v & flags) == 0u; ++spins) {
        if (spins >= max_polls) {
            fail(st, HYBRID_ETIMEOUT, -1);
            return dflt;
        }
        __nanosleep(64);
        v = ld_relaxed_u32(q);
    }
    return v;
}

// Self-test of the bounded wait: one thread waits for a flag that nothing sets.
__global__ void k_wait_selftest(const uint32_t *word, int max_polls, Status *st)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) (void)wait_flagged(word, 1u, max_polls, st, 0u);
}

__global__ void __launch_bounds__(256) k_digit_counts(const uint64_t *__restrict__ key, const Chunk *__restrict__ chunks,
                                                      int nchunks, uint32_t *__restrict__ counts)
{
    __shared__ uint32_t h[8][256];
    const int lane = threadIdx.x & 31;
    const unsigned ltmask = (1u << lane) - 1u;
    for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
        const Chunk ch = chunks[c];
        for (int t = threadIdx.x; t < 8 * 256; t += blockDim.x) (&h[0][0])[t] = 0;
        __syncthreads();
        for (int i0 = 0; i0 < ch.len; i0 += blockDim.x) {
            const int i = i0 + threadIdx.x;
            const bool ok = i < ch.len;
            const uint64_t k = ok ? key[ch.start + i] : 0ull;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const uint32_t d = ok ? (uint32_t)(k >> (8 * p)) & 0xffu : 256u;
                const unsigned peers = __match_any_sync(0xffffffffu, d);
                if (ok && (peers & ltmask) == 0u) atomicAdd(&h[p][d], (uint32_t)__popc(peers));
            }
        }
        __syncthreads();
        uint32_t *dst = counts + (size_t)ch.sys * 2048;
        for (int t = threadIdx.x; t < 2048; t += blockDim.x) {
            const uint32_t v = (&h[0][0])[t];
            if (v) atomicAdd(dst + t, v);
        }
        __syncthreads();
    }
}

template <int IPT>
__global__ void __launch_bounds__(256) k_onesweep(const uint64_t *__restrict__ kin, const uint32_t *__restrict__ vin,
                                                  uint64_t *__restrict__ kout, uint32_t *__restrict__ vout,
                                                  const Chunk *__restrict__ chunks, int nchunks, int pass,
                                                  const uint32_t *__restrict__ counts, uint32_t *look,
                                                  uint32_t *ticket, int64_t ntotal, Status *st)
{
    // the sort always runs (later kernels rely on a consistent permutation); st only records a timeout
    constexpr int TILE_K = RS_WARPS * 32 * IPT;
    __shared__ uint32_t whist[RS_WARPS][256];
    __shared__ uint32_t base[256];    // global position of the tile's first key of digit d
    __shared__ uint32_t tloc[256];    // position in the tile's sorted order of its first key of digit d
    __shared__ uint64_t wsum[RS_WARPS];
    __shared__ uint64_t skey[TILE_K];
    __shared__ uint32_t sval[TILE_K];
    __shared__ int cid;
    const int shift = 8 * pass;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned ltmask = (1u << lane) - 1u;
    for (;;) {
        if (threadIdx.x == 0) cid = (int)atomicAdd(ticket, 1u);
        for (int t = threadIdx.x; t < RS_WARPS * 256; t += blockDim.x) (&whist[0][0])[t] = 0;
        __syncthreads();
        const int c = cid;
        if (c >= nchunks) break;
        const Chunk ch = chunks[c];
        uint64_t k[IPT];
        uint32_t v[IPT], r[IPT];
        const int wbase = w * 32 * IPT;
#pragma unroll
        for (int it = 0; it < IPT; ++it) {   // every load in flight before the ranking starts
            const int li = wbase + it * 32 + lane;   // warp-striped: (it, lane) is input order
            const bool ok = li < ch.len;
            k[it] = ok ? kin[ch.start + li] : 0ull;
            v[it] = ok ? vin[ch.start + li] : 0u;
        }
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const int li = wbase + it * 32 + lane;
            const bool ok = li < ch.len;
            const uint32_t d = ok ? (uint32_t)(k[it] >> shift) & 0xffu : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = ok ? whist[w][d] : 0u;
            __syncwarp();
            if (ok && (peers & ltmask) == 0u) whist[w][d] = before + (uint32_t)__popc(peers);
            __syncwarp();
            r[it] = before + (uint32_t)__popc(peers & ltmask);
        }
        __syncthreads();
        const int d = threadIdx.x;
        // loads that do not depend on the look-back go out before it
        const uint32_t cd = counts[(size_t)ch.sys * 2048 + pass * 256 + d];
        const int64_t s0 = chunks[ch.first_chunk].start;
        uint32_t run = 0;   // tile count of digit d; whist becomes the exclusive prefix over the warps
        for (int ww = 0; ww < RS_WARPS; ++ww) {
            const uint32_t cnt = whist[ww][d];
            whist[ww][d] = run;
            run += cnt;
        }
        uint32_t *mine = look + (size_t)c * 256 + d;
        const bool first = (c == ch.first_chunk);
        st_relaxed_u32(mine, (first ? LB_INC : LB_AGG) | run);
        uint32_t excl = 0;
        if (!first) {
            for (int j = c - 1; j >= ch.first_chunk; --j) {
                const uint32_t *q = look + (size_t)j * 256 + d;
                const uint32_t vq = wait_flagged(q, LB_AGG | LB_INC, LB_SPIN_MAX, st, LB_INC);
                excl += vq & LB_CNT;
                if (vq & LB_INC) break;
            }
            st_relaxed_u32(mine, LB_INC | (excl + run));
        }
        // exclusive prefixes over digits, in one block scan: the system's counts (high 32 bits) and the
        // tile's counts (low 32 bits; at most 2048, so no carry crosses over)
        const uint64_t both = ((uint64_t)cd << 32) | run;
        uint64_t incl = both;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[w] = incl;
        __syncthreads();
        uint64_t wpre = 0;
        for (int ww = 0; ww < w; ++ww) wpre += wsum[ww];
        const uint64_t ex = wpre + incl - both;
        tloc[d] = (uint32_t)ex;
        base[d] = (uint32_t)(ex >> 32) + excl;
        __syncthreads();
        // reorder the tile in shared memory by (digit, rank), then write runs of equal digits
        // with consecutive threads on consecutive addresses
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const int li = wbase + it * 32 + lane;
            if (li < ch.len) {
                const uint32_t dd = (uint32_t)(k[it] >> shift) & 0xffu;
                const uint32_t lp = tloc[dd] + whist[w][dd] + r[it];
                skey[lp] = k[it];
                sval[lp] = v[it];
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const int lp = it * 256 + threadIdx.x;
            if (lp < ch.len) {
                const uint64_t kk = skey[lp];
                const uint32_t dd = (uint32_t)(kk >> shift) & 0xffu;
                const int64_t dst = s0 + (int64_t)(base[dd] + ((uint32_t)lp - tloc[dd]));
                if (dst < ntotal) {   // always true unless a look-back timed out (recorded in st)
                    kout[dst] = kk;
                    vout[dst] = sval[lp];
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Sample sort of the keys, for a state that is close to key order (the state
// stays in the order of the last build and moves by one drift in between).
// The stable order is the order of the composite (key, current index), so
// per system the last build's sorted keys at every SS_BUCKET-th position split
// the keys into nb buckets: particle i is tried in the bucket of its position
// (most are still there: two comparisons against keys a whole warp shares),
// then in buckets ever farther away, and its key and index are appended to the
// bucket's region (SS_CAP entries, fewer for a small system). One warp then
// sorts each bucket in registers (bitonic, by composite) and writes it to its
// place, the sum of the earlier buckets' counts. Keys end sorted in keys[0] with their source
// positions in vals[0], exactly as the radix sort leaves them. Splitters out
// of order (another batch's keys, a first build) only send every particle
// through one binary search, which gives the same bucket to equal composites
// and keeps buckets in order whatever the splitters are. A bucket of more than
// SS_CAP keys (a state far from key order) makes the build leave the order
// unchanged and record ST_SORT; that one build is then repeated with the radix
// sort, which leaves the splitters of the next. A system of at most SS_SMALL buckets takes splitters of its own instead
// (sort_small): a first build of it, or one after another system's, nearly
// always overflows, and the repetition cost more than the rest of the build
// (hybrid_build_tree of a new state: N = 600 203 -> 111 us, 4096 228 -> 151; with
// buckets of 4096 keys, which held any such system, 143 and 189).
// Two launches (four with the scan of many counts), each key written and read
// twice. Before: buckets of 1024 or
// 2048 keys, a splitter, a counting, a scan and a scatter launch, and a radix
// sort of each bucket in shared memory. Root box and key sort per soft step of
// 4 hard sub-steps (8 at 2^24): N = 4096 0.190 -> 0.079 ms, 2^17 0.222 ->
// 0.105, 2^20 0.61 -> 0.30, 2^24 12.4 -> 6.6 ms.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool comp_less(uint64_t ka, uint32_t va, uint64_t kb, uint32_t vb)
{
    return ka < kb || (ka == kb && va < vb);
}

// The key of every particle, its bucket, and its place in the bucket's region.
__global__ void __launch_bounds__(256) k_keys_append(int64_t N, const double *__restrict__ x,
                                                     const double *__restrict__ y, const double *__restrict__ z,
                                                     const int32_t *__restrict__ psys, int S,
                                                     const SysBox *__restrict__ box, const int64_t *__restrict__ off,
                                                     const SSys *__restrict__ ss, const uint64_t *__restrict__ old,
                                                     uint64_t *__restrict__ rk, uint32_t *__restrict__ rv,
                                                     uint32_t *__restrict__ cnt, uint32_t *flag, Status *st, int where)
{
    const int lane = threadIdx.x & 31;
    const bool ordered = flag[1] == 0u;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < N; i0 += stride) {
        const int64_t i = i0 + threadIdx.x;
        uint32_t b = ~0u, cap = 0u;
        bool small = false;
        uint64_t k = 0ull;
        int64_t region = 0;
        if (i < N) {
            const int sy = S == 1 ? 0 : psys[i];
            const SysBox &bx = box[sy];
            const int es = pow2_exponent(bx.scale);
            const uint32_t qx = cell_coord(x[i], bx.lo[0], es);
            const uint32_t qy = cell_coord(y[i], bx.lo[1], es);
            const uint32_t qz = cell_coord(z[i], bx.lo[2], es);
            k = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
            const SSys yy = ss[sy];
            const int64_t o = off[sy];
            // splitter j (1 <= j < nb) is the composite at position o + j SS_BUCKET of the last build
            auto above = [&](int j) {
                const int64_t p = o + (int64_t)j * SS_BUCKET;
                return !comp_less(k, (uint32_t)i, old[p], (uint32_t)p);
            };
            int lo = 0, hi = yy.nb;   // above(lo) (or lo = 0), not above(hi) (or hi = nb)
            if (ordered && hi > 1) {
                const int g = (int)(i - o) / SS_BUCKET;
                int step = 1;
                if (g == 0 || above(g)) {
                    lo = g;
                    while (lo + step < hi && above(lo + step)) {
                        lo += step;
                        step <<= 1;
                    }
                    hi = min(lo + step, hi);
                } else {
                    hi = g;
                    while (hi - step > 0 && !above(hi - step)) {
                        hi -= step;
                        step <<= 1;
                    }
                    lo = max(hi - step, 0);
                }
            }
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (above(mid)) lo = mid;
                else hi = mid;
            }
            b = (uint32_t)(yy.bbase + lo);
            cap = (uint32_t)yy.rcap;
            small = yy.nb <= SS_SMALL;
            region = yy.rbase + (int64_t)lo * yy.rcap;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, b);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if (b != ~0u && lane == leader) {
            base = atomicAdd(cnt + b, (uint32_t)__popc(peers));
            if (base + (uint32_t)__popc(peers) > cap) {
                atomicOr(flag, small ? 2u : 1u);
                if (!small) fail(st, ST_SORT, where);
            }
        }
        base = __shfl_sync(0xffffffffu, base, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
        if (b != ~0u && base < cap) {
            rk[region + base] = k;
            rv[region + base] = (uint32_t)i;
        }
    }
}

// Compare and exchange of registers r and r | j of a lane, over all r without bit j: ascending where up(r).
template <int R, int J, typename Up>
__device__ __forceinline__ void lane_step(uint64_t (&k)[R], uint32_t (&v)[R], Up &&up)
{
#pragma unroll
    for (int r = 0; r < R; ++r)
        if ((r & J) == 0) {
            const bool swap = comp_less(k[r | J], v[r | J], k[r], v[r]) == up(r);
            const uint64_t a = k[r], b = k[r | J];
            const uint32_t c = v[r], d = v[r | J];
            k[r] = swap ? b : a;
            k[r | J] = swap ? a : b;
            v[r] = swap ? d : c;
            v[r | J] = swap ? c : d;
        }
}
template <int R, int J, typename Up>
__device__ __forceinline__ void lane_steps(uint64_t (&k)[R], uint32_t (&v)[R], Up &&up)   // steps J, J / 2, .., 1
{
    lane_step<R, J>(k, v, up);
    if constexpr (J > 1) lane_steps<R, J / 2>(k, v, up);
}
template <int R, int SIZE>
__device__ __forceinline__ void lane_sorts(uint64_t (&k)[R], uint32_t (&v)[R])   // runs of SIZE, 2 SIZE, .., R / 2
{
    if constexpr (SIZE < R) {
        lane_steps<R, SIZE / 2>(k, v, [](int r) { return (r & SIZE) == 0; });
        lane_sorts<R, 2 * SIZE>(k, v);
    }
}

// Bitonic sort of 32 R composites by one warp, element lane R + r in register
// r. The steps between lanes are loops: unrolled, they are 50 to 140 KB of
// code, and fetching it took longer than running it once (k_ss_sort of 4096
// keys 62 us unrolled, 6.9 us looped; of 2^24 keys 2.15 ms and 0.33 ms).
template <int R>
__device__ __forceinline__ void warp_sort(uint64_t (&k)[R], uint32_t (&v)[R], int lane)
{
    lane_sorts<R, 2>(k, v);
#pragma unroll 1
    for (int lanes = 1; lanes <= 32; lanes <<= 1) {   // sorted runs of R x lanes
        const bool up = lanes == 32 || (lane & lanes) == 0;
#pragma unroll 1
        for (int m = lanes / 2; m >= 1; m >>= 1) {
            const bool low = ((lane & m) == 0) == up;   // this lane keeps the smaller one
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint64_t ok = __shfl_xor_sync(0xffffffffu, k[r], m);
                const uint32_t ov = __shfl_xor_sync(0xffffffffu, v[r], m);
                const bool take = comp_less(ok, ov, k[r], v[r]) == low;
                k[r] = take ? ok : k[r];
                v[r] = take ? ov : v[r];
            }
        }
        lane_steps<R, R / 2>(k, v, [up](int) { return up; });
    }
}

constexpr int SSB_THREADS = 128, SSB_WARPS = SSB_THREADS / 32;
constexpr int SS_PAD = SS_CAP + SS_CAP / 8;   // a bucket in shared memory, one entry of padding after every R

// n <= 32 R composites sorted by one warp (from global or shared memory).
template <int R>
__device__ __forceinline__ void sort_bucket(const uint64_t *rk, const uint32_t *rv, int n, uint64_t *k0, uint32_t *v0, uint64_t *sk,
                                      uint32_t *sv, int lane)
{
    uint64_t k[R];
    uint32_t v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {   // any order will do; slots past the run sort to the end
        const int e = r * 32 + lane;
        k[r] = e < n ? rk[e] : ~0ull;
        v[r] = e < n ? rv[e] : ~0u;
    }
    warp_sort<R>(k, v, lane);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        sk[lane * (R + 1) + r] = k[r];
        sv[lane * (R + 1) + r] = v[r];
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = r * 32 + lane;
        if (e < n) {
            k0[e] = sk[e + e / R];
            v0[e] = sv[e + e / R];
        }
    }
}

// The same, its code fetched once for all its callers: inlined three times in sort_small, a build of 600 new particles
// took 160 us, not 111. (The buckets' own sort is inlined: 2 us of a step of 2^17.)
template <int R>
__device__ __noinline__ void sort_run(const uint64_t *rk, const uint32_t *rv, int n, uint64_t *k0, uint32_t *v0, uint64_t *sk,
                                      uint32_t *sv, int lane)
{
    sort_bucket<R>(rk, rv, n, k0, v0, sk, sv, lane);
}

// A small system with an overflowed bucket, by the blocks that its buckets belong to, each by itself: keys made anew,
// splitters from the sorted keys of up to SS_SAMPLE of its particles, the block's buckets gathered from all of them, and
// their place from the number of keys before them. A bucket that overflows again sends the build to the radix sort.
constexpr int SS_SAMPLE = 256;
struct SmallArgs {
    const double *x, *y, *z;
    const SysBox *box;
    const int64_t *off;
    Status *st;
    int where;
};
struct SortMem {
    uint64_t k[SSB_WARPS][SS_PAD];   // a bucket per warp
    uint32_t v[SSB_WARPS][SS_PAD];
    uint64_t sk[SS_SAMPLE];          // the sample of a small system
    uint32_t sv[SS_SAMPLE];
    uint32_t cnt[SSB_WARPS + 1];     // keys of the block's buckets; before them
};

__device__ __noinline__ void sort_small(const SmallArgs &a, int s, const SSys &y, int b0, uint32_t *flag,
                                        uint64_t *__restrict__ k0, uint32_t *__restrict__ v0, SortMem &m)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t o = a.off[s];
    const int n = (int)(a.off[s + 1] - o), M = min(n, SS_SAMPLE);
    const SysBox b = a.box[s];
    const int es = pow2_exponent(b.scale);
    auto composite = [&](int i, uint64_t &k, uint32_t &v) {
        k = (spread3(cell_coord(a.x[o + i], b.lo[0], es)) << 2) | (spread3(cell_coord(a.y[o + i], b.lo[1], es)) << 1) |
            spread3(cell_coord(a.z[o + i], b.lo[2], es));
        v = (uint32_t)(o + i);
    };
    if (threadIdx.x <= SSB_WARPS) m.cnt[threadIdx.x] = 0u;
    for (int e = threadIdx.x; e < M; e += SSB_THREADS) composite(e * n / M, m.k[0][e], m.v[0][e]);
    __syncthreads();
    if (w == 0) sort_run<SS_SAMPLE / 32>(m.k[0], m.v[0], M, m.sk, m.sv, m.k[0], m.v[0], lane);
    __syncthreads();
    const int j0 = max(0, b0 - y.bbase), J = min(y.nb, b0 + SSB_WARPS - y.bbase) - j0;   // this block's buckets
    uint64_t ck[SSB_WARPS + 1];   // bucket q: composites from splitter q up to splitter q + 1
    uint32_t cv[SSB_WARPS + 1];
#pragma unroll
    for (int q = 0; q <= SSB_WARPS; ++q) {
        const int j = j0 + q;
        ck[q] = j == 0 ? 0ull : (j < y.nb ? m.sk[j * M / y.nb] : ~0ull);
        cv[q] = j == 0 ? 0u : (j < y.nb ? m.sv[j * M / y.nb] : ~0u);
    }
    for (int i = threadIdx.x; i < n; i += SSB_THREADS) {
        uint64_t k;
        uint32_t v;
        composite(i, k, v);
        int q = -1;
#pragma unroll
        for (int u = 0; u <= SSB_WARPS; ++u) q += comp_less(k, v, ck[u], cv[u]) ? 0 : 1;
        if (q < 0) {
            atomicAdd(m.cnt + SSB_WARPS, 1u);
        } else if (q < J) {
            const uint32_t at = atomicAdd(m.cnt + q, 1u);
            if (at < (uint32_t)SS_CAP) {
                m.k[q][at] = k;
                m.v[q][at] = v;
            }
        }
    }
    __syncthreads();
    if (w < J) {
        const int c = (int)m.cnt[w];
        uint32_t s0 = (uint32_t)o + m.cnt[SSB_WARPS];
        for (int q = 0; q < w; ++q) s0 += m.cnt[q];
        if (c > SS_CAP) {
            if (lane == 0) {
                atomicOr(flag, 1u);
                fail(a.st, ST_SORT, a.where);
            }
        } else if (c > 256) {
            sort_run<SS_CAP / 32>(m.k[w], m.v[w], c, k0 + s0, v0 + s0, m.k[w], m.v[w], lane);
        } else {
            sort_run<8>(m.k[w], m.v[w], c, k0 + s0, v0 + s0, m.k[w], m.v[w], lane);
        }
    }
    __syncthreads();   // the buckets and counts are used
}

// One warp per bucket. SCANNED: cnt holds the exclusive sums of the counts (nbk + 1 entries), else the counts,
// which each block adds up itself. rcap: entries of a region of a single system.
template <bool SCANNED>
__global__ void __launch_bounds__(SSB_THREADS, 4) k_ss_sort(int nbk, int S, int rcap, const SSys *__restrict__ ss,
                                                            const uint32_t *__restrict__ bsys,
                                                            const uint32_t *__restrict__ cnt,
                                                            const uint64_t *__restrict__ rk,
                                                            const uint32_t *__restrict__ rv, uint64_t *__restrict__ k0,
                                                            uint32_t *__restrict__ v0, uint32_t *flag,
                                                            const __grid_constant__ SmallArgs small)
{
    __shared__ SortMem m;
    __shared__ uint32_t wsum[SSB_WARPS];
    const uint32_t fl = *flag;
    if (fl & 1u) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // whether a small system has an overflowed bucket, by a whole warp
    auto overflowed = [&](const SSys &y) -> bool {
        const int b = y.bbase + lane;
        const bool on = y.nb <= SS_SMALL && lane < y.nb;
        return __any_sync(0xffffffffu, on && (SCANNED ? cnt[b + 1] - cnt[b] : cnt[b]) > (uint32_t)y.rcap);
    };
    for (int b0 = blockIdx.x * SSB_WARPS; b0 < nbk; b0 += gridDim.x * SSB_WARPS) {
        const int b = b0 + w;
        uint32_t s0, n;
        if (SCANNED) {
            s0 = b < nbk ? cnt[b] : 0u;
            n = b < nbk ? cnt[b + 1] - s0 : 0u;
        } else {
            uint32_t sum = 0;
            for (int k = threadIdx.x; k < b0; k += SSB_THREADS) sum += cnt[k];
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (lane == 0) wsum[w] = sum;
            __syncthreads();
            s0 = 0;
            for (int k = 0; k < SSB_WARPS; ++k) s0 += wsum[k];
            for (int k = b0; k < min(b, nbk); ++k) s0 += cnt[k];
            n = b < nbk ? cnt[b] : 0u;
            __syncthreads();
        }
        if (n > 0u) {   // the whole warp
            int64_t region = (int64_t)b * rcap;   // a single system's regions are known without a load
            if (S > 1) {
                const SSys y = ss[bsys[b]];
                region = y.rbase + (int64_t)(b - y.bbase) * y.rcap;
            }
            const uint64_t *kb = rk + region;
            const uint32_t *vb = rv + region;
            if ((fl & 2u) && overflowed(ss[S == 1 ? 0u : bsys[b]])) {
                // below
            } else if (n <= 256u) {
                sort_bucket<8>(kb, vb, (int)n, k0 + s0, v0 + s0, m.k[w], m.v[w], lane);
            } else {
                sort_bucket<SS_CAP / 32>(kb, vb, (int)n, k0 + s0, v0 + s0, m.k[w], m.v[w], lane);
            }
        }
        if (fl & 2u) {
            __syncthreads();
            const int last = min(b0 + SSB_WARPS, nbk) - 1;
            for (int s = S == 1 ? 0 : (int)bsys[b0]; s <= (S == 1 ? 0 : (int)bsys[last]); ++s) {
                const SSys y = ss[s];
                if (overflowed(y)) sort_small(small, s, y, b0, flag, k0, v0, m);
            }
        }
    }
}

// Gather of the state into key order; also writes the pair-kernel copies of
// the positions: FP32 hi/lo split (x = hi + lo to ~2^-48) or FP64 double4_32a.
struct PermArgs {
    const double *xin[7];
    double *xout[7];
    const int32_t *id_in;
    int32_t *id_out;
    const int32_t *orig_in;
    int32_t *orig_out;
    const uint32_t *src;
    float4 *phi, *plo;
    double4_32a *pd;
    float *disp;          // zeroed: distance moved since this build (reused lists), or null
    const int32_t *psys;
    const SysBox *box;
    int64_t N;
    unsigned long long *bmin, *bmax;   // reset for the next build (the root cubes are made)
    int S;
    uint32_t *flag;       // [0] bit 0: an overflowed sample sort: the order stays; [1] reset for the next build
};

// MINB blocks per SM: 8 (32 registers) for batches above 2^18 particles, where the gathers' bandwidth counts (2^24:
// tree build 30.1 -> 28.7 ms per soft step against 64 registers, 2^20 1.172 -> 1.138); below, a thread's loads all go
// out at once with 64 (2^12 and 2^17 2 and 1 % of the step faster). At 32 a thread spills about 270 bytes, out and in, in the
// grid-stride loop's body; they stay in L1: DRAM moves 153 + 184 MB for 2^21 particles (336 algorithmic) in 75 us.
template <int MINB>
__global__ void __launch_bounds__(256, MINB) k_permute(PermArgs a)
{
    // whatever the status: later kernels rely on a consistent permutation
    const bool keep = (a.flag[0] & 1u) != 0u;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < 3 * a.S; k += gridDim.x * blockDim.x) {
        a.bmin[k] = ~0ull;
        a.bmax[k] = 0ull;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a.flag[1] = 0u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.N; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t j = keep ? (uint32_t)i : a.src[i];
        double v[7];
#pragma unroll
        for (int f = 0; f < 7; ++f) {
            v[f] = a.xin[f][j];
            a.xout[f][i] = v[f];
        }
        if (a.id_in) a.id_out[i] = a.id_in[j];
        a.orig_out[i] = a.orig_in[j];
        if (a.phi) {
            const SysBox b = a.box[a.psys[i]];
            float h[3], l[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) grid_split(v[d], b.lo[d], b, h[d], l[d]);
            a.phi[i] = make_float4(h[0], h[1], h[2], narrow(v[6]));
            a.plo[i] = make_float4(l[0], l[1], l[2], 0.0f);
        }
        if (a.pd) a.pd[i] = make_double4_32a(v[0], v[1], v[2], v[6]);
        if (a.disp) a.disp[i] = 0.0f;
    }
}

// ---------------------------------------------------------------------------
// Octree topology and sink groups from the sorted keys, all levels at once, in
// two passes over the particles with one short scan between them (k_cells,
// scan, k_nodes), whatever the depth.
//
// c(i) = number of leading octal digits keys i-1 and i share (-1 at the first
// particle of a system): particle i starts a cell at every level l > c(i).
// The level-l cell around particle p holds more than n particles exactly when
// some n + 1 consecutive ones around p share l digits, so the deepest such
// level is L_n(p) = max over a in [p - n, p] of the digits that keys a and
// a + n share: a sliding maximum, taken by doubling in shared memory. The leaf
// depth is D(p) = L_n_leaf(p) + 1 (21 at most), and the sink group of p is its
// cell at level Dg(p) = min(D(p), L_n_crit(p) + 1).
//
// Particle i owns the nodes (l, first = i) for c(i) < l <= D(i). In
// breadth-first order (level, system, key) a node's index is the number of
// nodes at lower levels plus the number of level-l starts before i: counts per
// level and tile (k_cells), their scan, and ballots inside the tile (k_nodes)
// give it directly, and with it everything else: the parent of i's top node is
// the last start at level c(i); the node at level l that holds particle i-1
// ends at i when c(i) < l; its children end where the level l + 1 starts
// before i end. No node is searched for and nothing is sorted by level.
// Before, the sizes came from linear walks in shared memory, and records in
// particle order were sorted by level, searched for their ends and linked, and
// groups were flagged and compacted, by 14 more launches. Tree build per soft
// step of 4 hard sub-steps (8 at N = 2^24): N = 4096 0.56 -> 0.47 ms, 2^17
// 0.715 -> 0.595, 2^20 (absolute MAC) 1.84 -> 1.59, 2^24 43.3 -> 39.0 ms.
// ---------------------------------------------------------------------------
// c(i): common leading octal digits of keys i-1 and i; -1 at a system's first particle
__device__ __forceinline__ int shared_digits(uint64_t a, uint64_t b)
{
    const unsigned long long x = a ^ b;
    return x == 0ull ? LEVELS : (__clzll((long long)x) - 1) / 3;   // keys use bits 0..62
}
__device__ __forceinline__ int prefix_c(const uint64_t *__restrict__ key, const int32_t *__restrict__ psys, int64_t i)
{
    if (i == 0 || psys[i] != psys[i - 1]) return -1;
    return shared_digits(key[i - 1], key[i]);
}

// Tiles of CT_WARPS warps with ROWS rows of 32 particles each: 256, 512 or 1024 particles. Small systems take small
// tiles (more blocks, shorter ones), as long as the counts of all tiles are few enough for every block of k_nodes to
// add up by itself.
constexpr int CT_WARPS = 8;
constexpr int CT_MAX = CT_WARPS * 32 * 4;
constexpr int CT_SUM_MAX = 320;               // tiles up to which k_nodes adds up the counts; above, a scan does it
constexpr int NLEV = LEVELS + 1;              // levels 0..21
constexpr int CT_CNT = NLEV + 1;              // counts per tile: starts at each level, sink groups
// Sink groups of up to this size are marked in k_cells; larger n_crit take the node-based kernels
// (k_group_flag and on): the window costs one byte of shared memory per particle, twice.
constexpr int GROUP_WINDOW = 1024;

// deepest level at which the cell around tile particle x holds more than n particles, for every x of the
// tile (of len0), into m[0, len0) as level + 1 (0: none); m and t are byte arrays of cells_bytes(n) each
__host__ __device__ constexpr int cells_bytes(int n) { return (CT_MAX + n + 15) / 16 * 16 + 16; }

__device__ __forceinline__ uint8_t *window_max(const uint64_t *__restrict__ key, const int32_t *__restrict__ psys,
                                               bool one, int64_t N, int64_t b0, int len0, int n, uint8_t *m, uint8_t *t)
{
    const int len = len0 + n, words = (len + 3) / 4 + 1;
    for (int x = threadIdx.x; x < 4 * words; x += blockDim.x) {
        const int64_t a = b0 - n + x;
        int v = 0;
        if (x < len && a >= 0 && a + n < N && (one || psys[a] == psys[a + n])) v = shared_digits(key[a], key[a + n]) + 1;
        m[x] = (uint8_t)v;
    }
    __syncthreads();
    int s = 1;
    for (; 2 * s <= n + 1; s <<= 1) {   // m[x] = max over [x, x + s) -> [x, 2 s)
        const uint32_t *w = (const uint32_t *)m;
        for (int k = threadIdx.x; k < words; k += blockDim.x) {
            uint32_t o;
            if (s >= 4) o = k + s / 4 < words ? w[k + s / 4] : 0u;
            else o = __funnelshift_r(w[k], k + 1 < words ? w[k + 1] : 0u, 8 * s);
            ((uint32_t *)t)[k] = __vmaxu4(w[k], o);
        }
        __syncthreads();
        uint8_t *u = m;
        m = t;
        t = u;
    }
    // the window of n + 1 entries from x: two overlapping runs of s
    for (int x = threadIdx.x; x < len0; x += blockDim.x) t[x] = max(m[x], m[x + n + 1 - s]);
    __syncthreads();
    return t;
}

// Per particle the packed levels c + 1, D, Dg (5 bits each); per tile the numbers of nodes started at each level
// and of sink groups (cnt[row][tile]). Also clears the counters of the moments and of the walk.
template <int ROWS>
__global__ void __launch_bounds__(32 * CT_WARPS) k_cells(int64_t N, int S, const uint64_t *__restrict__ key,
                                                         const int32_t *__restrict__ psys, int n_leaf, int n_crit,
                                                         uint16_t *__restrict__ cells, int ntiles,
                                                         uint32_t *__restrict__ cnt, unsigned long long *counter,
                                                         const Status *st)
{
    if (st->code) return;
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ uint32_t wcnt[CT_WARPS][CT_CNT + 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nb = cells_bytes(max(n_leaf, n_crit));
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        constexpr int TILE_P = CT_WARPS * 32 * ROWS;
        const int64_t b0 = (int64_t)tile * TILE_P, p0 = b0 + w * (32 * ROWS) + lane;
        uint8_t D[ROWS], Dg[ROWS];
        const uint8_t *m = window_max(key, psys, S == 1, N, b0, TILE_P, n_leaf, sm, sm + nb);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) Dg[r] = D[r] = min((int)m[w * (32 * ROWS) + r * 32 + lane], LEVELS);
        if (n_crit > 0) {
            __syncthreads();
            m = window_max(key, psys, S == 1, N, b0, TILE_P, n_crit, sm, sm + nb);
#pragma unroll
            for (int r = 0; r < ROWS; ++r) Dg[r] = min(D[r], m[w * (32 * ROWS) + r * 32 + lane]);
        }
        uint32_t mine = 0;   // lane l: starts at level l (l < NLEV), lane NLEV: groups
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int64_t i = p0 + r * 32;
            int c = LEVELS + 1, d = 0;   // past the end: starts nothing
            bool g = false;
            if (i < N) {
                c = prefix_c(key, psys, i);
                d = D[r];
                g = n_crit > 0 && c < (int)Dg[r];
                cells[i] = (uint16_t)((c + 1) | (d << 5) | ((int)Dg[r] << 10));
            }
            const int lo = __reduce_min_sync(0xffffffffu, c) + 1, hi = __reduce_max_sync(0xffffffffu, d);
            for (int l = lo; l <= hi; ++l) {
                const uint32_t k = __popc(__ballot_sync(0xffffffffu, c < l && l <= d));
                if (lane == l) mine += k;
            }
            const uint32_t k = __popc(__ballot_sync(0xffffffffu, g));
            if (lane == NLEV) mine += k;
        }
        if (lane < CT_CNT) wcnt[w][lane] = mine;
        __syncthreads();
        if (threadIdx.x < CT_CNT) {
            uint32_t sum = 0;
            for (int k = 0; k < CT_WARPS; ++k) sum += wcnt[k][threadIdx.x];
            cnt[(size_t)threadIdx.x * ntiles + tile] = sum;
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        counter[9] = 0ull;                                       // chunk items of the moments
        counter[0] = counter[1] = 0ull;                          // the walk's groups,
        counter[10] = counter[11] = counter[12] = 0ull;          // list cursor and items
    }
}

struct NodeArgs {
    const uint16_t *cells;
    const int32_t *psys;
    const uint32_t *off;      // scanned counts: index of a tile's first start at each level, then of its first group
    const uint64_t *total;    // nodes + groups
    uint32_t *nfirst, *nend, *nlevel, *nchild, *nchend, *nparent, *sysroot, *lvl, *done;
    unsigned long long *bmax64;   // zeroed for the chunks' maxima, FP64 or FP32 form
    unsigned int *bmax32;         // (null: b_max by search)
    uint32_t *gnode, *gfirst, *gsys;   // null: groups come from the node-based kernels
    int64_t *ngroups;
    int64_t N, cap;
    int ntiles;
};

// Nodes (breadth-first) and sink groups (in particle order); see above.
template <int ROWS, bool SCANNED>
__global__ void __launch_bounds__(32 * CT_WARPS) k_nodes(NodeArgs a, Status *st, int where)
{
    if (st->code) return;
    __shared__ uint32_t wcnt[CT_WARPS][CT_CNT + 1];
    __shared__ uint32_t before[CT_CNT], start[CT_CNT + 1];   // counts of the earlier tiles; first index of a row
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    if (SCANNED) {
        if (threadIdx.x < CT_CNT) start[threadIdx.x] = a.off[(size_t)threadIdx.x * a.ntiles];
        if (threadIdx.x == 0) start[CT_CNT] = (uint32_t)*a.total;
        __syncthreads();
    } else {   // one tile per block
        for (int r = w; r < CT_CNT; r += CT_WARPS) {
            const uint32_t *row = a.off + (size_t)r * a.ntiles;
            uint32_t mine = 0, all = 0;
            for (int t = lane; t < a.ntiles; t += 32) {
                const uint32_t v = row[t];
                all += v;
                mine += t < (int)blockIdx.x ? v : 0u;
            }
            mine = __reduce_add_sync(0xffffffffu, mine);
            all = __reduce_add_sync(0xffffffffu, all);
            if (lane == 0) {
                before[r] = mine;
                wcnt[0][r] = all;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t run = 0;
            for (int r = 0; r < CT_CNT; ++r) {
                start[r] = run;
                run += wcnt[0][r];
            }
            start[CT_CNT] = run;
        }
        __syncthreads();
    }
    const uint32_t nodes = start[NLEV];   // start of the groups
    if ((int64_t)nodes > a.cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            fail(st, HYBRID_ECAPACITY, where);
            st->need[0] = (int64_t)nodes + (int64_t)(nodes >> 3) + 1024;
        }
        return;
    }
    if (blockIdx.x == 0) {
        if (threadIdx.x <= NLEV + 1) a.lvl[threadIdx.x] = threadIdx.x < NLEV ? start[threadIdx.x] : nodes;
        if (threadIdx.x == 0 && a.gnode) {
            const uint64_t ng = start[CT_CNT] - nodes;
            *a.ngroups = (int64_t)ng;
            a.gfirst[ng] = (uint32_t)a.N;
        }
    }
    for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        const int64_t p0 = (int64_t)tile * (CT_WARPS * 32 * ROWS) + w * (32 * ROWS) + lane;
        int c[ROWS], d[ROWS], dp[ROWS], dg[ROWS];   // dp: D of the particle before
        uint32_t mine = 0;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int64_t i = p0 + r * 32;
            c[r] = LEVELS + 1;
            d[r] = dp[r] = dg[r] = 0;
            if (i < a.N) {
                const int k = a.cells[i];
                c[r] = (k & 31) - 1;
                d[r] = (k >> 5) & 31;
                dg[r] = k >> 10;
            }
            if (i > 0 && i <= a.N) dp[r] = (a.cells[i - 1] >> 5) & 31;
            if (i == a.N) c[r] = -1;   // the end of the batch ends every cell around the last particle
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const bool real = p0 + r * 32 < a.N;
            const int lo = __reduce_min_sync(0xffffffffu, real ? c[r] : LEVELS + 1) + 1;
            const int hi = __reduce_max_sync(0xffffffffu, d[r]);
            for (int l = lo; l <= hi; ++l) {
                const uint32_t k = __popc(__ballot_sync(0xffffffffu, real && c[r] < l && l <= d[r]));
                if (lane == l) mine += k;
            }
            const uint32_t k = __popc(__ballot_sync(0xffffffffu, real && a.gnode && c[r] < dg[r]));
            if (lane == NLEV) mine += k;
        }
        if (lane < CT_CNT) wcnt[w][lane] = mine;
        __syncthreads();
        uint32_t base = 0;   // lane l: index of this warp's first start at level l; lane NLEV: of its first group
        if (lane < CT_CNT) {
            base = (SCANNED ? a.off[(size_t)lane * a.ntiles + tile] : start[lane] + before[lane]) - (lane == NLEV ? nodes : 0u);
            for (int k = 0; k < w; ++k) base += wcnt[k][lane];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int64_t i = p0 + r * 32;
            const bool real = i < a.N, here = i <= a.N;
            const unsigned gm = __ballot_sync(0xffffffffu, real && a.gnode && c[r] < dg[r]);
            const uint32_t g = __shfl_sync(0xffffffffu, base, NLEV) + __popc(gm & lt);
            const int sys = real ? a.psys[i] : 0;
            // levels: from the parent's (c) to one past the deepest node started or closed here
            const int lo = max(__reduce_min_sync(0xffffffffu, here ? c[r] : LEVELS + 1), 0);
            const int hi = __reduce_max_sync(0xffffffffu, max(d[r], dp[r])) + 1;
            uint32_t up = NONE;     // the node one level up: the parent of the next start
            uint32_t last = NONE;   // the node at level l - 1 that ends at i
            for (int l = lo; l <= hi; ++l) {
                const bool start = real && c[r] < l && l <= d[r];
                const unsigned m = __ballot_sync(0xffffffffu, start);
                const uint32_t x = __shfl_sync(0xffffffffu, base, l) + __popc(m & lt);   // starts before i at this level
                if (lane == l) base += __popc(m);
                if (last != NONE) a.nchend[last] = x;
                last = NONE;
                if (here && c[r] < l && l <= dp[r] && i > 0) {   // the cell of particle i - 1 ends
                    last = x - 1;
                    a.nend[last] = (uint32_t)i;
                }
                if (l == c[r]) up = x - 1;
                if (start) {
                    a.nfirst[x] = (uint32_t)i;
                    a.nlevel[x] = (uint32_t)l;
                    a.nparent[x] = up;
                    if (l > c[r] + 1) a.nchild[up] = x;
                    if (l == d[r]) a.nchild[x] = NONE;
                    a.done[x] = 0u;
                    if (a.bmax64) a.bmax64[x] = 0ull;
                    if (a.bmax32) a.bmax32[x] = 0u;
                    if (l == 0) a.sysroot[sys] = x;
                    if (l == dg[r] && ((gm >> lane) & 1u)) {
                        a.gnode[g] = x;
                        a.gfirst[g] = (uint32_t)i;
                        a.gsys[g] = (uint32_t)sys;
                    }
                    up = x;
                }
            }
            if (lane == NLEV) base += __popc(gm);
        }
    }
}

// ---------------------------------------------------------------------------
// Moments. A cell of at most MOM_CH particles sums its own particle range
// (one warp): M, centre of mass, B2 and b_max, with no wait on other cells.
// A larger cell is combined from its children by the last of them to finish
// (counted with an atomic; no wait anywhere): M = sum M_j, COM = sum M_j
// COM_j / M, B2 = sum_j [B2_j + M_j |COM_j - COM|^2] (parallel axis, no
// cancellation), in a fixed order. b_max of a larger cell is the largest
// distance of its particles to its centre of mass, taken afterwards (k_bmax_big or
// k_finish).
// ---------------------------------------------------------------------------
struct MomArgs {
    const uint32_t *lvl, *nfirst, *nend, *nchend, *nchild, *nparent, *nlevel;   // a node's particles and children: [first, end)
    const double *x, *y, *z, *m;
    const uint64_t *key;
    const int32_t *psys;
    int S;
    const SysBox *box;
    double *M, *cx, *cy, *cz, *B2;
    float4 *nA, *nB;
    uint32_t *done;
    const float4 *phi, *plo;
    unsigned long long *bmax64;   // FP64 form: b_max as FP64 bits
    unsigned int *bmax32;         // FP32 form: b_max as FP32 bits
    bool search;                  // FP32 form: b_max of the larger cells by search (k_finish), else by chunks (k_bmax_big)
};

__device__ __forceinline__ uint32_t digit_at(uint64_t key, int lev)
{
    return (uint32_t)(key >> (3 * (LEVELS - lev))) & 7u;
}

__device__ __forceinline__ void cell_geom(const SysBox &b, uint64_t key, uint32_t lev, double o[3], double *side)
{
    const double sd = ldexp(b.L, -(int)lev);
    // integer cell coordinate of the key prefix along each axis
    uint32_t q[3] = {0, 0, 0};
    for (uint32_t l = 1; l <= lev; ++l) {
        const uint32_t d = digit_at(key, (int)l);
        q[0] = (q[0] << 1) | ((d >> 2) & 1u);
        q[1] = (q[1] << 1) | ((d >> 1) & 1u);
        q[2] = (q[2] << 1) | (d & 1u);
    }
    for (int k = 0; k < 3; ++k) o[k] = __dadd_rn(b.lo[k], __dmul_rn((double)q[k], sd));
    *side = sd;
}

__device__ __forceinline__ void store_com(const MomArgs &a, uint32_t c, double M, double c0, double c1, double c2,
                                          double B2)
{
    a.M[c] = M;
    a.cx[c] = c0;
    a.cy[c] = c1;
    a.cz[c] = c2;
    a.B2[c] = B2;
}

// Moments straight from each cell's particle range, with no wait on the
// children: M, sum m (x - o) and Q = sum m |x - o|^2 with o = the cell's first
// particle; COM = o + sum m (x - o) / M and B2 = Q - M |COM - o|^2 (o lies
// inside the cell, so the subtraction loses little). Cells of at most MOM_CH
// particles: one warp each (at most 4 rounds of loads per lane). Larger cells: chunks of MOM_CH particles, one warp
// per chunk, then one warp per cell adds the chunk sums in chunk order.
constexpr uint32_t MOM_CH = 128;

struct MomSums {
    double M, sx, sy, sz, Q;
};

// FP32 form: offsets from the first particle from the hi/lo copies (hi parts
// on a common grid, so hi_i - hi_f is exact), sums of at most MOM_CH terms in
// FP32; the chunk sums of larger cells are added in FP64.
struct MomSumsF {
    float M, sx, sy, sz, Q;
};

// G lanes (a whole warp, G = 32, or an aligned group of G = 8 lanes with
// member mask gm; sl = lane within the group) sum a particle range.
template <int G>
__device__ __forceinline__ MomSumsF mom_range_f32(const float4 *__restrict__ phi, const float4 *__restrict__ plo,
                                                  uint32_t f, uint32_t n, uint32_t ref, int sl, unsigned gm)
{
    const float4 hr = phi[ref], lr = plo[ref];
    MomSumsF r = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
    for (uint32_t i = f + sl; i < f + n; i += G) {
        const float4 h = phi[i], l = plo[i];
        const float d0 = (h.x - hr.x) + (l.x - lr.x), d1 = (h.y - hr.y) + (l.y - lr.y), d2 = (h.z - hr.z) + (l.z - lr.z);
        const float mi = h.w;
        r.M += mi;
        r.sx = fmaf(mi, d0, r.sx);
        r.sy = fmaf(mi, d1, r.sy);
        r.sz = fmaf(mi, d2, r.sz);
        r.Q = fmaf(mi, fmaf(d0, d0, fmaf(d1, d1, d2 * d2)), r.Q);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        r.M += __shfl_xor_sync(gm, r.M, o, G);
        r.sx += __shfl_xor_sync(gm, r.sx, o, G);
        r.sy += __shfl_xor_sync(gm, r.sy, o, G);
        r.sz += __shfl_xor_sync(gm, r.sz, o, G);
        r.Q += __shfl_xor_sync(gm, r.Q, o, G);
    }
    return r;
}

// FP32 form: centre of mass as offsets e from the first particle f, stored
// as the grid-aligned hi/lo pair; B2 goes to nB.w. No FP64 instruction here:
// a single-lane FP64 instruction costs a full warp's FP64 pipe time.
__device__ __forceinline__ void mom_store_f32(const MomArgs &a, uint32_t c, uint32_t f, float M, float e0, float e1,
                                              float e2, float B2)
{
    const SysBox &b = a.box[a.S == 1 ? 0 : a.psys[f]];
    const float4 h = a.phi[f], l = a.plo[f];
    const float t0 = l.x + e0, t1 = l.y + e1, t2 = l.z + e2;
    const float g0 = rintf(t0 * b.inv_uf) * b.uf, g1 = rintf(t1 * b.inv_uf) * b.uf, g2 = rintf(t2 * b.inv_uf) * b.uf;
    a.nA[c] = make_float4(h.x + g0, h.y + g1, h.z + g2, M);
    a.nB[c] = make_float4(t0 - g0, t1 - g1, t2 - g2, B2);
}

// B2 of a small cell about its centre of mass e (offsets from particle ref),
// summed directly so that no M|e|^2 cancels against the second moment, and
// b_max, the largest distance of its particles to e (G lanes as above).
template <int G>
__device__ __forceinline__ void mom_b2_f32(const float4 *__restrict__ phi, const float4 *__restrict__ plo, uint32_t f,
                                           uint32_t n, uint32_t ref, float e0, float e1, float e2, int sl, unsigned gm,
                                           float &B2, float &bmax)
{
    const float4 hr = phi[ref], lr = plo[ref];
    float q = 0.0f, d2max = 0.0f;
    for (uint32_t i = f + sl; i < f + n; i += G) {
        const float4 h = phi[i], l = plo[i];
        const float d0 = ((h.x - hr.x) + (l.x - lr.x)) - e0, d1 = ((h.y - hr.y) + (l.y - lr.y)) - e1,
                    d2 = ((h.z - hr.z) + (l.z - lr.z)) - e2;
        const float r2 = fmaf(d0, d0, fmaf(d1, d1, d2 * d2));
        q = fmaf(h.w, r2, q);
        d2max = fmaxf(d2max, r2);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        q += __shfl_xor_sync(gm, q, o, G);
        d2max = fmaxf(d2max, __shfl_xor_sync(gm, d2max, o, G));
    }
    B2 = q;
    bmax = sqrtf(d2max);
}

template <int G>
__device__ __forceinline__ MomSums mom_range(const MomArgs &a, uint32_t f, uint32_t n, double o0, double o1, double o2,
                                             int sl, unsigned gm)
{
    MomSums r = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
    for (uint32_t i = f + sl; i < f + n; i += G) {
        const double mi = a.m[i];
        const double d0 = a.x[i] - o0, d1 = a.y[i] - o1, d2 = a.z[i] - o2;
        r.M += mi;
        r.sx += mi * d0;
        r.sy += mi * d1;
        r.sz += mi * d2;
        r.Q += mi * (d0 * d0 + d1 * d1 + d2 * d2);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {   // fixed butterfly: the same order every run
        r.M += __shfl_xor_sync(gm, r.M, o, G);
        r.sx += __shfl_xor_sync(gm, r.sx, o, G);
        r.sy += __shfl_xor_sync(gm, r.sy, o, G);
        r.sz += __shfl_xor_sync(gm, r.sz, o, G);
        r.Q += __shfl_xor_sync(gm, r.Q, o, G);
    }
    return r;
}

// (s0, s1, s2) / M, one quotient per lane: a division is some 8 dependent FP64 instructions, and they cost the same for
// one lane as for all
template <int G>
__device__ __forceinline__ void div3(double s0, double s1, double s2, double M, int lane, unsigned gm, double &q0,
                                     double &q1, double &q2)
{
    const double q = (lane == 1 ? s1 : (lane == 2 ? s2 : s0)) / M;
    q0 = __shfl_sync(gm, q, 0, G);
    q1 = __shfl_sync(gm, q, 1, G);
    q2 = __shfl_sync(gm, q, 2, G);
}

// by all G lanes, which have the same sums; the centre to (c0, c1, c2)
template <int G>
__device__ __forceinline__ void mom_store(const MomArgs &a, uint32_t c, const MomSums &r, double o0, double o1,
                                          double o2, int sl, unsigned gm, double &c0, double &c1, double &c2)
{
    double B2 = 0.0;
    if (r.M > 0.0) {
        double e0, e1, e2;
        div3<G>(r.sx, r.sy, r.sz, r.M, sl, gm, e0, e1, e2);
        c0 = o0 + e0;
        c1 = o1 + e1;
        c2 = o2 + e2;
        B2 = fmax(r.Q - r.M * (e0 * e0 + e1 * e1 + e2 * e2), 0.0);
    } else {   // massless cell: its geometric centre
        double o[3], sd;
        const uint32_t f = a.nfirst[c];
        cell_geom(a.box[a.psys[f]], a.key[f], a.nlevel[c], o, &sd);
        c0 = o[0] + 0.5 * sd;
        c1 = o[1] + 0.5 * sd;
        c2 = o[2] + 0.5 * sd;
    }
    if (sl == 0) store_com(a, c, r.M, c0, c1, c2, B2);
}

// sum over the first 8 of G lanes (the children of a cell), in all of them
template <int G>
__device__ __forceinline__ double sum8_d(double v, unsigned gm)
{
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(gm, v, o, G);
    return G > 8 ? __shfl_sync(gm, v, 0, G) : v;
}

// A larger cell from its (at most 8) children, one per lane, in a fixed order.
// FP64 form in FP64. FP32 form in FP32 on offsets from the first child's hi/lo
// centre of mass (hi differences exact), stored like a small cell's. By G lanes
// (a warp or an aligned group of 8 with mask gm).
// f: the cell's first particle; [ch0, ch0 + k): its children.
template <int G>
__device__ void mom_combine_f64(const MomArgs &a, uint32_t c, uint32_t f, uint32_t ch0, uint32_t k, int lane,
                                unsigned gm)
{
    const SysBox &b = a.box[a.S == 1 ? 0 : a.psys[f]];
    const bool on = (uint32_t)lane < k;
    double M = 0.0, x = 0.0, y = 0.0, z = 0.0, B2 = 0.0;
    if (on) {
        const uint32_t j = ch0 + lane;
        M = __ldcg(a.M + j);
        x = __ldcg(a.cx + j);
        y = __ldcg(a.cy + j);
        z = __ldcg(a.cz + j);
        B2 = __ldcg(a.B2 + j);
    }
    const double rx = __shfl_sync(gm, x, 0, G), ry = __shfl_sync(gm, y, 0, G), rz = __shfl_sync(gm, z, 0, G);
    const double dx = x - rx, dy = y - ry, dz = z - rz;
    const double Mt = sum8_d<G>(M, gm);   // the same in all lanes: the branch below has sums over them
    double c0, c1, c2, B2t = 0.0;
    if (Mt > 0.0) {
        double ex, ey, ez;
        div3<G>(sum8_d<G>(M * dx, gm), sum8_d<G>(M * dy, gm), sum8_d<G>(M * dz, gm), Mt, lane, gm, ex, ey, ez);
        c0 = rx + ex;
        c1 = ry + ey;
        c2 = rz + ez;
        const double qx = dx - ex, qy = dy - ey, qz = dz - ez;
        B2t = sum8_d<G>(on ? B2 + M * (qx * qx + qy * qy + qz * qz) : 0.0, gm);
    } else {   // massless cell: its geometric centre
        double o[3], sd;
        cell_geom(b, a.key[f], a.nlevel[c], o, &sd);
        c0 = o[0] + 0.5 * sd;
        c1 = o[1] + 0.5 * sd;
        c2 = o[2] + 0.5 * sd;
    }
    if (lane == 0) store_com(a, c, Mt, c0, c1, c2, B2t);
}

template <int G>
__device__ void mom_combine_f32(const MomArgs &a, uint32_t c, uint32_t f, uint32_t ch0, uint32_t k, int lane,
                                unsigned gm)
{
    const SysBox &b = a.box[a.S == 1 ? 0 : a.psys[f]];
    const bool on = (uint32_t)lane < k;
    float4 A = make_float4(0.0f, 0.0f, 0.0f, 0.0f), B = A;
    float rad = 0.0f;   // the child's particles lie within this of its centre of mass
    if (on) {
        A = __ldcg(a.nA + ch0 + lane);
        B = __ldcg(a.nB + ch0 + lane);
        if (a.search) rad = __uint_as_float(__ldcg(a.bmax32 + ch0 + lane));
    }
    const float hx = __shfl_sync(gm, A.x, 0, G), hy = __shfl_sync(gm, A.y, 0, G),
                hz = __shfl_sync(gm, A.z, 0, G);
    const float lx = __shfl_sync(gm, B.x, 0, G), ly = __shfl_sync(gm, B.y, 0, G),
                lz = __shfl_sync(gm, B.z, 0, G);
    const float M = A.w, dx = (A.x - hx) + (B.x - lx), dy = (A.y - hy) + (B.y - ly), dz = (A.z - hz) + (B.z - lz);
    float Mt = M, sx = M * dx, sy = M * dy, sz = M * dz;
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        Mt += __shfl_xor_sync(gm, Mt, o, G);
        sx += __shfl_xor_sync(gm, sx, o, G);
        sy += __shfl_xor_sync(gm, sy, o, G);
        sz += __shfl_xor_sync(gm, sz, o, G);
    }
    float e0, e1, e2, B2t = 0.0f;
    if (Mt > 0.0f) {
        e0 = sx / Mt;
        e1 = sy / Mt;
        e2 = sz / Mt;
        const float qx = dx - e0, qy = dy - e1, qz = dz - e2;
        B2t = on ? fmaf(M, qx * qx + qy * qy + qz * qz, B.w) : 0.0f;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) B2t += __shfl_xor_sync(gm, B2t, o, G);
    } else {   // massless cell: its geometric centre, relative to the first child's centre
        double o[3], sd;
        cell_geom(b, a.key[f], a.nlevel[c], o, &sd);
        e0 = (float)((o[0] + 0.5 * sd - b.lo[0]) - ((double)hx + (double)lx));
        e1 = (float)((o[1] + 0.5 * sd - b.lo[1]) - ((double)hy + (double)ly));
        e2 = (float)((o[2] + 0.5 * sd - b.lo[2]) - ((double)hz + (double)lz));
    }
    if (a.search) {   // and this cell's particles within this of its own: a bound, which k_finish replaces by b_max
        const float qx = dx - e0, qy = dy - e1, qz = dz - e2;
        rad = on ? (sqrtf(qx * qx + qy * qy + qz * qz) + rad) * 1.00001f : 0.0f;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) rad = fmaxf(rad, __shfl_xor_sync(gm, rad, o, G));
        if (lane == 0) a.bmax32[c] = __float_as_uint(rad);
    }
    if (lane == 0) {
        const float t0 = lx + e0, t1 = ly + e1, t2 = lz + e2;
        const float g0 = rintf(t0 * b.inv_uf) * b.uf, g1 = rintf(t1 * b.inv_uf) * b.uf,
                    g2 = rintf(t2 * b.inv_uf) * b.uf;
        a.nA[c] = make_float4(hx + g0, hy + g1, hz + g2, Mt);
        a.nB[c] = make_float4(t0 - g0, t1 - g1, t2 - g2, B2t);
    }
}

// After cell c (with parent p) is final: if its parent is a larger cell and c is
// the last of its children to finish, combine the parent, and so on upwards. G
// lanes (a warp, or an aligned group of 8 with mask gm; lane = lane within the
// group). This chain of levels is what k_mom_small's time on a small system is
// made of, so a level costs three waits: the parent's record (all fields at
// once), the count, the children's moments.
template <bool F64, int G>
__device__ void mom_climb(const MomArgs &a, uint32_t p, int lane, unsigned gm)
{
    while (p != NONE) {
        const uint32_t f = a.nfirst[p], e = a.nend[p], ch0 = a.nchild[p], k = a.nchend[p] - ch0, up = a.nparent[p];
        if (e - f <= MOM_CH) return;
        __syncwarp(gm);
        unsigned int old = 0;
        if (lane == 0) {   // release: the child's moments (stored by this lane) before the count; acquire: the others' after
            cuda::atomic_ref<unsigned int, cuda::thread_scope_device> cnt(a.done[p]);
            old = cnt.fetch_add(1u, cuda::memory_order_acq_rel);
        }
        old = __shfl_sync(gm, old, 0, G);
        if (old + 1u != k) return;
        __syncwarp(gm);
        if (F64) mom_combine_f64<G>(a, p, f, ch0, k, lane, gm);
        else mom_combine_f32<G>(a, p, f, ch0, k, lane, gm);
        p = up;
    }
}

// Per node: geometry, delta, MAC radius, walk criteria and packed topology.
struct FinArgs {
    const uint32_t *lvl, *nfirst, *nend, *nchend, *nchild, *nlevel;
    const uint64_t *key;
    const int32_t *psys;
    int S;
    const SysBox *box;
    const SysParams *sp;
    double *M, *cx, *cy, *cz, *B2;
    unsigned long long *bmax;
    unsigned int *bmax32;
    const float4 *nA, *nB;
    float2 *crit;
    uint4 *topo;
    double4_32a *nD;
    double *rb, *hr, *delta, *side, *org;
};

// every third bit of a key, from bit 0 (the inverse of spread3)
__device__ __forceinline__ uint32_t compact3(uint64_t x)
{
    x &= 0x1249249249249249ull;
    x = (x | (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x | (x >> 4)) & 0x100f00f00f00f00full;
    x = (x | (x >> 8)) & 0x1f0000ff0000ffull;
    x = (x | (x >> 16)) & 0x1f00000000ffffull;
    x = (x | (x >> 32)) & 0x1fffffull;
    return (uint32_t)x;
}

// integer cell coordinates of a key's level-lev cell
__device__ __forceinline__ void prefix_q(uint64_t key, uint32_t lev, uint32_t q[3])
{
    q[0] = compact3(key >> 2) >> (LEVELS - lev);
    q[1] = compact3(key >> 1) >> (LEVELS - lev);
    q[2] = compact3(key) >> (LEVELS - lev);
}

struct CritF {
    float rb, hr, delta;
};

// FP32 form: delta, r_b and the Eq. (15) radius from the hi/lo centre of mass (cell centres are exact in FP32 on the
// hi grid)
__device__ __forceinline__ CritF crit_f32(const float4 &A, const float4 &B, float bm, uint32_t lev, const uint32_t q[3],
                                          const SysParams &P, const SysBox &bx)
{
    // no FP64 instruction here (conversions count): the FP64 pipe has 2 lanes per SM
    const float sdf = bx.uf * __int_as_float((127 + 20 - (int)lev) << 23);   // L 2^-lev: exact
    // cell centre relative to the root corner: (q + 1/2) side, exact in FP32
    const float e0 = (A.x - ((float)q[0] + 0.5f) * sdf) + B.x;
    const float e1 = (A.y - ((float)q[1] + 0.5f) * sdf) + B.y;
    const float e2 = (A.z - ((float)q[2] + 0.5f) * sdf) + B.z;
    CritF r;
    r.delta = sqrtf(e0 * e0 + e1 * e1 + e2 * e2);
    if (P.mac == 1) r.rb = 0.5f * bm + sqrtf(0.25f * bm * bm + sqrtf(3.0f * B.w / P.a_errf));
    else r.rb = (P.thetaf > 0.0f) ? sdf / P.thetaf + r.delta : INFINITY;
    r.hr = P.R2f + P.skinf + bm;
    return r;
}

// FP32 form: what the walk reads of cell c (particles [f, e), centre of mass A, B, b_max bm)
__device__ __forceinline__ void finish_f32(const FinArgs &a, uint32_t c, uint32_t f, uint32_t e, const float4 &A,
                                           const float4 &B, float bm)
{
    const int s = a.S == 1 ? 0 : a.psys[f];
    const SysParams &P = a.sp[s];
    const uint32_t lev = a.nlevel[c], ch = a.nchild[c];
    uint32_t q[3];
    prefix_q(a.key[f], lev, q);
    const CritF r = crit_f32(A, B, bm, lev, q, P, a.box[s]);
    const float sacc = fmaxf(r.rb, r.hr);
    a.crit[c] = make_float2(sacc * sacc, P.has_hard ? r.hr * r.hr : -1.0f);
    a.topo[c] = make_uint4(ch, ch == NONE ? 0u : a.nchend[c] - ch, f, e - f);
    a.bmax32[c] = __float_as_uint(bm);
}

constexpr uint32_t BM_CH = 256;

// largest distance of particles [f, e) to (c0, c1, c2): the largest square, compared as an integer (squares are not
// negative; a NaN would win), and one square root at the end (it is monotone)
template <int G>
__device__ __forceinline__ double farthest_f64(const MomArgs &a, uint32_t f, uint32_t e, double c0, double c1, double c2,
                                               int sl, unsigned gm)
{
    long long m = 0;
    for (uint32_t i = f + sl; i < e; i += G) {
        const double d0 = a.x[i] - c0, d1 = a.y[i] - c1, d2 = a.z[i] - c2;
        m = max(m, __double_as_longlong(d0 * d0 + d1 * d1 + d2 * d2));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(gm, m, o, G));
    return sqrt(__longlong_as_double(m));
}

// FP64 form: moments of a cell from its particles, the climb, and b_max, by G lanes
template <int G>
__device__ __forceinline__ void mom_cell_f64(const MomArgs &a, uint32_t c, uint32_t f, uint32_t n, uint32_t up, int sl,
                                             unsigned gm)
{
    const double o0 = a.x[f], o1 = a.y[f], o2 = a.z[f];
    const MomSums r = mom_range<G>(a, f, n, o0, o1, o2, sl, gm);
    double c0, c1, c2;
    mom_store<G>(a, c, r, o0, o1, o2, sl, gm, c0, c1, c2);
    mom_climb<true, G>(a, up, sl, gm);   // others wait for this
    const double dm = farthest_f64<G>(a, f, f + n, c0, c1, c2, sl, gm);
    if (sl == 0) a.bmax64[c] = (unsigned long long)__double_as_longlong(dm);
}

// every cell of at most MOM_CH particles, and every leaf (a leaf holds more
// only when its particles share one level-21 cell): moments and b_max from its
// particles, then the climb; the larger cells are listed for their b_max, in
// chunks of BM_CH particles (once each where b_max is searched for)
template <bool F64>
__global__ void __launch_bounds__(256) k_mom_small(MomArgs a, unsigned long long *nitems, uint32_t *bigbase,
                                                   uint32_t *items, uint32_t cap_items, Status *st, int where)
{
    if (st->code) return;
    const uint32_t total = a.lvl[LEVELS + 1];
    const int lane = threadIdx.x & 31;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int sub = lane >> 3, sl = lane & 7;
    const unsigned gm = 0xFFu << (8 * sub);
    const uint32_t nq = (total + 3) / 4;
    auto list_big = [&](uint32_t c, uint32_t n) {   // by the cell's 8 lanes
        const uint32_t nch = a.search ? 1u : (n + BM_CH - 1) / BM_CH;
        unsigned long long base = 0;
        if (sl == 0) base = atomicAdd(nitems, (unsigned long long)nch);
        base = __shfl_sync(gm, base, 0, 8);
        if (base + nch > cap_items) {
            if (sl == 0) fail(st, HYBRID_ECAPACITY, where);
            return;
        }
        if (sl == 0) bigbase[c] = (uint32_t)base;
        for (uint32_t k = sl; k < nch; k += 8) items[base + k] = c;
    };
    if (F64) {
        // Four cells per warp: an FP64 instruction takes the pipe 16 clocks for a warp, however few of its lanes are
        // on, and most cells hold fewer than 16 particles (moments of a build at N = 30011: one warp per cell
        // 0.132 ms, so 0.098).
        // Leaves of more than MOM_CH particles come after that, by the whole warp.
        for (uint32_t q = warp; q < nq; q += nw) {
            const uint32_t c = 4 * q + sub;
            const bool valid = c < total;
            const uint32_t f = valid ? a.nfirst[c] : 0u, n = valid ? a.nend[c] - f : 0u, up = valid ? a.nparent[c] : NONE;
            const bool leaf = valid && a.nchild[c] == NONE;
            if (valid && n <= MOM_CH) {
                mom_cell_f64<8>(a, c, f, n, up, sl, gm);
            } else if (valid && !leaf) {
                list_big(c, n);
            }
            __syncwarp();
            for (unsigned todo = __ballot_sync(0xffffffffu, leaf && n > MOM_CH && sl == 0); todo; todo &= todo - 1) {
                const int from = __ffs(todo) - 1;
                mom_cell_f64<32>(a, __shfl_sync(0xffffffffu, c, from), __shfl_sync(0xffffffffu, f, from),
                                 __shfl_sync(0xffffffffu, n, from), __shfl_sync(0xffffffffu, up, from), lane, 0xffffffffu);
            }
        }
    } else {   // FP32 form: four cells per warp, eight lanes each (most cells are leaves of a few particles)
        for (uint32_t q = warp; q < nq; q += nw) {
            const uint32_t c = 4 * q + sub;
            if (c >= total) continue;
            const uint32_t f = a.nfirst[c], n = a.nend[c] - f, up = a.nparent[c];
            if (n <= MOM_CH || a.nchild[c] == NONE) {
                const MomSumsF r = mom_range_f32<8>(a.phi, a.plo, f, n, f, sl, gm);
                const float iM = r.M > 0.0f ? 1.0f / r.M : 0.0f;
                const float e0 = r.sx * iM, e1 = r.sy * iM, e2 = r.sz * iM;
                float B2, bm;
                mom_b2_f32<8>(a.phi, a.plo, f, n, f, e0, e1, e2, sl, gm, B2, bm);
                if (sl == 0) {
                    mom_store_f32(a, c, f, r.M, e0, e1, e2, B2);
                    a.bmax32[c] = __float_as_uint(bm);
                }
                mom_climb<false, 8>(a, up, sl, gm);
            } else {
                list_big(c, n);
            }
        }
    }
}

// b_max of the larger cells, one warp per chunk of BM_CH particles, one atomic
// max per chunk (non-negative floats order as their bit patterns)
template <bool F64>
__global__ void __launch_bounds__(256) k_bmax_big(MomArgs a, const unsigned long long *nitems,
                                                  const uint32_t *bigbase, const uint32_t *items, const Status *st)
{
    if (st->code) return;
    const uint32_t T = (uint32_t)*nitems;
    const int lane = threadIdx.x & 31;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < T; w += nw) {
        const uint32_t c = items[w];
        const uint32_t k = w - bigbase[c];
        const uint32_t f = a.nfirst[c], n = a.nend[c] - f;
        const uint32_t f0 = f + k * BM_CH, n0 = min(BM_CH, f + n - f0);
        if (F64) {
            const double c0 = a.cx[c], c1 = a.cy[c], c2 = a.cz[c];
            const double dm = farthest_f64<32>(a, f0, f0 + n0, c0, c1, c2, lane, 0xffffffffu);
            if (lane == 0) atomicMax(a.bmax64 + c, (unsigned long long)__double_as_longlong(dm));
        } else {
            const float4 A = a.nA[c], B = a.nB[c];
            float dm = 0.0f;
#pragma unroll 4
            for (uint32_t i = f0 + lane; i < f0 + n0; i += 32) {
                const float4 h = a.phi[i], l = a.plo[i];
                const float d0 = (h.x - A.x) + (l.x - B.x);
                const float d1 = (h.y - A.y) + (l.y - B.y);
                const float d2 = (h.z - A.z) + (l.z - B.z);
                dm = fmaxf(dm, d0 * d0 + d1 * d1 + d2 * d2);
            }
            dm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dm)));
            if (lane == 0) atomicMax(a.bmax32 + c, __float_as_uint(sqrtf(dm)));
        }
    }
}

// FP32 form: what the walk reads of every cell; with SEARCH, before that, b_max
// of the larger ones: the distance of the particle farthest from the centre of
// mass, one warp per cell; up to BIG_ALL particles by taking all of them, above
// by a search of the cell's subtree. A node's particles lie within r of its
// centre of mass, at d from the cell's (r = b_max up to MOM_CH particles, above
// the bound that its combine made of its children's, or by now its own b_max).
// It can hold the farthest particle only if d + r reaches the best distance so
// far; and it holds one at d - r at least (and at r - d, where r is b_max).
// Leaves left over are measured particle by particle, so the value is that of
// taking every particle (the bounds carry 1e-5 of slack for their rounding).
// Taking every particle (k_bmax_big) reads the state once per level of larger
// cells, a search about 50 nodes and 5 leaves, in a few steps that wait for one
// another: searching is for batches above 2^20 particles (moments per soft
// step: 2^24 13.6 -> 12.0 ms, 512 systems of 12.9 M particles 5.9 -> 4.7; below
// it loses: 2^17 0.177 -> 0.186, 2^20 0.465 -> 0.49). The other cells are
// finished meanwhile, one per thread: on one lane in eight, with their moments,
// the same work took longer.
constexpr int BIG_THREADS = 128, BIG_STACK = 1024, BIG_QUEUE = 512;
constexpr uint32_t BIG_ALL = 512;
constexpr int BIG_SLACK = 160;   // stack entries kept for a descent one node at a time: 7 more per level, 21 levels

template <bool SEARCH>
__global__ void __launch_bounds__(BIG_THREADS) k_finish(MomArgs a, FinArgs fa, const unsigned long long *nitems,
                                                        const uint32_t *items, const Status *st)
{
    __shared__ uint32_t stacks[SEARCH ? BIG_THREADS / 32 : 1][SEARCH ? BIG_STACK : 1];
    __shared__ uint32_t queues[SEARCH ? BIG_THREADS / 32 : 1][SEARCH ? BIG_QUEUE : 1];   // particles to measure
    if (st->code) return;
    const uint32_t T = SEARCH ? (uint32_t)*nitems : 0u;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t *stk = stacks[SEARCH ? threadIdx.x >> 5 : 0], *que = queues[SEARCH ? threadIdx.x >> 5 : 0];
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; SEARCH && w < T; w += nw) {
        const uint32_t c = items[w];
        const uint32_t f = a.nfirst[c], e = a.nend[c], ch0 = a.nchild[c];
        int sp = (int)(a.nchend[c] - ch0);
        const float4 A = a.nA[c], B = a.nB[c];
        float far = 0.0f, best2 = 0.0f;   // some particle is at least this far; this lane's farthest one, squared
        auto measure = [&](uint32_t i) {
            const float4 h = a.phi[i], l = a.plo[i];
            const float d0 = (h.x - A.x) + (l.x - B.x);
            const float d1 = (h.y - A.y) + (l.y - B.y);
            const float d2 = (h.z - A.z) + (l.z - B.z);
            best2 = fmaxf(best2, d0 * d0 + d1 * d1 + d2 * d2);
        };
        if (e - f <= BIG_ALL) {
#pragma unroll 4
            for (uint32_t i = f + lane; i < e; i += 32) measure(i);
            sp = 0;
        }
        if (lane < sp) stk[lane] = ch0 + lane;
        __syncwarp();
        while (sp > 0) {
            const int take = min(sp, max(1, min(32, (BIG_STACK - BIG_SLACK - sp) / 7)));
            const bool on = lane < take;
            uint32_t first = 0, count = 0, ch = NONE, k = 0;
            float least = 0.0f, reach = -1.0f;
            if (on) {
                const uint32_t q = stk[sp - take + lane];
                first = a.nfirst[q];
                count = a.nend[q] - first;
                ch = a.nchild[q];
                k = ch == NONE ? 0u : a.nchend[q] - ch;
                const float4 qa = a.nA[q], qb = a.nB[q];
                const float r = __uint_as_float(a.bmax32[q]);
                const float dx = (qa.x - A.x) + (qb.x - B.x), dy = (qa.y - A.y) + (qb.y - B.y), dz = (qa.z - A.z) + (qb.z - B.z);
                const float d = sqrtf(dx * dx + dy * dy + dz * dz);
                least = fmaxf(d - r, count <= MOM_CH || ch == NONE ? r - d : 0.0f);
                reach = (d + r) * 1.00001f;
            }
            sp -= take;
            // distances are >= 0: they order as integers
            far = fmaxf(far, 0.99999f * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(least))));
            const bool alive = on && reach >= far;
            const uint32_t np = alive && k == 0u ? count : 0u;
            if (__any_sync(0xffffffffu, np > 0u)) {
                if (__all_sync(0xffffffffu, np <= (uint32_t)(BIG_QUEUE / 32))) {   // all leaves' particles together
                    uint32_t ex = 0, tot = 0;
#pragma unroll
                    for (int b = 0; b < 5; ++b) {
                        const unsigned m = __ballot_sync(0xffffffffu, (np >> b) & 1u);
                        ex += (uint32_t)__popc(m & lt) << b;
                        tot += (uint32_t)__popc(m) << b;
                    }
                    for (uint32_t j = 0; j < np; ++j) que[ex + j] = first + j;
                    __syncwarp();
                    for (uint32_t i = lane; i < tot; i += 32) measure(que[i]);
                    __syncwarp();
                } else {
                    unsigned leaves = __ballot_sync(0xffffffffu, np > 0u);
                    do {
                        const int src = __ffs(leaves) - 1;
                        leaves &= leaves - 1u;
                        const uint32_t p0 = __shfl_sync(0xffffffffu, first, src), p1 = p0 + __shfl_sync(0xffffffffu, np, src);
                        for (uint32_t i = p0 + lane; i < p1; i += 32) measure(i);
                    } while (leaves);
                }
                far = fmaxf(far, 0.99999f * sqrtf(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best2)))));
            }
            const uint32_t push = alive && reach >= far ? k : 0u;
            uint32_t ex = 0, tot = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const unsigned m = __ballot_sync(0xffffffffu, (push >> b) & 1u);
                ex += (uint32_t)__popc(m & lt) << b;
                tot += (uint32_t)__popc(m) << b;
            }
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j)
                if (j < push) stk[sp + ex + j] = ch + j;
            sp += (int)tot;
            __syncwarp();
        }
        best2 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best2)));
        if (lane == 0) finish_f32(fa, c, f, e, A, B, sqrtf(best2));
    }
    const uint32_t total = a.lvl[LEVELS + 1];
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
        const uint32_t f = a.nfirst[c], e = a.nend[c];
        if (!SEARCH || e - f <= MOM_CH || a.nchild[c] == NONE) finish_f32(fa, c, f, e, a.nA[c], a.nB[c], __uint_as_float(a.bmax32[c]));
    }
}

// FP64 form: criteria from the FP64 moments, and what hybrid_tree_copy reports. (The FP32 form finishes a cell with its
// moments, and k_inspect makes the reports when they are asked for: 170 bytes and a dozen FP64 operations a node that
// no force needs.)
__global__ void __launch_bounds__(256) k_finalize(FinArgs a, const Status *st)
{
    if (st->code) return;
    const uint32_t total = a.lvl[LEVELS + 1];
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
        const uint32_t f = a.nfirst[c];
        const int s = a.S == 1 ? 0 : a.psys[f];
        const SysParams &P = a.sp[s];
        const SysBox &bx = a.box[s];
        const uint32_t lev = a.nlevel[c];
        uint32_t q[3];
        prefix_q(a.key[f], lev, q);
        const double sd = ldexp(bx.L, -(int)lev);
        double o[3], rb;
        for (int k = 0; k < 3; ++k) o[k] = __dadd_rn(bx.lo[k], __dmul_rn((double)q[k], sd));
        const double ctr0 = o[0] + 0.5 * sd, ctr1 = o[1] + 0.5 * sd, ctr2 = o[2] + 0.5 * sd;
        const double e0 = a.cx[c] - ctr0, e1 = a.cy[c] - ctr1, e2 = a.cz[c] - ctr2;
        const double delta = sqrt(e0 * e0 + e1 * e1 + e2 * e2);
        const double bm = __longlong_as_double((long long)a.bmax[c]);
        if (P.mac == 1) rb = 0.5 * bm + sqrt(0.25 * bm * bm + sqrt(3.0 * a.B2[c] / P.a_err));
        else rb = (P.theta > 0.0) ? sd / P.theta + delta : INFINITY;
        const double hr = P.R2 + P.skin + bm;   // Eq. (15) radius (plus the skin of reused lists)
        const double sacc = fmax(rb, hr);
        a.crit[c] = make_float2((float)(sacc * sacc), P.has_hard ? (float)(hr * hr) : -1.0f);
        a.nD[c] = make_double4_32a(a.cx[c], a.cy[c], a.cz[c], a.M[c]);
        for (int k = 0; k < 3; ++k) a.org[3 * (size_t)c + k] = o[k];
        a.rb[c] = rb;
        a.hr[c] = hr;
        a.delta[c] = delta;
        a.side[c] = sd;
        const uint32_t ch = a.nchild[c];
        a.topo[c] = make_uint4(ch, ch == NONE ? 0u : a.nchend[c] - ch, f, a.nend[c] - f);
    }
}

// FP32 form: the FP64 copies of the moments and the geometry that hybrid_tree_copy reports.
__global__ void __launch_bounds__(256) k_inspect(FinArgs a)
{
    const uint32_t total = a.lvl[LEVELS + 1];
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
        const uint32_t f = a.nfirst[c];
        const int s = a.psys[f];
        const SysBox &bx = a.box[s];
        const uint32_t lev = a.nlevel[c];
        uint32_t q[3];
        prefix_q(a.key[f], lev, q);
        const float4 A = a.nA[c], B = a.nB[c];
        const float bm = __uint_as_float(a.bmax32[c]);
        const CritF r = crit_f32(A, B, bm, lev, q, a.sp[s], bx);
        a.M[c] = (double)A.w;
        a.cx[c] = bx.lo[0] + ((double)A.x + (double)B.x);
        a.cy[c] = bx.lo[1] + ((double)A.y + (double)B.y);
        a.cz[c] = bx.lo[2] + ((double)A.z + (double)B.z);
        a.B2[c] = (double)B.w;
        a.bmax[c] = (unsigned long long)__double_as_longlong((double)bm);
        const double sd = ldexp(bx.L, -(int)lev);
        for (int k = 0; k < 3; ++k) a.org[3 * (size_t)c + k] = __dadd_rn(bx.lo[k], __dmul_rn((double)q[k], sd));
        a.rb[c] = r.rb;
        a.delta[c] = r.delta;
        a.side[c] = sd;
    }
}

// ---------------------------------------------------------------------------
// Sink groups: first cells (from the root) with count <= n_crit, or leaves.
// Marked at their first particle, compacted in particle order. Only for n_crit
// above GROUP_WINDOW (k_nodes makes the others).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_group_flag(const uint32_t *__restrict__ lvl,
                                                    const uint32_t *__restrict__ nfirst,
                                                    const uint32_t *__restrict__ nend,
                                                    const uint32_t *__restrict__ nchild,
                                                    const uint32_t *__restrict__ nparent, int n_crit,
                                                    uint32_t *__restrict__ gflag, const Status *st)
{
    if (st->code) return;
    const uint32_t total = lvl[LEVELS + 1];
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
        const bool stop = nend[c] - nfirst[c] <= (uint32_t)n_crit || nchild[c] == NONE;
        const uint32_t p = nparent[c];
        const bool parent_goes_on = (p == NONE) || (nend[p] - nfirst[p] > (uint32_t)n_crit);
        if (stop && parent_goes_on) gflag[nfirst[c]] = c;
    }
}

__global__ void __launch_bounds__(256) k_group_mark(int64_t N, const uint32_t *__restrict__ gflag,
                                                    uint32_t *__restrict__ gscan, const Status *st)
{
    if (st->code) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        gscan[i] = gflag[i] != NONE ? 1u : 0u;
}

__global__ void __launch_bounds__(256) k_group_compact(int64_t N, const uint32_t *__restrict__ gflag,
                                                       const uint32_t *__restrict__ gscan,
                                                       const int32_t *__restrict__ psys, uint32_t *gnode,
                                                       uint32_t *gfirst, uint32_t *gsys, const uint64_t *total, int64_t *ngroups, const Status *st)
{
    if (st->code) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *ngroups = (int64_t)*total;
        gfirst[*total] = (uint32_t)N;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = gflag[i];
        if (c != NONE) {
            const uint32_t g = gscan[i];
            gnode[g] = c;
            gfirst[g] = (uint32_t)i;
            gsys[g] = (uint32_t)psys[i];
        }
    }
}

// Box of each group's members (FP64, exact min/max), its centre as an FP32
// hi/lo pair and its half extents rounded up. Eight lanes per group (three
// exchange steps instead of five, and four groups at once), R groups after one
// another; then the FP64 finishing of the warp's 4 R groups at once, one lane
// each (a one-lane FP64 instruction costs the FP64 pipe a whole warp's time).
// Groups of more than GB_WARP particles (one level-21 cell's, or a large n_crit)
// take the whole warp. One warp per group and 145 registers before: N = 100000
// 18.5 -> 12.2 us, a soft step of 2^20 (absolute MAC) 0.289 -> 0.231 ms, of 2^24
// 6.57 -> 5.69 ms.
constexpr uint32_t GB_WARP = 1024;

// min and max of the three coordinates of particles [f, f + n), through their order-preserving integer images (no FP64
// pipe work), in all G lanes
template <int G>
__device__ __forceinline__ void group_min_max(const double *__restrict__ x, const double *__restrict__ y,
                                              const double *__restrict__ z, uint32_t f, uint32_t n, int sl, unsigned gm,
                                              unsigned long long u[6])
{
    for (int j = 0; j < 6; ++j) u[j] = j < 3 ? ~0ull : 0ull;
#pragma unroll 2
    for (uint32_t i = f + sl; i < f + n; i += G) {
        const unsigned long long p[3] = {ord_dbl(x[i]), ord_dbl(y[i]), ord_dbl(z[i])};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            u[j] = min(u[j], p[j]);
            u[j + 3] = max(u[j + 3], p[j]);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const unsigned long long v = __shfl_xor_sync(gm, u[j], o, G);
            u[j] = j < 3 ? min(u[j], v) : max(u[j], v);
        }
}

__global__ void __launch_bounds__(256, 4) k_group_box(const int64_t *__restrict__ ngroups,
                                                   const uint32_t *__restrict__ gfirst, const double *__restrict__ x,
                                                   const double *__restrict__ y, const double *__restrict__ z,
                                                   const int32_t *__restrict__ psys, const SysBox *__restrict__ box,
                                                   double *glo, double *ghi, GroupF *gF, const Status *st)
{
    if (st->code) return;
    const int lane = threadIdx.x & 31;
    const int64_t ng = *ngroups;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int sub = lane >> 3, sl = lane & 7;
    const unsigned gm = 0xFFu << (8 * sub);
    const int R = (int)max((int64_t)1, min((int64_t)8, ng / (nw * 8)));
    for (int64_t g0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (4 * R); g0 < ng; g0 += nw * (4 * R)) {
        // lane sl < R of a sub-warp has its sl-th group
        const int64_t g = g0 + sub * R + sl;
        const bool own = sl < R && g < ng;
        const uint32_t first = own ? gfirst[g] : 0u, size = own ? gfirst[g + 1] - first : 0u;
        unsigned long long mine[6];
        for (int k = 0; k < R; ++k) {
            const uint32_t f = __shfl_sync(0xffffffffu, first, k, 8), n = __shfl_sync(0xffffffffu, size, k, 8);
            unsigned long long u[6];
            group_min_max<8>(x, y, z, f, n <= GB_WARP ? n : 0u, sl, gm, u);
            if (sl == k)
                for (int j = 0; j < 6; ++j) mine[j] = u[j];
            __syncwarp();
            for (unsigned big = __ballot_sync(0xffffffffu, sl == k && n > GB_WARP); big; big &= big - 1) {
                const int at = __ffs(big) - 1;
                group_min_max<32>(x, y, z, __shfl_sync(0xffffffffu, f, at), __shfl_sync(0xffffffffu, n, at), lane,
                                  0xffffffffu, u);
                if (lane == at)
                    for (int j = 0; j < 6; ++j) mine[j] = u[j];
            }
        }
        if (own) {
            double v[6];
            for (int j = 0; j < 6; ++j) v[j] = unord_dbl(mine[j]);
            const SysBox &b = box[psys[first]];
            float hc[3], lc[3], he[3];
            for (int d = 0; d < 3; ++d) {
                glo[3 * g + d] = v[d];
                ghi[3 * g + d] = v[d + 3];
                const double cc = 0.5 * (v[d] + v[d + 3]) - b.lo[d];   // relative to the root corner
                hc[d] = (float)cc;
                lc[d] = (float)(cc - (double)hc[d]);
                he[d] = __double2float_ru(0.5 * (v[d + 3] - v[d]));
            }
            GroupF G;
            G.c_hi = make_float4(hc[0], hc[1], hc[2], he[0]);
            G.c_lo = make_float4(lc[0], lc[1], lc[2], he[1]);
            G.hz_root = make_float2(he[2], 0.0f);
            gF[g] = G;
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static int grid_for(hybrid_ctx *c, int64_t work, int threads, int per_sm = 8)
{
    int64_t g = (work + threads - 1) / threads;
    g = std::max<int64_t>(1, std::min<int64_t>(g, (int64_t)c->nsm * per_sm));
    return (int)g;
}

void launch_box(hybrid_ctx *c)
{
    if (c->box_done) {   // by the drift before this build
        c->box_done = false;
        return;
    }
    // the boxes are empty here: the copy into the working state and every permutation reset them
    k_box<<<std::min(c->nchunks, c->nsm * 16), 256, 0, c->st>>>(
        (const double *)c->x[0].p, (const double *)c->x[1].p, (const double *)c->x[2].p, (const Chunk *)c->chunks_dev.p,
        c->nchunks, box_args(c));
    c->launches += 1;
}

void launch_keys_sort(hybrid_ctx *c)
{
    Status *st = status_dev(c);
    const int64_t N = c->N;
    uint64_t *k0 = (uint64_t *)c->keys[0].p, *k1 = (uint64_t *)c->keys[1].p;
    uint32_t *v0 = (uint32_t *)c->vals[0].p, *v1 = (uint32_t *)c->vals[1].p;
    if (!c->sort_fallback) {
        uint32_t *cnt = (uint32_t *)c->ss_cnt.p, *flag = (uint32_t *)c->ss_flag.p;
        uint64_t *rk = (uint64_t *)c->ss_rk.p;
        uint32_t *rv = (uint32_t *)c->ss_rv.p;
        const SSys *ss = (const SSys *)c->ss_sys.p;
        const uint32_t *bsys = (const uint32_t *)c->ss_bsys.p;
        k_keys_append<<<grid_for(c, N, 256), 256, 0, c->st>>>(
            N, (const double *)c->x[0].p, (const double *)c->x[1].p, (const double *)c->x[2].p,
            (const int32_t *)c->psys.p, c->S, (const SysBox *)c->box.p, (const int64_t *)c->off_dev.p,
            ss, k0, rk, rv, cnt, flag, st, c->op);
        const SmallArgs small = {(const double *)c->x[0].p, (const double *)c->x[1].p, (const double *)c->x[2].p,
                                 (const SysBox *)c->box.p,  (const int64_t *)c->off_dev.p, st, c->op};
        const int grid = std::min((c->nbk + SSB_WARPS - 1) / SSB_WARPS, c->nsm * 16);
        // up to SS_SUM_MAX buckets every block of the sort adds up the counts before its buckets (at most 32 loads
        // a thread); above, a scan does it once
        if (c->nbk <= SS_SUM_MAX) {
            k_ss_sort<false><<<grid, SSB_THREADS, 0, c->st>>>(c->nbk, c->S, c->h_ss[0].rcap, ss, bsys, cnt, rk,
                                                              rv, k0, v0, flag, small);
        } else {
            scan_u32(c, cnt, c->nbk + 1, nullptr, c->nbk + 1, nullptr, true);
            k_ss_sort<true><<<grid, SSB_THREADS, 0, c->st>>>(c->nbk, c->S, c->h_ss[0].rcap, ss, bsys, cnt, rk,
                                                              rv, k0, v0, flag, small);
        }
        c->launches += 2;
        return;
    }
    k_keys<<<grid_for(c, N, 256), 256, 0, c->st>>>(N, (const double *)c->x[0].p, (const double *)c->x[1].p,
                                                    (const double *)c->x[2].p, (const int32_t *)c->psys.p, c->S,
                                                    (const SysBox *)c->box.p, k0, v0);
    c->launches++;
    uint32_t *rs = (uint32_t *)c->hist.p;
    uint32_t *counts = rs + RS_HDR, *look = counts + (size_t)2048 * c->S;
    cudaMemsetAsync(rs, 0, ((size_t)RS_HDR + (size_t)2048 * (c->S + c->nchunks)) * sizeof(uint32_t), c->st);
    k_digit_counts<<<std::min(c->nchunks, c->nsm * 4), 256, 0, c->st>>>(k0, (const Chunk *)c->chunks_dev.p, c->nchunks,
                                                                       counts);
    c->launches++;
    const int grid = std::min(c->nchunks, c->nsm * 4);
    const Chunk *chk = (const Chunk *)c->chunks_dev.p;
    for (int pass = 0; pass < 8; ++pass) {
        uint32_t *lk = look + (size_t)pass * 256 * c->nchunks;
        uint32_t *tk = rs + pass;
        switch (c->ipt) {
        case 2: k_onesweep<2><<<grid, 256, 0, c->st>>>(k0, v0, k1, v1, chk, c->nchunks, pass, counts, lk, tk, N, st); break;
        case 4: k_onesweep<4><<<grid, 256, 0, c->st>>>(k0, v0, k1, v1, chk, c->nchunks, pass, counts, lk, tk, N, st); break;
        default: k_onesweep<8><<<grid, 256, 0, c->st>>>(k0, v0, k1, v1, chk, c->nchunks, pass, counts, lk, tk, N, st);
        }
        c->launches++;
        std::swap(k0, k1);
        std::swap(v0, v1);
    }
    // after 8 passes the sorted keys/values are back in buffer 0
}

void launch_permute(hybrid_ctx *c)
{
    const int64_t N = c->N;
    uint32_t *v0 = (uint32_t *)c->vals[0].p;
    PermArgs a;
    for (int f = 0; f < 7; ++f) {
        a.xin[f] = (const double *)c->x[f].p;
        a.xout[f] = (double *)c->xa[f].p;
    }
    a.id_in = (const int32_t *)c->id.p;
    a.id_out = (int32_t *)c->ida.p;
    a.orig_in = (const int32_t *)c->orig.p;
    a.orig_out = (int32_t *)c->origa.p;
    a.src = v0;
    a.phi = c->p.precision == 1 ? (float4 *)c->phi.p : nullptr;
    a.plo = c->p.precision == 1 ? (float4 *)c->plo.p : nullptr;
    a.pd = c->p.precision == 0 ? (double4_32a *)c->pd.p : nullptr;
    a.disp = c->p.skin > 0.0 ? (float *)c->disp.p : nullptr;
    a.psys = (const int32_t *)c->psys.p;
    a.box = (const SysBox *)c->box.p;
    a.N = N;
    a.bmin = (unsigned long long *)c->boxmin.p;
    a.bmax = (unsigned long long *)c->boxmax.p;
    a.S = c->S;
    a.flag = (uint32_t *)c->ss_flag.p;
    if (N <= 1 << 18) k_permute<4><<<grid_for(c, N, 256), 256, 0, c->st>>>(a);
    else k_permute<8><<<grid_for(c, N, 256), 256, 0, c->st>>>(a);
    c->launches++;
    for (int f = 0; f < 7; ++f) std::swap(c->x[f], c->xa[f]);
    std::swap(c->id, c->ida);
    std::swap(c->orig, c->origa);
    c->swaps ^= 1;
}

// rows of the topology's tiles, and tiles of N + 1 positions (the end of the batch is one)
static int cell_rows(int64_t N)
{
    return N / (CT_MAX / 4) < CT_SUM_MAX ? 1 : (N / (CT_MAX / 2) < CT_SUM_MAX ? 2 : 4);
}
static int cell_tiles(int64_t N) { return (int)(N / (CT_WARPS * 32 * cell_rows(N))) + 1; }

// counts of every batch of up to N particles
size_t cell_count_bytes(int64_t N)
{
    return (size_t)CT_CNT * (std::max<int64_t>(CT_SUM_MAX, N / CT_MAX) + 1) * sizeof(uint32_t);
}

// FP32 form: b_max of the larger cells by search instead of taking every particle (see k_finish)
static bool bmax_by_search(const hybrid_ctx *c) { return c->p.precision == 1 && c->N > (int64_t)1 << 20; }

// sink groups marked with the cells (k_cells, k_nodes) or, for a large n_crit, from the nodes afterwards
static bool groups_in_nodes(const hybrid_ctx *c) { return c->p.n_crit <= GROUP_WINDOW; }

void launch_topology(hybrid_ctx *c)
{
    Status *st = status_dev(c);
    const int64_t N = c->N;
    const bool groups = groups_in_nodes(c);
    const int n_crit = groups ? c->p.n_crit : 0;
    const uint64_t *keys = (const uint64_t *)c->keys[0].p;
    const int32_t *psys = (const int32_t *)c->psys.p;
    uint64_t *d_tot = (uint64_t *)((char *)c->lvl.p + 256);
    uint32_t *cnt = (uint32_t *)c->ccnt.p;
    uint16_t *cells = (uint16_t *)c->cells.p;
    const int rows = cell_rows(N), ntiles = cell_tiles(N);
    const int grid = std::min(ntiles, c->nsm * 8);
    const size_t sh = 2 * (size_t)cells_bytes(std::max(c->p.n_leaf, n_crit));
    auto *kc = rows == 1 ? k_cells<1> : (rows == 2 ? k_cells<2> : k_cells<4>);
    kc<<<grid, 32 * CT_WARPS, sh, c->st>>>(N, c->S, keys, psys, c->p.n_leaf, n_crit, cells, ntiles, cnt,
                                           (unsigned long long *)c->counter.p, st);
    if (ntiles > CT_SUM_MAX) scan_u32(c, cnt, (int64_t)CT_CNT * ntiles, nullptr, (int64_t)CT_CNT * ntiles, d_tot);
    NodeArgs a;
    a.cells = cells;
    a.psys = psys;
    a.off = cnt;
    a.total = d_tot;
    a.nfirst = (uint32_t *)c->nfirst.p;
    a.nend = (uint32_t *)c->nend.p;
    a.nlevel = (uint32_t *)c->nlevel.p;
    a.nchild = (uint32_t *)c->nchild.p;
    a.nchend = (uint32_t *)c->nchend.p;
    a.nparent = (uint32_t *)c->nparent.p;
    a.sysroot = (uint32_t *)c->sysroot.p;
    a.lvl = (uint32_t *)c->lvl.p;
    a.done = (uint32_t *)c->ndone.p;
    a.bmax64 = c->p.precision == 0 ? (unsigned long long *)c->nbmax.p : nullptr;
    a.bmax32 = c->p.precision == 0 || bmax_by_search(c) ? nullptr : (unsigned int *)c->nbmax32.p;
    a.gnode = groups ? (uint32_t *)c->gnode.p : nullptr;
    a.gfirst = (uint32_t *)c->gfirst.p;
    a.gsys = (uint32_t *)c->gsys.p;
    a.ngroups = (int64_t *)c->ngroups_dev.p;
    a.N = N;
    a.cap = c->capNodes;
    a.ntiles = ntiles;
    if (ntiles > CT_SUM_MAX) k_nodes<4, true><<<grid, 32 * CT_WARPS, 0, c->st>>>(a, st, c->op);
    else if (rows == 1) k_nodes<1, false><<<ntiles, 32 * CT_WARPS, 0, c->st>>>(a, st, c->op);
    else if (rows == 2) k_nodes<2, false><<<ntiles, 32 * CT_WARPS, 0, c->st>>>(a, st, c->op);
    else k_nodes<4, false><<<ntiles, 32 * CT_WARPS, 0, c->st>>>(a, st, c->op);
    c->launches += 2;
    c->walk_clean = true;
}

static FinArgs fin_args(hybrid_ctx *c)
{
    FinArgs f;
    f.lvl = (const uint32_t *)c->lvl.p;
    f.nfirst = (const uint32_t *)c->nfirst.p;
    f.nend = (const uint32_t *)c->nend.p;
    f.nchend = (const uint32_t *)c->nchend.p;
    f.nchild = (const uint32_t *)c->nchild.p;
    f.nlevel = (const uint32_t *)c->nlevel.p;
    f.key = (const uint64_t *)c->keys[0].p;
    f.psys = (const int32_t *)c->psys.p;
    f.S = c->S;
    f.box = (const SysBox *)c->box.p;
    f.sp = (const SysParams *)c->sp_dev.p;
    f.M = (double *)c->nM.p;
    f.cx = (double *)c->ncx.p;
    f.cy = (double *)c->ncy.p;
    f.cz = (double *)c->ncz.p;
    f.B2 = (double *)c->nB2.p;
    f.bmax = (unsigned long long *)c->nbmax.p;
    f.bmax32 = (unsigned int *)c->nbmax32.p;
    f.nA = (const float4 *)c->nA.p;
    f.nB = (const float4 *)c->nB.p;
    f.crit = (float2 *)c->ncrit.p;
    f.topo = (uint4 *)c->ntopo.p;
    f.nD = (double4_32a *)c->nD.p;
    f.rb = (double *)c->nrb.p;
    f.hr = (double *)c->nhr.p;
    f.delta = (double *)c->ndelta.p;
    f.side = (double *)c->nside.p;
    f.org = (double *)c->norg.p;
    return f;
}

void launch_moments(hybrid_ctx *c)
{
    Status *st = status_dev(c);
    MomArgs a;
    a.lvl = (const uint32_t *)c->lvl.p;
    a.nfirst = (const uint32_t *)c->nfirst.p;
    a.nend = (const uint32_t *)c->nend.p;
    a.nchend = (const uint32_t *)c->nchend.p;
    a.nchild = (const uint32_t *)c->nchild.p;
    a.nparent = (const uint32_t *)c->nparent.p;
    a.nlevel = (const uint32_t *)c->nlevel.p;
    a.x = (const double *)c->x[0].p;
    a.y = (const double *)c->x[1].p;
    a.z = (const double *)c->x[2].p;
    a.m = (const double *)c->x[6].p;
    a.key = (const uint64_t *)c->keys[0].p;
    a.psys = (const int32_t *)c->psys.p;
    a.S = c->S;
    a.box = (const SysBox *)c->box.p;
    a.M = (double *)c->nM.p;
    a.cx = (double *)c->ncx.p;
    a.cy = (double *)c->ncy.p;
    a.cz = (double *)c->ncz.p;
    a.B2 = (double *)c->nB2.p;
    a.nA = (float4 *)c->nA.p;
    a.nB = (float4 *)c->nB.p;
    a.done = (uint32_t *)c->ndone.p;
    a.bmax64 = (unsigned long long *)c->nbmax.p;
    a.bmax32 = (unsigned int *)c->nbmax32.p;
    a.search = bmax_by_search(c);
    a.phi = (const float4 *)c->phi.p;
    a.plo = (const float4 *)c->plo.p;
    unsigned long long *nitems = (unsigned long long *)c->counter.p + 9;
    const int gridw = grid_for(c, c->capNodes * 32, 256, 16);
    uint32_t *bigbase = (uint32_t *)c->nbig.p, *items = (uint32_t *)c->mitems.p;
    const FinArgs f = fin_args(c);
    if (c->p.precision == 0) {
        k_mom_small<true><<<gridw, 256, 0, c->st>>>(a, nitems, bigbase, items, (uint32_t)c->capItems, st, c->op);
        k_bmax_big<true><<<gridw, 256, 0, c->st>>>(a, nitems, bigbase, items, st);
        k_finalize<<<grid_for(c, c->capNodes, 256, 8), 256, 0, c->st>>>(f, st);
        c->launches += 3;
    } else {
        k_mom_small<false><<<gridw, 256, 0, c->st>>>(a, nitems, bigbase, items, (uint32_t)c->capItems, st, c->op);
        const int gridf = grid_for(c, c->capNodes, BIG_THREADS, 16);
        if (a.search) {
            k_finish<true><<<gridf, BIG_THREADS, 0, c->st>>>(a, f, nitems, items, st);
        } else {
            k_bmax_big<false><<<gridw, 256, 0, c->st>>>(a, nitems, bigbase, items, st);
            k_finish<false><<<gridf, BIG_THREADS, 0, c->st>>>(a, f, nitems, items, st);
            c->launches += 1;
        }
        c->launches += 2;
    }
}

void launch_inspect(hybrid_ctx *c)
{
    if (c->p.precision == 0) return;
    k_inspect<<<grid_for(c, c->capNodes, 256, 8), 256, 0, c->st>>>(fin_args(c));
    c->launches += 1;
}

void launch_groups(hybrid_ctx *c)
{
    if (groups_in_nodes(c)) return;
    Status *st = status_dev(c);
    const int64_t N = c->N;
    cudaMemsetAsync(c->gflag.p, 0xff, (size_t)N * sizeof(uint32_t), c->st);
    k_group_flag<<<grid_for(c, c->capNodes, 256), 256, 0, c->st>>>(
        (const uint32_t *)c->lvl.p, (const uint32_t *)c->nfirst.p, (const uint32_t *)c->nend.p,
        (const uint32_t *)c->nchild.p, (const uint32_t *)c->nparent.p, c->p.n_crit, (uint32_t *)c->gflag.p, st);
    k_group_mark<<<grid_for(c, N, 256), 256, 0, c->st>>>(N, (const uint32_t *)c->gflag.p, (uint32_t *)c->gscan.p, st);
    uint64_t *d_tot = (uint64_t *)((char *)c->lvl.p + 64 * sizeof(uint32_t) + 64 + 8);
    scan_u32(c, (uint32_t *)c->gscan.p, N, nullptr, N, d_tot);
    k_group_compact<<<grid_for(c, N, 256), 256, 0, c->st>>>(
        N, (const uint32_t *)c->gflag.p, (const uint32_t *)c->gscan.p, (const int32_t *)c->psys.p,
        (uint32_t *)c->gnode.p, (uint32_t *)c->gfirst.p, (uint32_t *)c->gsys.p, d_tot, (int64_t *)c->ngroups_dev.p, st);
    c->launches += 3;
}

void launch_group_boxes(hybrid_ctx *c)
{
    Status *st = status_dev(c);
    const int64_t N = c->N;
    k_group_box<<<grid_for(c, N * 32 / 16, 256), 256, 0, c->st>>>(
        (const int64_t *)c->ngroups_dev.p, (const uint32_t *)c->gfirst.p, (const double *)c->x[0].p, (const double *)c->x[1].p, (const double *)c->x[2].p, (const int32_t *)c->psys.p,
        (const SysBox *)c->box.p, (double *)c->glo.p, (double *)c->ghi.p, (GroupF *)c->gF.p, st);
    c->launches += 1;
}

cudaError_t init_tree_kernels()
{
    // leaves of up to 24448 particles, as far as their window fits in shared memory
    for (auto *k : {k_cells<1>, k_cells<2>, k_cells<4>}) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * cells_bytes(24448));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void launch_wait_selftest(hybrid_ctx *c, int max_polls)
{
    uint32_t *word = (uint32_t *)((unsigned long long *)c->counter.p + 15);   // a slot nothing else uses
    cudaMemsetAsync(word, 0, sizeof(uint32_t), c->st);
    k_wait_selftest<<<1, 32, 0, c->st>>>(word, max_polls, status_dev(c));
    c->launches++;
}

}  // namespace hy
