// walk.cu -- grouped tree walk that emits interaction lists (Sec. II-B
// traversal rule; Eq. 11 with the box of a sink group in place of the n_vec
// sinks; Eq. 15 for the hard neighbours and for the cutoff test).
//
// One warp walks one group at a time, starting at its system's root. Each
// iteration pops up to 32 pending cells (one per lane) from a per-warp stack,
// tests them, and with warp ballots/scans appends:
//   cells           taken whole: r >= r_b and r >= R2 + b_max (K = 0 for
//                   every pair, weight 1),
//   far particles   members of leaves the soft walk opens with
//                   r >= R2 + b_max (K = 0 for every pair, weight 1),
//   near particles  members of leaves with r < R2 + b_max, reached by the
//                   soft or the hard walk: the only pairs where K can be
//                   non-zero (soft weight 1 - K, hard weight K),
// and pushes the children of opened cells. r is the distance from the cell's
// centre of mass to the group box.
//
// FP32 form (one pass): each warp writes the three kinds of entries into
// regions of the list buffer it claims with an atomic add (at least
// WALK_REGION entries per kind at a time), so a group's entries of one kind
// are contiguous until a region runs out; every contiguous run becomes pair
// work items of at most item_len entries, appended to the far (cells, far
// particles) or near item array, which the pair kernels consume directly (the
// near items of groups well inside R2 from the array's other end).
// FP64 form (two passes): the count pass sizes every list, a scan turns
// counts into offsets, and the fill pass writes them (one list per group and
// kind, for the deterministic FP64 pair kernel).
#include "hy_internal.cuh"

namespace hy {

namespace {

constexpr int WALK_THREADS = 128;

struct WalkArgs {
    const int64_t *ngroups;
    const uint32_t *gnode, *gsys;
    const GroupF *gF;
    const double *glo, *ghi;
    const uint32_t *sysroot;
    const SysParams *sp;
    const uint4 *topo;
    const float4 *nA, *nB;
    const float2 *crit;
    const double4_32a *nD;
    const double *rb, *hr;
    uint64_t *cnt;          // count pass: counts; fill pass: offsets ([3][ng] + total)
    int64_t *d_n3;
    const uint64_t *list_total;
    uint32_t *list;
    int64_t cap_list;
    uint32_t *stack;
    int64_t cap_stack;
    unsigned long long *counter;
    int mode;
    Status *st;
    int where;
    unsigned long long *queue;   // [0], [1]: next far / near item or unit of the pair kernels, [6]: next dense near item;
                                 // zeroed here with
    unsigned long long *pairs;   // [0], [1]: the pair counts
    float *acc_s[3], *acc_h[3];  // FP32 form: the accelerations this walk's pair kernels add to, zeroed here
    // one-pass form
    const uint32_t *gfirst;
    unsigned long long *list_cursor;     // next free list entry
    unsigned long long *item_count;      // [0] far items, [1] near items (low half) and dense near items (high half)
    WorkItem *items_far, *items_near;
    int64_t cap_items;
    int lch_far, lch_near;               // base lengths of far and near work items
};

constexpr uint32_t WALK_REGION = 2048;
// A group is dense (near_dense in pair.cu) when its box fits in a sphere of sqrt(NEAR_DENSE) R2: its near leaves, which are
// no larger, then lie within about twice R2, and a good part of them within R2. Marked in its size (see gd).
constexpr float NEAR_DENSE = 0.7f;
constexpr uint32_t GROUP_DENSE = 0x80000000u;
constexpr int WALK_SSTK = 1024;   // entries of a warp's stack kept in shared memory (one walk iteration pushes <= 256)

__device__ __forceinline__ void fail(Status *st, int code, int where)
{
    // the first failure wins and keeps its op index: later kernels of the same sequence may fail too (a build
    // after an unsorted one), and the sequence resumes at the first
    if (atomicCAS(&st->code, 0, code) == 0) st->where = where;
}

__device__ __forceinline__ uint32_t warp_excl_scan(uint32_t v, uint32_t &total)
{
    const int lane = threadIdx.x & 31;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    total = __shfl_sync(0xffffffffu, inc, 31);
    return inc - v;
}

// square of the distance from p to the box [lo, hi], per axis max(lo - p, 0, p - hi) (signs from the bits: a
// comparison of doubles takes the FP64 pipe, 2 lanes per SM and clock)
__device__ __forceinline__ double dist2_box_f64(double p0, double p1, double p2, const double *lo, const double *hi)
{
    const double p[3] = {p0, p1, p2};
    double s = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double a = lo[d] - p[d], b = p[d] - hi[d];
        const double g = __double2hiint(a) > 0 ? a : (__double2hiint(b) > 0 ? b : 0.0);
        s += g * g;
    }
    return s;
}

// whether a distance reaches a radius, from the FP32 nearest to their squares: 1 yes, 0 no, -1 within FP32's rounding
// (or out of its range)
__device__ __forceinline__ int reaches(float d2, float r2)
{
    if (!(d2 > 1e-30f && r2 > 1e-30f && r2 < 1e30f)) return -1;
    return d2 > r2 * 1.000001f ? 1 : (d2 < r2 * 0.999999f ? 0 : -1);
}

// What the pair kernels after this walk count from (the far counts only when the soft force follows).
__device__ __forceinline__ void clear_pair_counters(const WalkArgs &a)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.queue[0] = a.queue[1] = a.queue[6] = 0ull;
        if (a.mode & 1) a.pairs[0] = 0ull;
        a.pairs[1] = 0ull;
    }
}

// FP64 form: count pass, then fill pass, the same walk twice. Tests are decided in FP32 wherever its rounding allows,
// and the emission is k_walk1's.
template <bool FILL>
__global__ void __launch_bounds__(WALK_THREADS) k_walk(WalkArgs a)
{
    Status *st = a.st;
    if (st->code) return;
    if (FILL) clear_pair_counters(a);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t ng = *a.ngroups;
    if (!FILL && blockIdx.x == 0 && threadIdx.x == 0) *a.d_n3 = 3 * ng;
    if (FILL) {
        const uint64_t total = *a.list_total;
        if ((int64_t)total > a.cap_list) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                fail(st, HYBRID_ECAPACITY, a.where);
                st->need[1] = (int64_t)total;
            }
            return;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) a.cnt[3 * ng] = total;
    }
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    uint32_t *stk = a.stack + gw * a.cap_stack;   // overflow part of the stack (older entries)
    __shared__ uint32_t sstk_all[WALK_THREADS / 32][WALK_SSTK];
    uint32_t *sstk = sstk_all[threadIdx.x >> 5];  // top part of the stack
    const bool want_soft = a.mode & 1, want_hard = (a.mode >> 1) & 1;

    // A warp's first group by its place in the grid, the later ones in turn. Taken in turn from the start, neighbouring
    // groups, which are heavy together, go to the four warps of a block and their SM's FP64 pipe: walks of one step at
    // N = 30011 0.497 -> 0.320 ms, of 5 at N = 4096 0.319 -> 0.288.
    int64_t g = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (g < ng) {
        const uint32_t s = a.gsys[g];
        const bool has_hard = a.sp[s].has_hard != 0;
        const bool wh0 = want_hard && has_hard;
        double blo[3], bhi[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            blo[d] = a.glo[3 * g + d];
            bhi[d] = a.ghi[3 * g + d];
        }
        uint64_t nc = 0, np = 0, nh = 0, oc = 0, op = 0, oh = 0;
        if (FILL) {
            oc = a.cnt[g];
            op = a.cnt[ng + g];
            oh = a.cnt[2 * ng + g];
        }
        int sp = 0;        // entries in the shared-memory part
        int64_t gp = 0;    // entries in the global part
        if (want_soft || wh0) {
            if (lane == 0) sstk[0] = a.sysroot[s] | ((uint32_t)want_soft << 30) | ((uint32_t)wh0 << 31);
            sp = 1;
        }
        __syncwarp();
        bool overflow = false;
        // the particles of the lanes' leaves, [first, first + k) each (k = 0: none), counted or written from dst
        auto leaves = [&](uint64_t dst, uint32_t first, uint32_t k) -> uint32_t {
            if (!FILL) return __reduce_add_sync(0xffffffffu, k);
            uint32_t tot, ex;
            if (__all_sync(0xffffffffu, k < 32u)) {
                ex = tot = 0u;
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const unsigned b = __ballot_sync(0xffffffffu, (k >> q) & 1u);
                    ex += (uint32_t)__popc(b & lt) << q;
                    tot += (uint32_t)__popc(b) << q;
                }
            } else {
                ex = warp_excl_scan(k, tot);
            }
            uint32_t *to = a.list + dst + ex;
            const uint32_t most = __reduce_max_sync(0xffffffffu, k);
            for (uint32_t j = 0; j < most; j += 4)
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q)
                    if (j + q < k) to[j + q] = first + j + q;
            return tot;
        };
        while (sp > 0 || gp > 0) {
            if (sp == 0) {   // refill the shared part from the top of the global part
                const int m = (int)(gp < WALK_SSTK / 2 ? gp : WALK_SSTK / 2);
                for (int j = lane; j < m; j += 32) sstk[j] = stk[gp - m + j];
                gp -= m;
                sp = m;
                __syncwarp();
            }
            const int take = sp < 32 ? sp : 32;
            uint32_t e = 0;
            if (lane < take) e = sstk[sp - take + lane];
            sp -= take;
            __syncwarp();
            const bool valid = lane < take;
            const uint32_t c = e & 0x3fffffffu;
            const bool ws = (e >> 30) & 1u, wh = (e >> 31) & 1u;
            bool accept = false, near = false;
            uint4 T = make_uint4(NONE, 0, 0, 0);
            if (valid) {
                T = a.topo[c];
                const double4_32a D = a.nD[c];
                const float2 cr = a.crit[c];   // max(r_b, R2 + b_max)^2 and (R2 + b_max)^2
                const double d2 = dist2_box_f64(D.x, D.y, D.z, blo, bhi);
                const float d2f = narrow(d2);
                const int far_enough = reaches(d2f, cr.x), beyond = has_hard ? reaches(d2f, cr.y) : 1;
                accept = far_enough > 0;
                near = beyond == 0;
                if (far_enough < 0 || beyond < 0) {
                    const double d = sqrt(d2), hr = a.hr[c];
                    if (far_enough < 0) accept = d >= a.rb[c] && d >= hr;
                    if (beyond < 0) near = d < hr;
                }
            }
            const bool leaf = (T.y == 0);
            const bool open_s = ws && !accept;             // the soft walk goes on below c
            const bool open_h = wh && near;                // the hard walk goes on below c
            const bool take_cell = valid && ws && accept;
            const bool soft_leaf = valid && leaf && open_s && !near;        // far particles
            const bool hard_leaf = valid && leaf && (open_s || open_h) && near;   // near particles
            const bool open = valid && !leaf && (open_s || open_h);
            // taken cells
            const unsigned bm = __ballot_sync(0xffffffffu, take_cell);
            if (FILL && take_cell) a.list[oc + nc + __popc(bm & lt)] = c;
            nc += (uint64_t)__popc(bm);
            if (__any_sync(0xffffffffu, soft_leaf)) np += leaves(op + np, T.z, soft_leaf ? T.w : 0u);
            if (__any_sync(0xffffffffu, hard_leaf)) nh += leaves(oh + nh, T.z, hard_leaf ? T.w : 0u);
            if (__any_sync(0xffffffffu, open)) {   // children of opened cells (at most 8 each)
                const uint32_t fl = ((uint32_t)open_s << 30) | ((uint32_t)open_h << 31);
                const uint32_t k = open ? T.y : 0u;
                uint32_t ex = 0, sum = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned b = __ballot_sync(0xffffffffu, (k >> q) & 1u);
                    ex += (uint32_t)__popc(b & lt) << q;
                    sum += (uint32_t)__popc(b) << q;
                }
                if (sp + (int)sum > WALK_SSTK) {   // move the shared part under the global part
                    if (gp + sp > a.cap_stack) {
                        overflow = true;
                        break;
                    }
                    for (int j = lane; j < sp; j += 32) stk[gp + j] = sstk[j];
                    gp += sp;
                    sp = 0;
                    __syncwarp();
                }
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j)
                    if (j < k) sstk[sp + ex + j] = (T.x + j) | fl;
                sp += (int)sum;
            }
            __syncwarp();
        }
        if (overflow) {
            if (lane == 0) {
                fail(st, HYBRID_ECAPACITY, a.where);
                st->need[2] = 2 * a.cap_stack;
            }
            break;
        }
        if (!FILL && lane == 0) {
            a.cnt[g] = nc;
            a.cnt[ng + g] = np;
            a.cnt[2 * ng + g] = nh;
        }
        unsigned long long gg = 0;
        if (lane == 0) gg = atomicAdd(a.counter, 1ull);
        g = (int64_t)__shfl_sync(0xffffffffu, gg, 0) + (int64_t)(WALK_THREADS / 32) * gridDim.x;
    }
}

// Work items, of at most per entries, of one contiguous run [start, start +
// len) of a group's entries of kind t (0 cells, 1 far particles, 2 near
// particles; those of a dense group fill the near items' array from its end);
// all lanes call it.
__device__ __forceinline__ bool emit_items(const WalkArgs &a, int t, uint64_t start, uint32_t len, uint32_t per,
                                           uint32_t first, uint32_t n, uint32_t sys, bool multi, int lane)
{
    const int cls = t == 2 ? 1 : 0;
    const bool dense = t == 2 && (n & GROUP_DENSE);
    n &= ~GROUP_DENSE;
    const uint32_t m = (len + per - 1) / per;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(a.item_count + cls, (unsigned long long)m << (dense ? 32 : 0));
    base = __shfl_sync(0xffffffffu, base, 0);
    const int64_t lo = (uint32_t)base, hi = (int64_t)(base >> 32);
    if (lo + hi + m > a.cap_items) return false;
    WorkItem *dst = (cls ? a.items_near : a.items_far) + (dense ? a.cap_items - hi - m : lo);
    for (uint32_t j = lane; j < m; j += 32) {
        WorkItem d;
        d.cbase = t == 0 ? start : 0;
        d.pbase = t == 0 ? 0 : start;
        d.Lc = t == 0 ? len : 0u;
        d.e0 = j * per;
        d.e1 = min(len, d.e0 + per);
        d.first = first;
        d.n = n | (multi ? ITEM_MULTI : 0u);
        d.sys = sys;
        dst[j] = d;
    }
    return true;
}

// One kind's place in the list buffer (0 cells, 1 far, 2 near particles), the same on every lane: the next free
// entry, the entries left in the claimed region, and the length of the group's open run, which ends at the next entry.
struct WalkRun {
    uint64_t pos;
    uint32_t left, len;
};

// FP32 form of the walk in one pass (see the top of the file). A batch of 32
// cells tests one node per lane; of its ~300 instructions most went into the
// few leaves and opened cells it has, and the SMs are bound by instructions
// and the latency of dependent ones. So the prefix sums of what the lanes emit
// are taken bit by bit from independent ballots (a scan is a chain of five
// shuffles), a kind that no lane has is skipped, entries go out in runs of
// predicated stores, and the places in the list buffer are kept on every lane.
// (All lanes writing one owner's entries after the other was slower from two
// owners up.) Walk per soft step: N = 4096 0.132 -> 0.109 ms, 2^17 0.277 ->
// 0.241, 2^20 (absolute MAC) 0.633 -> 0.528, 2^24 24.4 -> 20.9 ms.
// MINB blocks per SM: 6 (80 registers) for batches of at most 2^20 particles, whose groups are fewer than the
// resident warps; 8 (64 registers, a few spilled) above, where more warps hide more of the node loads.
template <int MINB>
__global__ void __launch_bounds__(WALK_THREADS, MINB) k_walk1(WalkArgs a)
{
    Status *st = a.st;
    if (st->code) return;
    clear_pair_counters(a);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t ng = *a.ngroups;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    uint32_t *stk = a.stack + gw * a.cap_stack;   // overflow part of the stack (older entries)
    __shared__ uint32_t sstk_all[WALK_THREADS / 32][WALK_SSTK];
    uint32_t *sstk = sstk_all[threadIdx.x >> 5];    // top part of the stack
    const bool want_soft = a.mode & 1, want_hard = (a.mode >> 1) & 1;
    WalkRun run[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) run[t] = WalkRun{0, 0, 0};
    bool fail_list = false, fail_items = false, overflow = false;

    for (;;) {
        unsigned long long gg = 0;
        if (lane == 0) gg = atomicAdd(a.counter, 1ull);
        const int64_t g = (int64_t)__shfl_sync(0xffffffffu, gg, 0);
        if (g >= ng) break;
        const uint32_t s = a.gsys[g];
        const bool has_hard = a.sp[s].has_hard != 0;
        const bool wh0 = want_hard && has_hard;
        const uint32_t gfirst = a.gfirst[g], gn = a.gfirst[g + 1] - gfirst;
        const GroupF G = a.gF[g];
        const float cx = G.c_hi.x, cy = G.c_hi.y, cz = G.c_hi.z, hx = G.c_hi.w;
        const float lx = G.c_lo.x, ly = G.c_lo.y, lz = G.c_lo.z, hy = G.c_lo.w, hz = G.hz_root.x;
        for (uint32_t i = gfirst + lane; i < gfirst + gn; i += 32)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (want_soft) a.acc_s[d][i] = 0.0f;
                if (want_hard) a.acc_h[d][i] = 0.0f;
            }
        run[0].len = run[1].len = run[2].len = 0;
        const uint32_t per_far = item_len(gn, a.lch_far), per_near = item_len(gn, a.lch_near);
        const uint32_t gd = gn | (hx * hx + hy * hy + hz * hz < NEAR_DENSE * a.sp[s].R2sqf ? GROUP_DENSE : 0u);
        uint32_t early_far = 0, early_near = 0;   // items already emitted for this group
        int sp = 0;        // entries in the shared-memory part
        int64_t gp = 0;    // entries in the global part
        if (want_soft || wh0) {
            if (lane == 0) sstk[0] = a.sysroot[s] | ((uint32_t)want_soft << 30) | ((uint32_t)wh0 << 31);
            sp = 1;
        }
        __syncwarp();
        // room for tot more entries of kind t at run.pos (the caller moves on); closes the open run and claims a new
        // region when the current one is too small; false on failure
        auto reserve = [&](WalkRun &r, int t, uint32_t tot) -> bool {
            if (tot <= r.left) return true;
            if (r.len > 0) {
                const uint32_t per = t == 2 ? per_near : per_far;
                if (!emit_items(a, t, r.pos - r.len, r.len, per, gfirst, gd, s, true, lane)) {
                    fail_items = true;
                    return false;
                }
                (t == 2 ? early_near : early_far) += (r.len + per - 1) / per;
            }
            const uint32_t size = tot > WALK_REGION ? tot : WALK_REGION;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(a.list_cursor, (unsigned long long)size);
            base = __shfl_sync(0xffffffffu, base, 0);
            if ((int64_t)(base + size) > a.cap_list) {
                fail_list = true;
                return false;
            }
            r = WalkRun{base, size, 0};
            return true;
        };
        auto advance = [](WalkRun &r, uint32_t tot) {
            r.pos += tot;
            r.left -= tot;
            r.len += tot;
        };
        // the particles of the lanes' leaves (mine: whether this lane has one), [first, first + count) each, as entries of
        // kind t
        auto leaves = [&](WalkRun &r, int t, bool mine, uint32_t first, uint32_t count) -> bool {
            const uint32_t k = mine ? count : 0u;
            uint32_t tot, ex;
            if (__all_sync(0xffffffffu, k < 32u)) {   // bit by bit: independent ballots instead of a chain of shuffles
                ex = tot = 0u;
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const unsigned b = __ballot_sync(0xffffffffu, (k >> q) & 1u);
                    ex += (uint32_t)__popc(b & lt) << q;
                    tot += (uint32_t)__popc(b) << q;
                }
            } else {
                ex = warp_excl_scan(k, tot);
            }
            if (!reserve(r, t, tot)) return false;
            uint32_t *dst = a.list + r.pos + ex;
            const uint32_t most = __reduce_max_sync(0xffffffffu, k);
            for (uint32_t j = 0; j < most; j += 4)
#pragma unroll
                for (uint32_t q = 0; q < 4; ++q)
                    if (j + q < k) dst[j + q] = first + j + q;
            advance(r, tot);
            return true;
        };
        while (sp > 0 || gp > 0) {
            if (sp == 0) {   // refill the shared part from the top of the global part
                const int m = (int)(gp < WALK_SSTK / 2 ? gp : WALK_SSTK / 2);
                for (int j = lane; j < m; j += 32) sstk[j] = stk[gp - m + j];
                gp -= m;
                sp = m;
                __syncwarp();
            }
            const int take = sp < 32 ? sp : 32;
            uint32_t e = 0;
            if (lane < take) e = sstk[sp - take + lane];
            sp -= take;
            __syncwarp();
            const bool valid = lane < take;
            const uint32_t c = e & 0x3fffffffu;
            const bool ws = (e >> 30) & 1u, wh = (e >> 31) & 1u;
            bool accept = false, near = false;
            uint4 T = make_uint4(NONE, 0, 0, 0);
            if (valid) {
                T = a.topo[c];
                const float4 A = a.nA[c], B = a.nB[c];
                const float2 cr = a.crit[c];
                const float rx = fmaxf(fabsf((A.x - cx) + (B.x - lx)) - hx, 0.0f);
                const float ry = fmaxf(fabsf((A.y - cy) + (B.y - ly)) - hy, 0.0f);
                const float rz = fmaxf(fabsf((A.z - cz) + (B.z - lz)) - hz, 0.0f);
                const float d2 = rx * rx + ry * ry + rz * rz;
                accept = d2 >= cr.x;
                near = has_hard && (d2 < cr.y);
            }
            const bool leaf = (T.y == 0);
            const bool open_s = ws && !accept;
            const bool open_h = wh && near;
            const bool take_cell = valid && ws && accept;
            const bool soft_leaf = valid && leaf && open_s && !near;
            const bool hard_leaf = valid && leaf && (open_s || open_h) && near;
            const bool open = valid && !leaf && (open_s || open_h);
            const unsigned cm = __ballot_sync(0xffffffffu, take_cell), fm = __ballot_sync(0xffffffffu, soft_leaf);
            const unsigned nm = __ballot_sync(0xffffffffu, hard_leaf), om = __ballot_sync(0xffffffffu, open);
            if (cm) {
                if (!reserve(run[0], 0, (uint32_t)__popc(cm))) break;
                if (take_cell) a.list[run[0].pos + __popc(cm & lt)] = c;
                advance(run[0], (uint32_t)__popc(cm));
            }
            if (fm && !leaves(run[1], 1, soft_leaf, T.z, T.w)) break;
            if (nm && !leaves(run[2], 2, hard_leaf, T.z, T.w)) break;
            if (om) {   // children of opened cells (at most 8 each)
                const uint32_t fl = ((uint32_t)open_s << 30) | ((uint32_t)open_h << 31);
                const uint32_t k = open ? T.y : 0u;
                uint32_t ex = 0, sum = 0;   // the earlier lanes' counts, bit by bit, and all of them
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned b = __ballot_sync(0xffffffffu, (k >> q) & 1u);
                    ex += (uint32_t)__popc(b & lt) << q;
                    sum += (uint32_t)__popc(b) << q;
                }
                const int tot = (int)sum;
                if (sp + tot > WALK_SSTK) {   // move the shared part under the global part
                    if (gp + sp > a.cap_stack) {
                        overflow = true;
                        break;
                    }
                    for (int j = lane; j < sp; j += 32) stk[gp + j] = sstk[j];
                    gp += sp;
                    sp = 0;
                    __syncwarp();
                }
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j)
                    if (j < k) sstk[sp + ex + j] = (T.x + j) | fl;
                sp += tot;
            }
            __syncwarp();
        }
        if (overflow || fail_list || fail_items) break;
        // the group's final runs: several items of one kind add atomically, a single one stores
        uint32_t fin_far = early_far, fin_near = early_near;
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const uint32_t per = t == 2 ? per_near : per_far;
            (t == 2 ? fin_near : fin_far) += (run[t].len + per - 1) / per;
        }
#pragma unroll
        for (int t = 0; t < 3; ++t)
            if (run[t].len > 0 && !fail_items)
                if (!emit_items(a, t, run[t].pos - run[t].len, run[t].len, t == 2 ? per_near : per_far, gfirst, gd, s,
                                (t == 2 ? fin_near : fin_far) > 1, lane))
                    fail_items = true;
        if (fail_items) break;
    }
    if (lane == 0) {
        if (overflow) {
            fail(st, HYBRID_ECAPACITY, a.where);
            st->need[2] = 2 * a.cap_stack;
        }
        if (fail_list) {
            fail(st, HYBRID_ECAPACITY, a.where);
            atomicMax((unsigned long long *)&st->need[1], (unsigned long long)(2 * a.cap_list));
        }
        if (fail_items) {
            fail(st, HYBRID_ECAPACITY, a.where);
            atomicMax((unsigned long long *)&st->need[3], (unsigned long long)(2 * a.cap_items));
        }
    }
}

}  // namespace

void launch_walk(hybrid_ctx *c, int mode)
{
    Status *st = status_dev(c);
    WalkArgs a;
    a.ngroups = (const int64_t *)c->ngroups_dev.p;
    a.gnode = (const uint32_t *)c->gnode.p;
    a.gsys = (const uint32_t *)c->gsys.p;
    a.gF = (const GroupF *)c->gF.p;
    a.glo = (const double *)c->glo.p;
    a.ghi = (const double *)c->ghi.p;
    a.sysroot = (const uint32_t *)c->sysroot.p;
    a.sp = (const SysParams *)c->sp_dev.p;
    a.topo = (const uint4 *)c->ntopo.p;
    a.nA = (const float4 *)c->nA.p;
    a.nB = (const float4 *)c->nB.p;
    a.crit = (const float2 *)c->ncrit.p;
    a.nD = (const double4_32a *)c->nD.p;
    a.rb = (const double *)c->nrb.p;
    a.hr = (const double *)c->nhr.p;
    a.cnt = (uint64_t *)c->lcnt.p;
    int64_t *d_n3 = (int64_t *)c->counter.p + 4;
    uint64_t *d_total = (uint64_t *)c->counter.p + 5;
    a.d_n3 = d_n3;
    a.list_total = d_total;
    a.list = (uint32_t *)c->list.p;
    a.cap_list = c->capList;
    a.stack = (uint32_t *)c->stack.p;
    a.cap_stack = c->capStack;
    a.mode = mode;
    a.st = st;
    a.where = c->op;
    a.gfirst = (const uint32_t *)c->gfirst.p;
    a.queue = (unsigned long long *)c->counter.p + 2;
    a.pairs = (unsigned long long *)c->counter.p + 6;
    for (int d = 0; d < 3; ++d) {
        a.acc_s[d] = (float *)c->acc_s[d].p;
        a.acc_h[d] = (float *)c->acc_h[d].p;
    }
    a.list_cursor = (unsigned long long *)c->counter.p + 10;
    a.item_count = (unsigned long long *)c->counter.p + 11;
    a.items_far = (WorkItem *)c->wmap.p;
    a.items_near = (WorkItem *)c->wnear.p;
    a.cap_items = c->capWork;
    // Far items: on a small job short items even out the warps' ends; on a large job long ones hide the set-up of
    // each item (its descriptor, sinks and first gathers) behind more tiles.
    const bool small_job = c->N <= (int64_t)1 << 20;
    // Near items (one block each, tiles of 128 sources): as long as there are enough of them for every resident block.
    // Near time per step with 64, 128, 256 entries: N = 2^12 0.071, 0.077, 0.083 ms; 2^17 0.292, 0.256, 0.266;
    // 2^20 1.51, 1.17, 1.09; with 512 and 1024: 2^24 35.6, 35.2.
    a.lch_near = c->N <= 1 << 15 ? 64 : (c->N <= 1 << 18 ? 128 : (c->N <= 1 << 20 ? 256 : 1024));
    // Far time per step with 64, 128, 256 entries: N = 2^10 0.029, 0.033, 0.034 ms; 2^12 0.038, 0.045, 0.055; 2^14
    // 0.061, 0.062, 0.065; 2^15 0.105, 0.099, 0.103; 2^17 0.391, 0.335, 0.319.
    a.lch_far = c->N <= 1 << 14 ? 64 : (small_job ? LCH_FAR_SMALL : LCH_FAR);
    const int grid = c->walk_warps * 32 / WALK_THREADS;
    cudaEvent_t e0 = nullptr;
    prof_begin(c, PROF_WALK, &e0);
    // the group counters, the list cursor and the item counts start at 0: the build before this walk zeroed them
    if (!c->walk_clean) {
        cudaMemsetAsync(c->counter.p, 0, 2 * sizeof(unsigned long long), c->st);
        cudaMemsetAsync((unsigned long long *)c->counter.p + 10, 0, 3 * sizeof(unsigned long long), c->st);
    }
    c->walk_clean = false;
    c->pairs_clean = mode;
    if (c->p.precision == 1) {   // one pass
        a.counter = (unsigned long long *)c->counter.p;
        if (small_job) k_walk1<6><<<grid, WALK_THREADS, 0, c->st>>>(a);
        else k_walk1<8><<<grid, WALK_THREADS, 0, c->st>>>(a);
        prof_end(c, PROF_WALK, e0);
        c->launches += 1;
        c->last_walk_mode = mode;
        return;
    }
    // count pass
    a.counter = (unsigned long long *)c->counter.p;
    k_walk<false><<<grid, WALK_THREADS, 0, c->st>>>(a);
    scan_u64(c, (uint64_t *)c->lcnt.p, 0, d_n3, 3 * c->capGroups, d_total);
    // fill pass
    a.counter = (unsigned long long *)c->counter.p + 1;
    k_walk<true><<<grid, WALK_THREADS, 0, c->st>>>(a);
    prof_end(c, PROF_WALK, e0);
    c->launches += 2;
    c->last_walk_mode = mode;
}

}  // namespace hy
