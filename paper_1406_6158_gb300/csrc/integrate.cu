// integrate.cu -- leap-frog kick and drift (Eq. 3-4), the copies between the
// caller's arrays and the context's working state, and the energy diagnostic.
//
// Kicks and drifts run in FP64 with one rounding per product and per sum
// (v <- v + h a; x <- x + dt v), in the order the integrator states them, so
// the FP64 path reproduces a plain CPU evaluation of the same sequence.
#include "hy_internal.cuh"

#include "energy_pairs.cuh"
#include "root_box.cuh"

namespace hy {

namespace {

struct StatePtrs {
    double *x[7];
    int32_t *id, *orig, *psys;
    void *as[3], *ah[3];
    float4 *phi, *plo;      // FP32 hi/lo positions (precision 1)
    float *disp;            // distance bound since the last build (skin > 0), or null
    const SysBox *box;
};

__device__ __forceinline__ void fail(Status *st, int code, int where)
{
    // the first failure wins and keeps its op index: later kernels of the same sequence may fail too (a build
    // after an unsorted one), and the sequence resumes at the first
    if (atomicCAS(&st->code, 0, code) == 0) st->where = where;
}

// system of batch position i: binary search over the offsets (S + 1 entries)
__device__ __forceinline__ int sys_of(const int64_t *__restrict__ off, int S, int64_t i)
{
    int lo = 0, hi = S;   // off[lo] <= i < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= i) lo = mid;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(256) k_copy_in(int64_t N, int S, const int64_t *__restrict__ off,
                                                 const SysIO *__restrict__ io, StatePtrs w, int prec, int with_acc,
                                                 unsigned long long *bmin, unsigned long long *bmax, uint32_t *ss_flag)
{
    // a new state: empty root boxes and no verdict on the sample sort's splitters yet
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < 3 * S; k += gridDim.x * blockDim.x) {
        bmin[k] = ~0ull;
        bmax[k] = 0ull;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ss_flag[1] = 0u;
    for (int64_t gi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gi < N; gi += (int64_t)gridDim.x * blockDim.x) {
        const int s = sys_of(off, S, gi);
        const SysIO &y = io[s];
        const int64_t li = gi - y.off;
#pragma unroll
        for (int f = 0; f < 7; ++f) w.x[f][gi] = y.x[f][li];
        w.id[gi] = y.id ? y.id[li] : (int32_t)li;
        w.orig[gi] = (int32_t)li;
        w.psys[gi] = s;
        if (with_acc) {
            for (int d = 0; d < 3; ++d) {
                if (prec == 1) {
                    ((float *)w.as[d])[gi] = ((const float *)y.as[d])[li];
                    ((float *)w.ah[d])[gi] = ((const float *)y.ah[d])[li];
                } else {
                    ((double *)w.as[d])[gi] = ((const double *)y.as[d])[li];
                    ((double *)w.ah[d])[gi] = ((const double *)y.ah[d])[li];
                }
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_copy_out(int64_t N, const int32_t *__restrict__ psys,
                                                  const SysIO *__restrict__ io, StatePtrs w, int prec, int state,
                                                  int acc_s, int acc_h, const Status *st)
{
    if (st->code) return;
    for (int64_t gi = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; gi < N; gi += (int64_t)gridDim.x * blockDim.x) {
        const SysIO &y = io[psys[gi]];
        const int64_t li = gi - y.off;
        if (state) {
#pragma unroll
            for (int f = 0; f < 7; ++f) y.x[f][li] = w.x[f][gi];
            if (y.id) y.id[li] = w.id[gi];
        }
        for (int d = 0; d < 3; ++d) {
            if (prec == 1) {
                if (acc_s) ((float *)y.as[d])[li] = ((const float *)w.as[d])[gi];
                if (acc_h) ((float *)y.ah[d])[li] = ((const float *)w.ah[d])[gi];
            } else {
                if (acc_s) ((double *)y.as[d])[li] = ((const double *)w.as[d])[gi];
                if (acc_h) ((double *)y.ah[d])[li] = ((const double *)w.ah[d])[gi];
            }
        }
    }
}

struct KickSpec {
    int n;            // number of kicks, applied in order
    int which[4];     // 0 soft, 1 hard
    int mode[4];      // 0: h = val; 1: h = dt_soft / 2; 2: h = (dt_soft / n_hard) / 2
    double val[4];
    int dmode;        // -1: no drift; 0: dt = dval; 2: dt = dt_soft / n_hard
    double dval;
    int resplit;      // after the drift: new FP32 hi/lo positions and the distance bound (reused lists)
    int where;        // op index, recorded when a particle has moved more than skin / 2
};

// Exact FP32 -> FP64 conversion of a normal number with integer operations
// (sign, exponent rebiased by 1023 - 127, mantissa moved up 29 bits); zero keeps
// its sign, and subnormals, infinities and NaNs take the ordinary conversion.
__device__ __forceinline__ double widen(float f)
{
    const uint32_t b = __float_as_uint(f);
    const uint32_t e = (b >> 23) & 0xffu;
    const uint64_t sign = (uint64_t)(b & 0x80000000u) << 32;
    if (e == 0u || e == 0xffu) return (b & 0x7fffffffu) == 0u ? __longlong_as_double((long long)sign) : (double)f;
    return __longlong_as_double((long long)(sign | ((uint64_t)(e + 896u) << 52) | ((uint64_t)(b & 0x7fffffu) << 29)));
}
__device__ __forceinline__ double widen(double f) { return f; }

// The step sizes of each kind are per-system constants (SysParams), so a
// particle's update is the three products and sums per vector and nothing else.
// Every array a particle needs is loaded before the first kick: at small sizes
// the launch lasts as long as its chain of loads.
// BOX: a build of this (single) system follows, and its bounds and the start of
// its sort are made here, from the positions at hand, instead of by a launch
// that reads them again (drift, bounds and key sort per soft step: N = 4096
// 0.124 -> 0.1145 ms, 2^17 0.178 -> 0.1635 ms; 2^24 unchanged).
template <typename A, bool BOX>
__global__ void __launch_bounds__(256) k_kick_drift(int64_t N, StatePtrs w, const SysParams *__restrict__ sp,
                                                    KickSpec ks, int S, Status *st, BoxArgs box)
{
    const bool skip = st->code != 0;
    if (!BOX && skip) return;
    Bounds bounds;
    if (BOX) begin_sort(box);
    bool soft = false, hard = false, tripped = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        soft = soft || (k < ks.n && ks.which[k] == 0);
        hard = hard || (k < ks.n && ks.which[k] != 0);
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const SysParams &P = sp[S == 1 ? 0 : w.psys[i]];
        double v0 = w.x[3][i], v1 = w.x[4][i], v2 = w.x[5][i], x0 = 0.0, x1 = 0.0, x2 = 0.0;
        A s0 = 0, s1 = 0, s2 = 0, h0 = 0, h1 = 0, h2 = 0;
        if (soft) {
            s0 = ((const A *)w.as[0])[i];
            s1 = ((const A *)w.as[1])[i];
            s2 = ((const A *)w.as[2])[i];
        }
        if (hard) {
            h0 = ((const A *)w.ah[0])[i];
            h1 = ((const A *)w.ah[1])[i];
            h2 = ((const A *)w.ah[2])[i];
        }
        if (ks.dmode >= 0) {
            x0 = w.x[0][i];
            x1 = w.x[1][i];
            x2 = w.x[2][i];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < ks.n) {
                const double h = ks.mode[k] == 1 ? P.h_soft : ks.mode[k] == 2 ? P.h_hard : ks.val[k];
                const bool hd = ks.which[k] != 0;
                v0 = __dadd_rn(v0, __dmul_rn(h, widen(hd ? h0 : s0)));
                v1 = __dadd_rn(v1, __dmul_rn(h, widen(hd ? h1 : s1)));
                v2 = __dadd_rn(v2, __dmul_rn(h, widen(hd ? h2 : s2)));
            }
        if (BOX && skip) {   // after a failure the state stays, but the build sorts it all the same
            bounds.add(x0, x1, x2);
            continue;
        }
        w.x[3][i] = v0;
        w.x[4][i] = v1;
        w.x[5][i] = v2;
        if (ks.dmode >= 0) {
            const double dt = ks.dmode == 0 ? ks.dval : P.dt_hard;
            x0 = __dadd_rn(x0, __dmul_rn(dt, v0));
            x1 = __dadd_rn(x1, __dmul_rn(dt, v1));
            x2 = __dadd_rn(x2, __dmul_rn(dt, v2));
            w.x[0][i] = x0;
            w.x[1][i] = x1;
            w.x[2][i] = x2;
            if (BOX) bounds.add(x0, x1, x2);
            if (ks.resplit) {
                // the pair kernels' copy of the moved positions, and the distance of this drift (from the old
                // and new hi/lo copies: hi differences are exact) added to the bound since the last build
                const SysBox &b = w.box[S == 1 ? 0 : w.psys[i]];
                float g0, g1, g2, l0, l1, l2;
                grid_split(x0, b.lo[0], b, g0, l0);
                grid_split(x1, b.lo[1], b, g1, l1);
                grid_split(x2, b.lo[2], b, g2, l2);
                const float4 oh = w.phi[i], ol = w.plo[i];
                const float d0 = (g0 - oh.x) + (l0 - ol.x), d1 = (g1 - oh.y) + (l1 - ol.y), d2 = (g2 - oh.z) + (l2 - ol.z);
                w.phi[i] = make_float4(g0, g1, g2, oh.w);
                w.plo[i] = make_float4(l0, l1, l2, 0.0f);
                // rounded up by a few units in the last place: a bound, not an estimate
                const float moved = w.disp[i] + sqrtf(d0 * d0 + d1 * d1 + d2 * d2) * 1.000001f + 1e-30f;
                w.disp[i] = moved;
                tripped = tripped || moved > P.half_skinf;
            }
        }
    }
    if (BOX) {
        bounds.reduce_block(box, 0);
        finish_boxes(box);
    } else if (ks.resplit) {
        // The sequence resumes after this drift, which therefore has to be whole: a block that started after the
        // status was set would return at the top and lose its particles' kicks and drift. So the blocks only note
        // that a particle went too far, and the last one to get here (a ticket, no waiting) records it.
        const bool any = __syncthreads_or(tripped);
        if (threadIdx.x == 0) {
            if (any) atomicExch(box.trip, 1u);
            __threadfence();   // this block's note is visible before its ticket
            if (atomicAdd(box.ticket, 1u) == gridDim.x - 1) {
                __threadfence();
                if (atomicExch(box.trip, 0u)) fail(st, ST_SKIN, ks.where);
                *box.ticket = 0u;
            }
        }
    }
}

// caller-array kick and drift (hybrid_kick / hybrid_drift)
template <typename A>
__global__ void __launch_bounds__(256) k_kick_ext(int64_t n, double *vx, double *vy, double *vz, const A *ax,
                                                  const A *ay, const A *az, double h)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        vx[i] = __dadd_rn(vx[i], __dmul_rn(h, widen(ax[i])));
        vy[i] = __dadd_rn(vy[i], __dmul_rn(h, widen(ay[i])));
        vz[i] = __dadd_rn(vz[i], __dmul_rn(h, widen(az[i])));
    }
}

__global__ void __launch_bounds__(256) k_drift_ext(int64_t n, double *x, double *y, double *z, const double *vx,
                                                   const double *vy, const double *vz, double dt)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        x[i] = __dadd_rn(x[i], __dmul_rn(dt, vx[i]));
        y[i] = __dadd_rn(y[i], __dmul_rn(dt, vy[i]));
        z[i] = __dadd_rn(z[i], __dmul_rn(dt, vz[i]));
    }
}

// Softened energies of the (single) system in the working state; see energy_pairs.cuh.
__global__ void __launch_bounds__(EN_ROW) k_energy(EnergyArgs a, double *part)
{
    energy_block(a, part + 2 * (int64_t)blockIdx.x);
}

__global__ void __launch_bounds__(EN_ROW) k_energy_sum(int nb, const double *part, double *out)
{
    energy_total(nb, part, out);
}

StatePtrs state_ptrs(hybrid_ctx *c)
{
    StatePtrs w;
    for (int f = 0; f < 7; ++f) w.x[f] = (double *)c->x[f].p;
    w.id = (int32_t *)c->id.p;
    w.orig = (int32_t *)c->orig.p;
    w.psys = (int32_t *)c->psys.p;
    for (int d = 0; d < 3; ++d) {
        w.as[d] = c->acc_s[d].p;
        w.ah[d] = c->acc_h[d].p;
    }
    w.phi = (float4 *)c->phi.p;
    w.plo = (float4 *)c->plo.p;
    w.disp = (float *)c->disp.p;
    w.box = (const SysBox *)c->box.p;
    return w;
}

}  // namespace

static int grid_n(hybrid_ctx *c, int64_t n)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)c->nsm * 8));
}

void launch_copy_in(hybrid_ctx *c, const SysIO *d_io, bool with_acc)
{
    k_copy_in<<<grid_n(c, c->N), 256, 0, c->st>>>(c->N, c->S, (const int64_t *)c->off_dev.p, d_io, state_ptrs(c),
                                                   c->p.precision, with_acc ? 1 : 0,
                                                   (unsigned long long *)c->boxmin.p, (unsigned long long *)c->boxmax.p,
                                                   (uint32_t *)c->ss_flag.p);
    c->launches++;
}

void launch_copy_out(hybrid_ctx *c, const SysIO *d_io, bool state, bool acc_s, bool acc_h)
{
    k_copy_out<<<grid_n(c, c->N), 256, 0, c->st>>>(c->N, (const int32_t *)c->psys.p, d_io, state_ptrs(c),
                                                    c->p.precision, state, acc_s, acc_h, status_dev(c));
    c->launches++;
}

void launch_kick_seq(hybrid_ctx *c, int n, const int *which, const int *mode, const double *val, int dmode,
                     double dval, bool resplit, bool box)
{
    KickSpec ks;
    ks.resplit = resplit && dmode >= 0 && c->p.precision == 1 && c->p.skin > 0.0;
    ks.where = c->op;
    ks.n = n;
    for (int k = 0; k < 4; ++k) {
        ks.which[k] = k < n ? which[k] : 0;
        ks.mode[k] = k < n ? mode[k] : 0;
        ks.val[k] = k < n ? val[k] : 0.0;
    }
    ks.dmode = dmode;
    ks.dval = dval;
    const int64_t N = c->N;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((N + 255) / 256, (int64_t)c->nsm * 8));
    cudaEvent_t e0 = nullptr;
    prof_begin(c, PROF_INTEG, &e0);
    const StatePtrs w = state_ptrs(c);
    const SysParams *sp = (const SysParams *)c->sp_dev.p;
    const BoxArgs ba = box_args(c);
    const bool with_box = box && c->S == 1 && dmode >= 0;
    if (c->p.precision == 1) {
        if (with_box) k_kick_drift<float, true><<<grid, 256, 0, c->st>>>(N, w, sp, ks, c->S, status_dev(c), ba);
        else k_kick_drift<float, false><<<grid, 256, 0, c->st>>>(N, w, sp, ks, c->S, status_dev(c), ba);
    } else {
        if (with_box) k_kick_drift<double, true><<<grid, 256, 0, c->st>>>(N, w, sp, ks, c->S, status_dev(c), ba);
        else k_kick_drift<double, false><<<grid, 256, 0, c->st>>>(N, w, sp, ks, c->S, status_dev(c), ba);
    }
    c->box_done = with_box;
    prof_end(c, PROF_INTEG, e0);
    c->launches++;
}

void launch_kick_ext(hybrid_ctx *c, const hybrid_system *s, int which, double h)
{
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((s->n + 255) / 256, (int64_t)c->nsm * 8));
    void *ax = which ? s->ax_h : s->ax_s, *ay = which ? s->ay_h : s->ay_s, *az = which ? s->az_h : s->az_s;
    if (c->p.precision == 1)
        k_kick_ext<float><<<grid, 256, 0, c->st>>>(s->n, s->vx, s->vy, s->vz, (const float *)ax, (const float *)ay,
                                                    (const float *)az, h);
    else
        k_kick_ext<double><<<grid, 256, 0, c->st>>>(s->n, s->vx, s->vy, s->vz, (const double *)ax,
                                                     (const double *)ay, (const double *)az, h);
    c->launches++;
}

void launch_drift_ext(hybrid_ctx *c, const hybrid_system *s, double dt)
{
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((s->n + 255) / 256, (int64_t)c->nsm * 8));
    k_drift_ext<<<grid, 256, 0, c->st>>>(s->n, s->x, s->y, s->z, s->vx, s->vy, s->vz, dt);
    c->launches++;
}

size_t energy_scratch_bytes(int nsm) { return ((size_t)2 * EN_BLOCKS_PER_SM * nsm + 2) * sizeof(double); }

void launch_energy(hybrid_ctx *c, double *d_out)
{
    const int grid = (int)std::min<int64_t>(energy_items(c->N), (int64_t)c->nsm * EN_BLOCKS_PER_SM);
    EnergyArgs a;
    a.n = c->N;
    const double **xs[7] = {&a.x, &a.y, &a.z, &a.vx, &a.vy, &a.vz, &a.m};
    for (int f = 0; f < 7; ++f) *xs[f] = (const double *)c->x[f].p;
    a.G = c->h_sp[0].G;
    a.eps2 = c->h_sp[0].eps2;
    double *part = d_out + 2;
    k_energy<<<grid, EN_ROW, 0, c->st>>>(a, part);
    k_energy_sum<<<1, EN_ROW, 0, c->st>>>(grid, part, d_out);
    c->launches += 2;
}

}  // namespace hy
