// Allocation-free energy diagnostic: the softened kinetic and potential
// energies of one system by direct FP64 summation (the total-energy check of
// Sec. IV-A), like hybrid_energy, but with no context and no device
// allocation of any kind.
//
// Who needs it: callers that cannot call cudaMalloc/cudaFree (or any library
// call that allocates), namely
//  - code that runs when the device has no free memory left, e.g. a
//    diagnostic taken from an out-of-memory handler, or in a process whose
//    caching allocator already holds the whole device;
//  - latency-sensitive loops that must not pay the implicit device-wide
//    synchronisation cudaFree performs, nor the first-touch cost of a new
//    allocation.
// hybrid_create and hybrid_energy allocate their working buffers, so such
// callers cannot use them.
//
// Scratch is a file-scope __device__ array of fixed size: one (kinetic,
// potential) pair per block plus the two totals. Its address is looked up
// once per device with cudaGetSymbolAddress, with that device current, on the
// first call made there. Every slot a call reads is written earlier in the
// same call (per-block partials, then the totals), so nothing has to start at
// zero. The scratch is shared by every call on the device: calls that overlap
// in time (two streams, two host threads) race on it.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "../../include/hybrid.h"
#include "energy_pairs.cuh"

namespace {

constexpr int64_t ES_SLOTS = 16384;   // block sums: far above EN_BLOCKS_PER_SM blocks on every SM
constexpr int ES_MAX_DEVICES = 64;

// [2 * block] kinetic, [2 * block + 1] potential; the last two slots hold the totals
__device__ __align__(256) double es_scratch[2 * ES_SLOTS + 2];

double *g_scratch[ES_MAX_DEVICES];
std::mutex g_mu;

__global__ void __launch_bounds__(hy::EN_ROW) k_energy_tiles(hy::EnergyArgs a, double *__restrict__ part)
{
    hy::energy_block(a, part + 2 * (int64_t)blockIdx.x);
}

// One block: the block sums in a fixed order; the totals go after the last slot.
__global__ void __launch_bounds__(hy::EN_ROW) k_energy_total(int nb, double *part)
{
    hy::energy_total(nb, part, part + 2 * ES_SLOTS);
}

// Scratch address on the current device, looked up on the first call there.
// The same set-up queries both kernels' attributes, which loads them: under
// lazy module loading a kernel is otherwise loaded (and its code given device
// memory) at its first launch, which an allocation-free caller cannot afford.
cudaError_t scratch_for_current(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= ES_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, es_scratch);
        if (e != cudaSuccess) return e;
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, k_energy_tiles);
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_energy_total);
        if (e != cudaSuccess) return e;
        g_scratch[dev] = (double *)p;
    }
    *out = g_scratch[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" hybrid_status hybrid_energy_noalloc(int64_t n, const double *x, const double *y, const double *z,
                                               const double *vx, const double *vy, const double *vz,
                                               const double *m, double G, double eps, void *stream,
                                               double *kinetic, double *potential)
{
    if (!kinetic || !potential || n < 0 || !(eps >= 0.0)) return HYBRID_EINVAL;
    if (n > HYBRID_ENERGY_NOALLOC_MAX_N) return HYBRID_ETOOLARGE;
    if (n > 0 && (!x || !y || !z || !vx || !vy || !vz || !m)) return HYBRID_EINVAL;
    double *scratch = nullptr;
    if (scratch_for_current(&scratch) != cudaSuccess) return HYBRID_ECUDA;
    if (n == 0) {
        *kinetic = 0.0;
        *potential = 0.0;
        return HYBRID_OK;
    }
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return HYBRID_ECUDA;
    const int64_t most = nsm * hy::EN_BLOCKS_PER_SM < ES_SLOTS ? nsm * hy::EN_BLOCKS_PER_SM : ES_SLOTS;
    const int grid = (int)(hy::energy_items(n) < most ? hy::energy_items(n) : most);
    const hy::EnergyArgs a = {n, x, y, z, vx, vy, vz, m, G, eps * eps};
    k_energy_tiles<<<grid, hy::EN_ROW, 0, st>>>(a, scratch);
    k_energy_total<<<1, hy::EN_ROW, 0, st>>>(grid, scratch);
    double v[2];
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(v, scratch + 2 * ES_SLOTS, sizeof v, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return HYBRID_ECUDA;
    *kinetic = v[0];
    *potential = v[1];
    return HYBRID_OK;
}
