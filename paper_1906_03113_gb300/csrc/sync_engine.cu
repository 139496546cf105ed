// Level-synchronous BFS engine for sm_103a: one search on a team of CTAs that
// are resident together.
//
// The unit scheduler (engine.cu) lets any CTA take work of any search, which
// batches and serving need, and pays for it with a hand-off of 10-20 us
// between levels (publish, poll, take, block lists, unit starts, flush,
// count down).  A single search needs none of that: its levels are separated
// by one barrier whose word also carries the next level's size, so a level
// costs its dependent chain -- row index, claim, barrier -- and nothing else.
//
// Three kinds of level, chosen from the totals the barrier delivers (see
// sync_levels.cuh): thin (claims on the key words, private lists in shared
// memory), wide (bitmap test, reductions, extraction), and the hybrid's
// bottom-up levels.
#include <atomic>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "sync_search.cuh"
#include "internal.h"

namespace abfs {

template <bool SIG>
__global__ void __launch_bounds__(kSyncThreads, 1) sync_kernel(const __grid_constant__ SyncSearch S) {
    __shared__ SyncSmem sm;
    Team T;
    T.rank = blockIdx.x;
    T.size = gridDim.x;
    T.expect = min(gridDim.x + S.hold_units, 255u);
    sync_search<SIG>(sm, S, T);
}

static_assert(sizeof(SyncSmem) <= 31 * 1024, "two lists under the 32 KB shared-memory split");

namespace {

// Shared-memory split and co-resident CTAs of the kernels on a device, looked
// up once per device.
constexpr int kMaxDevices = 64;
std::atomic<int> g_ctas[kMaxDevices];

template <bool SIG>
cudaError_t prepare(int sms, int* ctas) {
    cudaError_t e = cudaFuncSetAttribute(sync_kernel<SIG>, cudaFuncAttributePreferredSharedMemoryCarveout, 14);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sync_kernel<SIG>, kSyncThreads, 0);
    *ctas = per_sm * sms;
    return e;
}

}  // namespace

// The largest team, 0 when the kernel does not fit the device.  Arrivals are
// counted in 8 bits.
int sync_max_ctas(int device, int sms) {
    const bool slot = device >= 0 && device < kMaxDevices;
    if (slot) {
        const int have = g_ctas[device].load(std::memory_order_acquire);
        if (have) return have < 0 ? 0 : have;
    }
    int a = 0, b = 0;
    if (prepare<false>(sms, &a) != cudaSuccess || prepare<true>(sms, &b) != cudaSuccess) {
        cudaGetLastError();
        a = b = 0;
    }
    int c = a < b ? a : b;
    if (c > sms) c = sms;
    if (c > 240) c = 240;
    if (slot) g_ctas[device].store(c ? c : -1, std::memory_order_release);
    return c;
}

cudaError_t launch_sync(const SyncSearch& S, int ctas, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kSyncThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = ctas > 1 ? 1 : 0;
    cudaError_t e = S.sigma ? cudaLaunchKernelEx(&cfg, sync_kernel<true>, S)
                            : cudaLaunchKernelEx(&cfg, sync_kernel<false>, S);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace abfs
