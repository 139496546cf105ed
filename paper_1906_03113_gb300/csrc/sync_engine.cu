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
#include <algorithm>
#include <atomic>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "sync_multi.cuh"
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

// A batch: this CTA's part of the teams it belongs to, then searches of one CTA.
template <bool SIG>
__global__ void __launch_bounds__(kSyncThreads, 1) sync_batch_kernel(const __grid_constant__ SyncBatch B) {
    __shared__ SyncSmem sm;
    __shared__ SyncSearch S;
    __shared__ uint32_t taken;
    uint32_t at = B.off[blockIdx.x];
    const uint32_t end = B.off[blockIdx.x + 1];
    for (;;) {
        Team T;
        uint32_t q;
        if (at < end) {
            const SyncStep st = B.steps[at++];
            q = st.search;
            T.rank = st.rank;
            T.size = st.size;
        } else {
            if (threadIdx.x == 0) taken = atomicAdd(&B.next[0], 1u);
            __syncthreads();
            if (taken >= B.nqueue) break;
            q = B.queue[taken];
            T.rank = 0;
            T.size = 1;
        }
        T.expect = min(T.size + B.hold_units, 255u);
        __syncthreads();  // (the previous search's descriptor and counters are read no more)
        const uint32_t* src = reinterpret_cast<const uint32_t*>(B.searches + q);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&S);
        for (uint32_t w = threadIdx.x; w < sizeof(SyncSearch) / 4; w += kSyncThreads) dst[w] = src[w];
        __syncthreads();
        if (!SIG && S.ms) ms_search(sm, S, T);
        else sync_search<SIG>(sm, S, T);
        __syncthreads();
    }
    // the last CTA to leave resets the queue for the next launch
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicInc(&B.next[1], gridDim.x - 1) == gridDim.x - 1) B.next[0] = 0;
    }
}

static_assert(sizeof(SyncSmem) <= 31 * 1024, "two lists under the 32 KB shared-memory split");

namespace {

// Shared-memory split and co-resident CTAs of the kernels on a device, looked
// up once per device.
constexpr int kMaxDevices = 64;
std::atomic<int> g_ctas[kMaxDevices];

template <class Kernel>
cudaError_t prepare(Kernel kernel, int sms, int* ctas) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 14);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kSyncThreads, 0);
    *ctas = std::min(*ctas, per_sm * sms);
    return e;
}

}  // namespace

// The largest team, 0 when the kernels do not fit the device.
int sync_max_ctas(int device, int sms) {
    const bool slot = device >= 0 && device < kMaxDevices;
    if (slot) {
        const int have = g_ctas[device].load(std::memory_order_acquire);
        if (have) return have < 0 ? 0 : have;
    }
    // arrivals are counted in 8 bits
    int c = std::min(sms, 240);
    if (prepare(sync_kernel<false>, sms, &c) != cudaSuccess || prepare(sync_kernel<true>, sms, &c) != cudaSuccess ||
        prepare(sync_batch_kernel<false>, sms, &c) != cudaSuccess ||
        prepare(sync_batch_kernel<true>, sms, &c) != cudaSuccess) {
        cudaGetLastError();
        c = 0;
    }
    if (slot) g_ctas[device].store(c ? c : -1, std::memory_order_release);
    return c;
}

// Launch configuration: `ctas` CTAs that are resident together.
static cudaLaunchConfig_t sync_config(int ctas, cudaStream_t s, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kSyncThreads);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = ctas > 1 ? 1 : 0;
    return cfg;
}

cudaError_t launch_sync(const SyncSearch& S, int ctas, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = sync_config(ctas, s, at);
    cudaError_t e = S.sigma ? cudaLaunchKernelEx(&cfg, sync_kernel<true>, S)
                            : cudaLaunchKernelEx(&cfg, sync_kernel<false>, S);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_sync_batch(const SyncBatch& B, bool sigma, int ctas, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = sync_config(ctas, s, at);
    cudaError_t e = sigma ? cudaLaunchKernelEx(&cfg, sync_batch_kernel<true>, B)
                          : cudaLaunchKernelEx(&cfg, sync_batch_kernel<false>, B);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace abfs
