// Level-synchronous BFS engine for sm_103a: one search on a team of CTAs that
// are resident together.
//
// The unit scheduler (engine.cu) lets any CTA take work of any search and pays
// for it with a hand-off of 10-20 us between levels (publish, poll, take, block
// lists, unit starts, flush, count down).  A search on a team of its own needs
// none of that: its levels are separated by one barrier whose word also carries
// the next level's size, so a level costs its dependent chain -- row index,
// claim, barrier -- and nothing else.
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
#include "serve_team.h"

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

// ---------------------------------------------------------------------------
// serving: a long-lived launch over a table of slots
// ---------------------------------------------------------------------------
// A CTA without a search first joins a team that is being formed, else claims a
// newly submitted query.  The query gets a share of the CTAs in proportion to
// its part of the work at hand (all of them when it is alone): the claiming CTA
// opens a team of that size, waits for others to come free, a quarter of the
// time the query then takes and at most kJoinWaitNs, closes the team and runs
// the query with whoever came.  While fewer than half have come it waits on, up
// to half of what the query would take those few: the last CTA to come free, too
// late for the other teams, took a query alone while they were about to finish
// (16 queries on a 64^3 mesh 4.7 -> 1.1 ms, on 100^3 16.8 -> 3.9; the unit
// scheduler 2.1 and 10.8).  Only CTAs that have joined are waited for
// afterwards, so the launch needs no co-residency of all its CTAs, and a CTA
// that idles out is never missed.  Claims are made one at a time, so that CTAs
// that come free together do not each open a team that nobody is left to join.
// (Counting on free CTAs alone left large queries on one CTA whenever the
// launch was busy: 256 queries on 16 graphs 3.6 -> 6.7 ms.)
constexpr unsigned long long kJoinWaitNs = 150000, kJoinWaitMinNs = 5000;
constexpr unsigned long long kFewWaitNs = 100000000ull, kMemberWaitNs = 1000000000ull;

struct ServeCmd {
    uint32_t what;  // 0: nothing to do, 1: run slot q, 2: leave
    uint32_t q, rank, size;
    uint32_t busy;  // some slot holds a query that is submitted or running
};

// The accesses of a slot's word (serve_team.h).
struct JoinIo {
    unsigned long long* word;
    __device__ __forceinline__ unsigned long long load() { return ld_relaxed64(word); }
    __device__ __forceinline__ unsigned long long close() { return atomicAnd(word, ~kJoinOpen); }
    __device__ __forceinline__ unsigned long long now() { return globaltimer(); }
};

// Warp 0: something to do, or nothing.
__device__ __forceinline__ ServeCmd serve_poll(const SyncServe& A, uint32_t cursor) {
    const uint32_t lane = threadIdx.x & 31;
    ServeCmd c = {0, 0, 0, 0, 0};
    unsigned long long work = 0;  // of all queries submitted or running
    uint32_t near = ~0u;          // submitted query nearest after the cursor: its distance
    for (uint32_t b = 0; b < A.nslots; b += 32) {
        const uint32_t q = b + lane;
        unsigned long long w = 0;
        uint32_t st = 0;
        if (q < A.nslots) {
            w = ld_relaxed64(A.join + q);
            st = ld_relaxed(A.state + q);
        }
        uint32_t m = __ballot_sync(0xFFFFFFFFu, join_room(w));
        while (m) {
            const uint32_t l = __ffs(m) - 1;
            m &= m - 1;
            uint32_t rank = 0, size = 0;
            if (lane == l) {
                for (int tries = 0; tries < 8; ++tries) {
                    if (!join_room(w)) break;
                    const unsigned long long seen = atomicCAS(A.join + q, w, w + 1);
                    if (seen == w) {
                        rank = join_count(w);
                        __threadfence();  // acquire: the slot's descriptor
                        JoinIo io{A.join + q};
                        size = team_form(io, false, kMemberWaitNs);
                        break;
                    }
                    w = seen;
                }
            }
            size = __shfl_sync(0xFFFFFFFFu, size, l);
            if (size) {
                c.what = 1;
                c.q = b + l;
                c.rank = __shfl_sync(0xFFFFFFFFu, rank, l);
                c.size = size;
                return c;
            }
        }
        c.busy |= st & 0xFFu;
        if (st & 0xFFu) work += st >> kSlotWorkShift;
        if ((st & 0xFFu) == kSlotSubmitted) near = min(near, q >= cursor ? q - cursor : q + A.nslots - cursor);
    }
    near = __reduce_min_sync(0xFFFFFFFFu, near);
    c.busy = __any_sync(0xFFFFFFFFu, c.busy != 0);
    if (near == ~0u) return c;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) work += __shfl_xor_sync(0xFFFFFFFFu, work, d);
    const uint32_t q = (near + cursor) % A.nslots;
    uint32_t size = 0;
    if (lane == 0) {
        if (atomicCAS(A.claim, 0u, 1u) == 0u) {
            const uint32_t st = ld_relaxed(A.state + q);
            const uint32_t run = (st & ~0xFFu) | kSlotRunning;
            unsigned long long w = 0, wait = 0, few = 0;
            // (a launch that has been closed claims nothing more)
            if ((st & 0xFFu) == kSlotSubmitted && ld_relaxed(A.closed) != A.launch &&
                atomicCAS(A.state + q, st, run) == st) {
                __threadfence();  // acquire: the descriptor the host wrote before the state
                const unsigned long long mine = max(st >> kSlotWorkShift, 1u);
                const unsigned long long part = (mine * gridDim.x + work - 1) / max(work, 1ull);
                size = max(1u, (uint32_t)min(part, (unsigned long long)ld_l2(&A.slots[q].cap)));
                if (size > 1) {
                    // (work is in eighths of a microsecond)
                    wait = min(kJoinWaitNs, max(kJoinWaitMinNs, 125ull * mine / (4 * size)));
                    few = min(kFewWaitNs, 125ull * mine / 2);
                    w = join_opened(ld_relaxed64(A.join + q), size);
                    __threadfence();
                    st_relaxed64(A.join + q, w);
                }
            }
            // (the team is open before the next claim can be made)
            __threadfence();
            st_relaxed(A.claim, 0u);
            if (w) {
                JoinIo io{A.join + q};
                size = team_form(io, true, wait, few);
            }
        }
    }
    size = __shfl_sync(0xFFFFFFFFu, size, 0);
    if (size) {
        c.what = 1;
        c.q = q;
        c.size = size;
    }
    return c;
}

// Warp 0, having found no query for idle_exit_ns: closes the launch unless one
// has come meanwhile.  Under the claimers' lock, so that no query is claimed by a
// launch whose other CTAs are leaving.
__device__ __forceinline__ bool serve_close(const SyncServe& A) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t locked = 0;
    if (lane == 0) locked = atomicCAS(A.claim, 0u, 1u) == 0u;
    if (!__shfl_sync(0xFFFFFFFFu, locked, 0)) return false;
    __threadfence();
    uint32_t busy = 0;
    for (uint32_t q = lane; q < A.nslots; q += 32) busy |= ld_relaxed(A.state + q) & 0xFFu;
    busy = __any_sync(0xFFFFFFFFu, busy != 0);
    if (lane == 0) {
        if (!busy) st_relaxed(A.closed, A.launch);
        __threadfence();
        st_relaxed(A.claim, 0u);
    }
    return !busy;
}

__global__ void __launch_bounds__(kSyncThreads, 1) sync_serve_kernel(const __grid_constant__ SyncServe A) {
    __shared__ SyncSmem sm;
    __shared__ SyncSlot slot;
    __shared__ ServeCmd cmd;
    uint64_t idle_since = 0;
    uint32_t backoff = 64;
    for (;;) {
        if (threadIdx.x < 32) {
            ServeCmd c = {2, 0, 0, 0, 0};
            if (ld_relaxed(A.stop_flag) == 0 && ld_relaxed(A.closed) != A.launch) {
                c = serve_poll(A, blockIdx.x * 7u % A.nslots);
                if (c.what == 0) {
                    // Nothing to do: sleep, or end the launch after idle_exit_ns in
                    // which no slot held a query (the host relaunches on demand).
                    // While one runs, however long, every CTA stays for the next;
                    // and the CTAs leave together, so that a launch that goes on
                    // has the whole GPU.
                    const uint64_t now = globaltimer();
                    if (c.busy || idle_since == 0) idle_since = now;
                    else if (now - idle_since > A.idle_exit_ns && serve_close(A)) c.what = 2;
                    if (c.what == 0) __nanosleep(backoff);
                    if (backoff < 1024) backoff <<= 1;
                } else {
                    backoff = 64;
                    idle_since = 0;
                }
            }
            if (threadIdx.x == 0) cmd = c;
        }
        __syncthreads();
        const ServeCmd c = cmd;
        if (c.what == 2) break;
        if (c.what == 1) {
            // read through L2: the slot held another query before
            const uint32_t* src = reinterpret_cast<const uint32_t*>(A.slots + c.q);
            uint32_t* dst = reinterpret_cast<uint32_t*>(&slot);
            for (uint32_t w = threadIdx.x; w < sizeof(SyncSlot) / 4; w += kSyncThreads) dst[w] = ld_l2(src + w);
            Team T;
            T.rank = c.rank;
            T.size = T.expect = c.size;
            __syncthreads();
            const bool last = sync_search<false>(sm, slot.search, T);
            if (threadIdx.x == 0 && last) {
                // ticket and status reach the host's word after every write of
                // the search (each CTA fenced its own before it left)
                st_relaxed(A.state + c.q, kSlotFree);
                __threadfence_system();
                const unsigned long long word = slot.ticket << 8 | (ld_relaxed(&slot.search.ctl->err) & 0xFFu);
                asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(slot.notify), "l"(word) : "memory");
            }
        }
        __syncthreads();
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
        prepare(sync_batch_kernel<true>, sms, &c) != cudaSuccess || prepare(sync_serve_kernel, sms, &c) != cudaSuccess) {
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
    if (test_refuse_teams()) return cudaErrorCooperativeLaunchTooLarge;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = sync_config(ctas, s, at);
    cudaError_t e = S.sigma ? cudaLaunchKernelEx(&cfg, sync_kernel<true>, S)
                            : cudaLaunchKernelEx(&cfg, sync_kernel<false>, S);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_sync_serve(const SyncServe& A, int ctas, cudaStream_t s) {
    sync_serve_kernel<<<ctas, kSyncThreads, 0, s>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_sync_batch(const SyncBatch& B, bool sigma, int ctas, cudaStream_t s) {
    if (test_refuse_teams()) return cudaErrorCooperativeLaunchTooLarge;
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = sync_config(ctas, s, at);
    cudaError_t e = sigma ? cudaLaunchKernelEx(&cfg, sync_batch_kernel<true>, B)
                          : cudaLaunchKernelEx(&cfg, sync_batch_kernel<false>, B);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace abfs
