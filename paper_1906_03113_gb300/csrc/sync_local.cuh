// Level-synchronous engine: searches of small graphs, whole in one CTA.
// Part of sync_engine.cu, split by topic; included in order.
#pragma once

#include "sync_levels.cuh"

namespace abfs {

// On a graph of a few thousand vertices a search is nothing but latency: the
// general engine waits in every level for a row index, a 64-bit claim at the L2
// and a column, each about 0.4 us.  Here the keys are 32-bit words in shared
// memory (level << kLocalShift | parent, the order of the 64-bit keys), the
// frontiers are stretches of one queue of vertices, and the graph is brought
// into the L1 by one pass of independent loads before the first level, so that
// no level waits for the L2: ER of 1000 vertices, degree 8, 31.7 -> 18.0 us, most
// of the rest the launch.
constexpr uint32_t kLocalShift = 12;
static_assert(kLocalN == 1u << kLocalShift, "a parent fits below the level");

struct LocalSmem {
    uint32_t key[kLocalN];
    uint16_t queue[kLocalN];  // every vertex enters once; a level is a stretch
};
static_assert(sizeof(LocalSmem) <= sizeof(SyncSmem::ij) + sizeof(SyncSmem::ib) + sizeof(SyncSmem::il) &&
                  offsetof(SyncSmem, ij) == 0 && offsetof(SyncSmem, app) == sizeof(SyncSmem::ij) * 3,
              "in the place of the thin levels' lists");

__device__ __forceinline__ void touch(const uint32_t* p) {
    asm volatile("{\n\t.reg .u32 x;\n\tld.global.nc.u32 x, [%0];\n\t}" ::"l"(p));
}

// Runs one search on this CTA.  Whole CTA; the outputs and the control block
// are written when it returns.
__device__ __noinline__ void local_search(SyncSmem& sm, const SyncSearch& S) {
    LocalSmem& L = *reinterpret_cast<LocalSmem*>(&sm);
    uint32_t* const cnt = sm.wsum;  // vertices appended by level k: cnt[k % 3]
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // one word of every 32-byte sector
    for (uint32_t i = 8 * tid; i <= S.n; i += 8 * kSyncThreads) {
        touch(S.colptr + i);
    }
    for (uint32_t i = 8 * tid; i < S.nnz; i += 8 * kSyncThreads) {
        touch(S.rowidx + i);
    }
    for (uint32_t v = tid; v < S.n; v += kSyncThreads) L.key[v] = v == S.src ? v : kUnset;
    if (tid < 3) cnt[tid] = 0;
    if (tid == 0) {
        L.queue[0] = (uint16_t)S.src;
        sm.st_read = sm.st_unmasked = 0;
    }
    __syncthreads();
    uint32_t a = 0, b = 1, k = 0, read = 0, unmasked = 0;
    while (a < b) {
        // (read by nobody since the last level's barrier)
        if (tid == 0) cnt[(k + 1) % 3] = 0;
        const uint32_t c = b - a;
        // batches of 32 vertices, their number rounded up to a power of two; the
        // warps of a batch take its groups of 32 entries in turn
        const uint32_t lb = c > 32 ? min(32 - __clz((c - 1) / 32), 5) : 0;
        const uint32_t step = (32 * kSyncWarps) >> lb;
        for (uint32_t i0 = 32 * (warp & ((1u << lb) - 1u)); i0 < c; i0 += 32 * kSyncWarps) {
            uint32_t j = 0, beg = 0, len = 0;
            if (i0 + lane < c) {
                j = L.queue[a + i0 + lane];
                beg = ld_ro(S.colptr + j);
                len = ld_ro(S.colptr + j + 1) - beg;
            }
            const uint32_t incl = warp_incl_scan(len);
            const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
            const uint32_t shift = beg - (incl - len);
            for (uint32_t g = 32 * (warp >> lb); g < total; g += step) {
                // the vertex of entry g + lane: the first whose inclusive count exceeds it
                uint32_t own = 0;
#pragma unroll
                for (uint32_t d = 16; d > 0; d >>= 1)
                    if (g + lane >= __shfl_sync(0xFFFFFFFFu, incl, own + d - 1)) own += d;
                const uint32_t pos = __shfl_sync(0xFFFFFFFFu, shift, own) + g + lane;
                const uint32_t jj = __shfl_sync(0xFFFFFFFFu, j, own);
                bool win = false;
                uint32_t r = 0;
                if (g + lane < total) {
                    r = ld_ro(S.rowidx + pos);
                    const uint32_t old = atomicMin(&L.key[r], (k + 1) << kLocalShift | jj);
                    ++read;
                    unmasked += (old >> kLocalShift) > k;
                    win = old == kUnset;
                }
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, win);
                if (m) {
                    uint32_t at = 0;
                    if (lane == 0) at = atomicAdd(&cnt[k % 3], __popc(m));
                    at = __shfl_sync(0xFFFFFFFFu, at, 0);
                    if (win) L.queue[b + at + __popc(m & lanemask_lt())] = (uint16_t)r;
                }
            }
        }
        __syncthreads();
        a = b;
        b += cnt[k % 3];
        ++k;
    }
    tally_add(sm, read, unmasked);
    for (uint32_t v = tid; v < S.n; v += kSyncThreads) {
        const uint32_t x = L.key[v];
        S.level[v] = x == kUnset ? -1 : (int32_t)(x >> kLocalShift);
        S.parent[v] = x == kUnset ? kUnset : x & (kLocalN - 1u);
    }
    uint32_t* const c = reinterpret_cast<uint32_t*>(S.ctl);
    for (uint32_t w = tid; w < sizeof(InstCtl) / 4; w += kSyncThreads) c[w] = 0u;
    __syncthreads();
    if (tid == 0) {
        // every reached column was read whole, once
        S.ctl->entries_read = S.ctl->nnz_reached = sm.st_read;
        S.ctl->entries_unmasked = S.ctl->claims = sm.st_unmasked;
        S.ctl->reached = b;
        S.ctl->levels = k;
    }
}

}  // namespace abfs
