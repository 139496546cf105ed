// Level-synchronous engine: multi-source searches (batches).
// Part of sync_engine.cu, split by topic; included in order.
//
// Up to 64 sources of one undirected graph with ascending columns search
// together, one bit each of a 64-bit mask per vertex (Theorem 1 applied to X_k
// with one column per source).  At level k the bits of vertex i's next frontier
// are those of its column's frontier masks that i lacks, and the parent for
// each bit is the first column entry that holds it (the least index, since the
// column ascends).  One scan of a column finds bits and parents together, so a
// level is evaluated in one of two ways:
//   pulled: every vertex that some source has not reached scans its column for
//     any missing bit;
//   pushed, while the frontier's columns are a small part of what a pull would
//     read: the frontier's columns are expanded into next-bit masks first, and
//     only vertices with new bits scan their columns, for exactly those bits.
// (Pushing every level read each column once per level it is in the union
// frontier and added a 64-bit reduction per entry: 64 sources on R-MAT-22
// 17.5 ms.)
#pragma once

#include "sync_search.cuh"

namespace abfs {

// A pull reads the open entries (of vertices some source has not reached), most
// of them; a push reads the frontier's entries, with a mask load and often a
// reduction each, and scans besides.
constexpr uint32_t kMsPushShare = 8;
// Columns longer than this are scanned by a whole CTA, 4096 entries a round.
constexpr uint32_t kMsLong = 2048;
constexpr uint32_t kMsIlp = 4;

__device__ __forceinline__ void ms_parents(const SyncSearch& S, uint32_t v, uint32_t j,
                                           unsigned long long bits) {
    while (bits) {
        const uint32_t s = (uint32_t)(__ffsll((long long)bits) - 1);
        bits &= bits - 1;
        S.ms_parent[s][v] = (int32_t)j;
    }
}
__device__ __forceinline__ unsigned long long warp_or64(unsigned long long x) {
    return (unsigned long long)__reduce_or_sync(0xFFFFFFFFu, (uint32_t)(x >> 32)) << 32 |
           __reduce_or_sync(0xFFFFFFFFu, (uint32_t)x);
}
// The bits of x that no lower lane holds.
__device__ __forceinline__ unsigned long long warp_first64(unsigned long long x) {
    const uint32_t lane = threadIdx.x & 31;
    unsigned long long incl = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl |= y;
    }
    const unsigned long long below = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
    return lane ? x & ~below : x;
}

// The hits of 32 * kMsIlp consecutive entries from x on (entry x + 32 u + lane in
// h[u], column index j[u]): frontier masks limited to `rem`.
__device__ __forceinline__ void ms_load(const SyncSearch& S, const unsigned long long* fr, uint32_t x,
                                        uint32_t end, unsigned long long rem, uint32_t (&j)[kMsIlp],
                                        unsigned long long (&h)[kMsIlp]) {
    const uint32_t lane = threadIdx.x & 31;
#pragma unroll
    for (uint32_t u = 0; u < kMsIlp; ++u) {
        const uint32_t at = x + 32 * u + lane;
        j[u] = at < end ? ld_ro(S.rowidx + at) : kUnset;
    }
#pragma unroll
    for (uint32_t u = 0; u < kMsIlp; ++u) h[u] = j[u] != kUnset ? (ld_l2(fr + j[u]) & rem) : 0ull;
}
// Writes the parents of vertex v for the bits among `rem` that these entries
// hold first; returns the bits left.  Whole warp.
__device__ __forceinline__ unsigned long long ms_take(const SyncSearch& S, uint32_t v, unsigned long long rem,
                                                      const uint32_t (&j)[kMsIlp],
                                                      const unsigned long long (&h)[kMsIlp]) {
#pragma unroll
    for (uint32_t u = 0; u < kMsIlp; ++u) {
        const unsigned long long x = h[u] & rem;
        const unsigned long long any = warp_or64(x);
        if (!any) continue;
        ms_parents(S, v, j[u], warp_first64(x));
        rem &= ~any;
    }
    return rem;
}

// New bits of every vertex at level k: masks, levels, parents, the frontier
// masks of level k + 1.  pushed: the candidates are in ms_nx.  Whole team; the
// CTAs take words in turn.
__device__ __noinline__ void ms_scan(SyncSmem& sm, const SyncSearch& S, const Team& T, uint32_t k, bool pushed) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t p = k & 1, pn = p ^ 1;
    const unsigned long long* const fr = S.ms_fr[p];
    const unsigned long long all = S.ms == 64 ? ~0ull : (1ull << S.ms) - 1;
    uint32_t verts = 0, entries = 0;
    unsigned long long open = 0;
    for (;;) {
        uint32_t x = 0;
        if (lane == 0) {
            x = atomicAdd(&sm.tick, 1u);
            sync_beat(S, x, 32);
        }
        x = __shfl_sync(0xFFFFFFFFu, x, 0);
        const unsigned long long w = (unsigned long long)x * T.size + T.rank;
        if (w >= S.nwords) break;
        const uint32_t v = (uint32_t)w * 32 + lane;
        const bool have = v < S.n;
        unsigned long long want = 0, vis = 0;
        uint32_t cb = 0, end = 0;
        if (have) {
            if (pushed) {
                want = ld_l2(S.ms_nx + v);
                if (want) {
                    S.ms_nx[v] = 0ull;
                    vis = ld_l2(S.ms_vis + v);
                }
            } else {
                vis = ld_l2(S.ms_vis + v);
                want = all & ~vis;
            }
            if (want) {
                cb = ld_ro(S.colptr + v);
                end = ld_ro(S.colptr + v + 1);
            }
        }
        // long columns wait for the whole CTA
        bool later = false;
        if (end - cb > kMsLong) {
            const uint32_t at = atomicAdd(&sm.nlong, 1u);
            if (at < kThinCap) {
                sm.ij[0][at] = v;
                sm.ib[0][at] = (uint32_t)want;
                sm.il[0][at] = (uint32_t)(want >> 32);
                later = true;
            }
        }
        unsigned long long rem = later ? 0ull : want;
        // the first 16 entries: a lane each
        uint32_t e = cb;
        for (uint32_t b = 0; b < 4 && rem && e < end; ++b) {
            uint32_t jj[4];
            unsigned long long fm[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) jj[q] = e + q < end ? ld_ro(S.rowidx + e + q) : kUnset;
#pragma unroll
            for (int q = 0; q < 4; ++q) fm[q] = jj[q] != kUnset ? ld_l2(fr + jj[q]) : 0ull;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned long long hit = fm[q] & rem;
                if (hit) {
                    ms_parents(S, v, jj[q], hit);
                    rem &= ~hit;
                }
            }
            e += 4;
        }
        // the rest: the warp together, column by column
        uint32_t dm = __ballot_sync(0xFFFFFFFFu, rem != 0ull && e < end);
        while (dm) {
            const uint32_t o = __ffs(dm) - 1;
            dm &= dm - 1;
            const uint32_t ov = __shfl_sync(0xFFFFFFFFu, v, o), oe = __shfl_sync(0xFFFFFFFFu, end, o);
            unsigned long long orem = __shfl_sync(0xFFFFFFFFu, rem, o);
            for (uint32_t y = __shfl_sync(0xFFFFFFFFu, e, o); y < oe && orem; y += 32 * kMsIlp) {
                uint32_t j[kMsIlp];
                unsigned long long h[kMsIlp];
                ms_load(S, fr, y, oe, orem, j, h);
                orem = ms_take(S, ov, orem, j, h);
            }
            if (lane == o) rem = orem;
        }
        if (have && !later) {
            const unsigned long long got = want & ~rem;
            S.ms_fr[pn][v] = got;
            if (got) {
                S.ms_vis[v] = vis | got;
                ++verts;
                entries += end - cb;
            }
            if (rem) open += end - cb;
            want = got;
        } else {
            want = 0ull;
        }
        // levels source by source: the lanes that hold a bit write consecutive
        // vertices of that source's array
        unsigned long long un = warp_or64(want);
        while (un) {
            const uint32_t s = (uint32_t)(__ffsll((long long)un) - 1);
            un &= un - 1;
            if ((want >> s) & 1ull) S.ms_level[s][v] = (int32_t)(k + 1);
        }
    }
    __syncthreads();
    const uint32_t longs = min(sm.nlong, kThinCap);
    uint32_t round = 0;
    for (uint32_t i = 0; i < longs; ++i) {
        if (threadIdx.x == 0) sync_beat(S, 0, 1);
        const uint32_t v = sm.ij[0][i];
        const unsigned long long want = (unsigned long long)sm.il[0][i] << 32 | sm.ib[0][i];
        const uint32_t cb = ld_ro(S.colptr + v), end = ld_ro(S.colptr + v + 1);
        unsigned long long rem = want;
        for (uint32_t y = cb; y < end && rem; y += 32 * kMsIlp * kSyncWarps, ++round) {
            uint32_t j[kMsIlp];
            unsigned long long h[kMsIlp];
            ms_load(S, fr, y + 32 * kMsIlp * warp, end, rem, j, h);
            const unsigned long long mine = warp_or64(h[0] | h[1] | h[2] | h[3]);
            unsigned long long* const wm = sm.wm[round & 1];
            if (lane == 0) wm[warp] = mine;
            __syncthreads();
            const unsigned long long x = wm[lane];
            const unsigned long long below = warp_or64(lane < warp ? x : 0ull);
            if (mine & ~below) ms_take(S, v, rem & ~below, j, h);
            rem &= ~warp_or64(x);
        }
        const unsigned long long got = want & ~rem;
        if (threadIdx.x < S.ms && ((got >> threadIdx.x) & 1ull))
            S.ms_level[threadIdx.x][v] = (int32_t)(k + 1);
        if (threadIdx.x == 0) {
            S.ms_fr[pn][v] = got;
            if (got) {
                S.ms_vis[v] = ld_l2(S.ms_vis + v) | got;
                ++verts;
                entries += end - cb;
            }
            if (rem) open += end - cb;
        }
    }
    verts = __reduce_add_sync(0xFFFFFFFFu, verts);
    entries = __reduce_add_sync(0xFFFFFFFFu, entries);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) open += __shfl_xor_sync(0xFFFFFFFFu, open, d);
    if (lane == 0) {
        if (verts) {
            atomicAdd(&sm.verts, verts);
            atomicAdd(&sm.ent, entries);
        }
        if (open) atomicAdd(&sm.open, open);
    }
    __syncthreads();
}

// Runs one multi-source search on this team.
__device__ __forceinline__ void ms_search(SyncSmem& sm, const SyncSearch& S, const Team& T) {
    const bool lead = threadIdx.x == 0;
    const uint32_t stride = T.size * kSyncThreads, t0 = T.rank * kSyncThreads + threadIdx.x;
    const bool slow = sync_long_pass(S, T);
    for (uint32_t v = t0; v < S.n; v += stride) {
        if (slow) red_add64(&S.bar->beat, 1ull);
        S.ms_vis[v] = 0ull;
        S.ms_fr[0][v] = 0ull;
        S.ms_nx[v] = 0ull;
    }
    if (T.rank == 0) {
        uint32_t* c = reinterpret_cast<uint32_t*>(S.ctl);
        for (uint32_t w = threadIdx.x; w < sizeof(InstCtl) / 4; w += kSyncThreads) c[w] = 0u;
    }
    if (lead) {
        sm.step = sm.tick = sm.nlong = 0;
        sm.word[0] = sm.word[1] = sm.aux[0] = sm.aux[1] = 0;
        sm.app[0][0] = sm.verts = sm.ent = 0;
        sm.open = 0;
    }
    bool ok = team_sync(sm, S, T);
    if (ok && T.rank == 0 && threadIdx.x < S.ms) {
        const uint32_t v = S.ms_src[threadIdx.x];
        atomicOr(S.ms_vis + v, 1ull << threadIdx.x);
        atomicOr(S.ms_fr[0] + v, 1ull << threadIdx.x);
        S.ms_level[threadIdx.x][v] = 0;
        S.ms_parent[threadIdx.x][v] = (int32_t)v;
    }
    ok = ok && team_sync(sm, S, T);
    // the sources' columns as the first list (the frontier of "level k + 1" for
    // the pass, so k is -1)
    unsigned long long open = S.nnz, ent = 0;
    uint32_t k = 0, reached = 0;
    bool list = false;  // the frontier's list is there
    bool more = ok;
    if (ok) {
        sync_extract<kFromMasks>(sm, S, T, ~0u);
        __syncthreads();
        const uint32_t c = sm.app[0][0], v = sm.verts;
        ok = team_sync(sm, S, T, c, (unsigned long long)v << kAuxShift | sm.ent);
        reached = (uint32_t)(sm.entries >> kAuxShift);
        ent = sm.entries & ((1ull << kAuxShift) - 1);
        list = true;
        more = ok && sm.items != 0;
        __syncthreads();
        if (lead) sm.app[0][0] = sm.verts = sm.ent = 0;
        __syncthreads();
    }
    while (more) {
        const bool push = ent * kMsPushShare < open;
        if (push && !list) {
            sync_extract<kFromMasks>(sm, S, T, k - 1);
            __syncthreads();
            const uint32_t c = sm.app[0][0];
            ok = team_sync(sm, S, T, c, sm.ent);
            __syncthreads();
            if (lead) sm.app[0][0] = sm.verts = sm.ent = 0;
            __syncthreads();
            if (!ok) break;
        }
        if (push) {
            const unsigned long long items = sm.items;
            if (T.rank == 0 && lead) st_relaxed(&S.bar->lcnt[k & 1], 0u);
            if (lead) sm.entries = ent;
            __syncthreads();
            wide_expand<kWideMulti, false>(sm, S, T, k, items);
            ok = team_sync(sm, S, T);
            if (!ok) break;
            if (lead) sm.tick = 0;
            __syncthreads();
        } else if (list && T.rank == 0 && lead) {
            st_relaxed(&S.bar->lcnt[k & 1], 0u);  // a list that nobody read
        }
        list = false;
        ms_scan(sm, S, T, k, push);
        const uint32_t v = sm.verts, e = sm.ent;
        const unsigned long long o = sm.open;
        ok = team_sync(sm, S, T, o, (unsigned long long)v << kAuxShift | e);
        if (lead) {
            sm.tick = sm.nlong = sm.verts = sm.ent = 0;
            sm.open = 0;
            sm.act = ld_relaxed(&S.bar->err);  // a failed append
        }
        if (!push) open = sm.items;
        const uint32_t nv = (uint32_t)(sm.entries >> kAuxShift);
        ent = sm.entries & ((1ull << kAuxShift) - 1);
        reached += nv;
        __syncthreads();
        ok = ok && sm.act == 0;
        more = ok && nv != 0;
        ++k;
    }
    if (ok) {
        // what was not reached reads -1 (everything else has been written)
        const unsigned long long all = S.ms == 64 ? ~0ull : (1ull << S.ms) - 1;
        const uint32_t lane = threadIdx.x & 31, W = T.size * kSyncWarps;
        for (uint32_t w = T.rank * kSyncWarps + (threadIdx.x >> 5); w < S.nwords; w += W) {
            if (slow) red_add64(&S.bar->beat, 1ull);
            const uint32_t v = w * 32 + lane;
            const unsigned long long lack = v < S.n ? all & ~ld_l2(S.ms_vis + v) : 0ull;
            unsigned long long un = warp_or64(lack);
            while (un) {
                const uint32_t s = (uint32_t)(__ffsll((long long)un) - 1);
                un &= un - 1;
                if ((lack >> s) & 1ull) {
                    S.ms_level[s][v] = -1;
                    S.ms_parent[s][v] = -1;
                }
            }
        }
    }
    __syncthreads();
    if (lead) {
        if (T.rank == 0) {
            st_relaxed(&S.ctl->levels, k);
            st_relaxed(&S.ctl->reached, reached);
        }
        sync_leave(S, T);
    }
}

}  // namespace abfs
