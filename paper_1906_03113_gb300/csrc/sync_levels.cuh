// Level-synchronous engine: the levels of a search.
// Part of sync_engine.cu, split by topic; included in order.
#pragma once

#include "sync_common.cuh"

namespace abfs {

// ---------------------------------------------------------------------------
// thin levels
// ---------------------------------------------------------------------------
// The frontier is spread over the CTAs' private lists: a CTA expands the
// columns it listed and lists the rows it wins, so a level needs no shared
// queue, no reservation in global memory and no reload -- its dependent chain
// is row index, atomicMin, barrier.  The lists are evened out only when a few
// CTAs hold much more than their share (see sync_search).

// The general case of thin_append: the warp's `tot` items (lane l's: the column
// [cb, cb + len) of label j; inclusive counts incl) go to positions at... of the
// list, those from kThinCap on to the global list, written by the warp together.
__device__ __noinline__ void thin_append_long(SyncSmem& sm, const SyncSearch& S, uint32_t k, uint32_t q,
                                              uint32_t at, uint32_t tot, uint32_t incl, uint32_t j,
                                              uint32_t cb, uint32_t len) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t p = (k + 1) & 1;
    const uint32_t before = incl - items_of(cb, len);
    const uint32_t room = at < kThinCap ? min(kThinCap - at, tot) : 0u;
    uint32_t spill = 0;
    if (room < tot) {
        if (lane == 0) spill = atomicAdd(&S.bar->lcnt[p], tot - room);
        spill = __shfl_sync(0xFFFFFFFFu, spill, 0);
    }
#pragma unroll 1
    for (uint32_t x0 = 0; x0 < tot; x0 += 32) {
        const uint32_t x = x0 + lane;
        uint32_t own = 0;  // the first lane whose inclusive count exceeds x
#pragma unroll
        for (uint32_t d = 16; d > 0; d >>= 1)
            if (x >= __shfl_sync(0xFFFFFFFFu, incl, own + d - 1)) own += d;
        const uint32_t oj = __shfl_sync(0xFFFFFFFFu, j, own), ob = __shfl_sync(0xFFFFFFFFu, cb, own);
        const uint32_t ol = __shfl_sync(0xFFFFFFFFu, len, own);
        const uint32_t of = __shfl_sync(0xFFFFFFFFu, before, own);
        if (x < tot) {
            uint32_t b, l;
            item_at(ob, ol, x - of, b, l);
            if (x < room) {
                sm.ij[q][at + x] = oj;
                sm.ib[q][at + x] = b;
                sm.il[q][at + x] = l;
            } else {
                list_put(S, p, (unsigned long long)spill + (x - room), oj, b, l);
            }
        }
    }
}

// Appends the rows won by this warp's lanes (row r, column [cb, ce)) to the
// CTA's list `q` (level k + 1); what does not fit goes to the global list.
// Whole warp.
__device__ __forceinline__ void thin_append(SyncSmem& sm, const SyncSearch& S, uint32_t k, uint32_t q,
                                            bool win, uint32_t r, uint32_t cb, uint32_t ce) {
    if (!__any_sync(0xFFFFFFFFu, win)) return;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t len = win ? ce - cb : 0u;
    const uint32_t ns = items_of(cb, len);
    const uint32_t ent = __reduce_add_sync(0xFFFFFFFFu, len);
    const uint32_t j = ns && S.lab ? ld_ro(S.lab + r) : r;
    // the next level starts with these row indices
    if (ns) asm volatile("prefetch.global.L2 [%0];" ::"l"(S.rowidx + cb));
    const bool longs = __any_sync(0xFFFFFFFFu, ns > 1);
    uint32_t incl, tot;
    if (longs) {
        incl = warp_incl_scan(ns);
        tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
    } else {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, ns != 0);
        tot = __popc(m);
        incl = __popc(m & lanemask_lt()) + ns;
    }
    // lane 0 reserves the items, lane 1 counts the entries
    uint32_t at = 0;
    if (lane < 2) at = atomicAdd(&sm.app[q][lane], lane ? ent : tot);
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (longs || at + tot > kThinCap) {
        thin_append_long(sm, S, k, q, at, tot, incl, j, cb, len);
    } else if (ns) {
        sm.ij[q][at + incl - 1] = j;
        sm.ib[q][at + incl - 1] = cb;
        sm.il[q][at + incl - 1] = len;
    }
}

// Expands the columns of this CTA's list of level k (list k & 1) into its list
// of level k + 1.  The warps share the list's batches of 32 items evenly; the
// warps of a batch take its groups of 32 entries in turn, one entry per lane
// and kThinIlp groups in flight, so that one hub or a handful of columns keeps
// all of them busy.
//
// A warp's first groups are staged while the team's barrier is under way: the
// row indices (and, where a CTA has few entries and the level is bound by
// latency, the rows' columns; their key words are brought to the L2) depend on
// this CTA's list alone.  The chain from one barrier to the next is then claim,
// append, arrive: 4096^2 grid 19.7 -> 15.4 ms, RGG 2^22 10.8 -> 8.7 ms.
constexpr int kThinIlp = 2;
// Entries per CTA up to which the columns of all rows are staged instead of
// looked up for the rows that are won, and the key words prefetched (the grid
// 16.5 ms without the prefetch), and up to which a list is staged before the
// barrier at all: a longer list is bound by its claims, and often the next
// level turns out to be wide (R-MAT-20 5 us slower with every list staged).
constexpr uint32_t kThinEarly = 1024, kThinPrefetch = 512, kThinAhead = 2048;

struct ThinStage {
    uint32_t r[kThinIlp], jj[kThinIlp], cb[kThinIlp], ce[kThinIlp];
    uint32_t j, first, shift;  // this lane's item: column, first entry, its position less that
    uint32_t e0, total, step;  // the warp's next group, the batch's entries, entries between groups
    bool early;                // cb and ce are there
};

// The rows and columns of kThinIlp groups from st.e0 on.
__device__ __forceinline__ void thin_groups(const SyncSearch& S, ThinStage& st) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t le_mask = (2u << lane) - 1u;
#pragma unroll
    for (int u = 0; u < kThinIlp; ++u) {
        const uint32_t g = st.e0 + u * st.step;
        st.r[u] = kUnset;
        st.jj[u] = 0;
        if (g < st.total) {
            const uint32_t rel = st.first - g;
            const uint32_t before = __popc(__ballot_sync(0xFFFFFFFFu, st.first < g));
            const uint32_t w = __reduce_or_sync(0xFFFFFFFFu, rel < 32u ? 1u << rel : 0u);
            // the item of entry g + lane
            const uint32_t own = (before + __popc(w & le_mask) - 1u) & 31u;
            const uint32_t pos = __shfl_sync(0xFFFFFFFFu, st.shift, own) + g + lane;
            st.jj[u] = __shfl_sync(0xFFFFFFFFu, st.j, own);
            if (g + lane < st.total) st.r[u] = ld_ro(S.rowidx + pos);
        }
    }
}

// Whole CTA.
__device__ __forceinline__ void thin_stage(const SyncSmem& sm, const SyncSearch& S, uint32_t cur, ThinStage& st) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t cnt = min(sm.app[cur][0], kThinCap);
    // batches of 32 items, rounded up to a power of two (at most one per warp)
    const uint32_t lb = cnt > 32 ? 32 - __clz((cnt - 1) / 32) : 0;
    const uint32_t batch = warp & ((1u << lb) - 1u), nth = warp >> lb;
    const uint32_t i0 = 32 * batch;
    st.e0 = 32 * nth;
    st.total = 0;
    if (i0 >= cnt || (lb == 0 && st.e0 >= sm.app[cur][1])) return;
    st.step = (32 * kSyncWarps) >> lb;
    uint32_t beg = 0, len = 0;
    st.j = 0;
    if (lane < cnt - i0) {
        st.j = sm.ij[cur][i0 + lane];
        beg = sm.ib[cur][i0 + lane];
        len = sm.il[cur][i0 + lane];
    }
    const uint32_t incl = warp_incl_scan(len);
    st.total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    // (lanes without an item are past every group)
    st.first = lane < cnt - i0 ? incl - len : kUnset;
    st.shift = beg - st.first;
    st.early = (st.total << lb) <= kThinEarly;
    thin_groups(S, st);
    if (!st.early) return;
    const bool far = (st.total << lb) <= kThinPrefetch;
#pragma unroll
    for (int u = 0; u < kThinIlp; ++u) {
        if (st.r[u] == kUnset) continue;
        if (far) asm volatile("prefetch.global.L2 [%0];" ::"l"(S.key + st.r[u]));
        st.cb[u] = ld_ro(S.colptr + st.r[u]);
        st.ce[u] = ld_ro(S.colptr + st.r[u] + 1);
    }
}

// Whole CTA.
template <bool SIG>
__device__ __forceinline__ void thin_claims(SyncSmem& sm, const SyncSearch& S, uint32_t k, ThinStage& st,
                                            SyncTally& t) {
    const uint32_t cur = k & 1;
    const unsigned long long hi = (unsigned long long)(k + 1) << 32;
#pragma unroll 1
    while (st.e0 < st.total) {
        unsigned long long old[kThinIlp];
#pragma unroll
        for (int u = 0; u < kThinIlp; ++u) {
            old[u] = 0;
            if (st.r[u] != kUnset) old[u] = atomicMin(S.key + st.r[u], hi | st.jj[u]);
        }
#pragma unroll
        for (int u = 0; u < kThinIlp; ++u) {
            if (st.e0 + u * st.step >= st.total) break;
            const bool have = st.r[u] != kUnset;
            const bool pass = have && (uint32_t)(old[u] >> 32) > k;
            const bool win = pass && old[u] == kKeyUnset;
            t.read += have;
            t.unmasked += pass;
            if (win) {
                ++t.verts;
                t.levels = k + 2;
            }
            if (SIG && pass) red_add64(S.sigma + st.r[u], ld_l2(S.sigma + st.jj[u]));
            uint32_t cb = 0, ce = 0;
            if (win) {
                cb = st.early ? st.cb[u] : ld_ro(S.colptr + st.r[u]);
                ce = st.early ? st.ce[u] : ld_ro(S.colptr + st.r[u] + 1);
            }
            thin_append(sm, S, k, cur ^ 1, win, st.r[u], cb, ce);
        }
        st.e0 += kThinIlp * st.step;
        if (st.e0 >= st.total) break;
        st.early = false;
        thin_groups(S, st);
    }
}

// ---------------------------------------------------------------------------
// wide levels
// ---------------------------------------------------------------------------
// The frontier is a list in global memory.  A row is tested against the
// visited bitmap (frozen during the level) and claimed by a 32-bit reduction
// on the low half of its key word, whose all-ones high half still says
// "unset"; after a barrier, sync_extract reads the new rows off the bitmap and
// the keys.  (The bitmap in shared memory, whole or in part, costs the L1 that
// the misses of the other loads wait in: an R-MAT of scale 20 the same, of
// scale 22 758 -> 877 us.)

// Bits of word w that stand for vertices.
__device__ __forceinline__ uint32_t word_mask(const SyncSearch& S, uint32_t w) {
    return w == S.nwords - 1 && (S.n & 31) ? (1u << (S.n & 31)) - 1u : 0xFFFFFFFFu;
}

// Expands the `items` items of the global list of level k.  A warp takes up to
// 32 items at a time and walks their chunks of four row indices, one 16-byte
// load per lane and step, the next step's loads issued before this step's
// tests; there is no barrier inside.  Whole CTA.
enum WideKind : int {
    kWidePlain = 0,
    kWideCounts = 1,  // and shortest-path counts
    kWideMulti = 2,   // multi-source search: every row gets the frontier bits of the column
                      // that it lacks, in the next-bit masks
};

// BITS: the graph has at most kBitsN vertices, and its bitmap is copied into the
// place of the thin levels' lists, which a wide level does not need: a test then
// costs a bank conflict or two instead of a cycle per entry for its cache line
// (a batch of 32 graphs of 2^12..2^17 vertices, 317 -> 213 us).
static_assert(kBitsN / 8 == sizeof(SyncSmem::ij) + sizeof(SyncSmem::ib) + sizeof(SyncSmem::il), "the lists' bytes");

template <int KIND, bool BITS>
__device__ __noinline__ void wide_expand(SyncSmem& sm, const SyncSearch& S, const Team& T, uint32_t k,
                                         unsigned long long items) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t le_mask = (2u << lane) - 1u;
    const uint32_t p = k & 1;
    // The list is dealt out to the CTAs in runs of items, round robin, and a CTA's
    // runs to its warps as they become free, by a counter in shared memory (one
    // counter for the whole team, taken at about 2 ns a time, set the pace of a
    // level of 25 000 runs).  A run is about four steps of 32 chunks, so that one
    // full of hub items does not outlast the level, and short enough for four
    // per warp.
    // (a list's positions fit 32 bits)
    const uint32_t W = T.size * kSyncWarps, n = (uint32_t)items;
    const float avg = __fdividef((float)sm.entries, (float)n) + (float)kChunk;
    const uint32_t four = (uint32_t)__fdividef(4.f * 32 * kChunk, avg);
    const uint32_t run = max(1u, min(min(32u, four), n / (4u * W)));
    const uint32_t runs = (n + run - 1) / run;
    const uint64_t pol = evict_first_policy();
    const uint32_t* const bm = BITS ? &sm.ij[0][0] : S.bm;
    if (BITS) {
        for (uint32_t w = threadIdx.x; w < S.nwords; w += kSyncThreads) (&sm.ij[0][0])[w] = ld_l2(S.bm + w);
        __syncthreads();
    }
    uint32_t* const klo = reinterpret_cast<uint32_t*>(S.key);
    SyncTally t;
    // the items of the run after the current one
    uint32_t nj = 0, nbeg = 0, nlen = 0;
    auto fetch = [&]() {
        uint32_t x = 0;
        if (lane == 0) {
            x = atomicAdd(&sm.tick, 1u);
            sync_beat(S, x, 256);
        }
        const unsigned long long c = (unsigned long long)__shfl_sync(0xFFFFFFFFu, x, 0) * T.size + T.rank;
        const unsigned long long at = c * run + lane;
        nj = nbeg = nlen = 0;
        if (lane < run && at < items) {
            nj = ld_l2(S.lj[p] + at);
            nbeg = ld_l2(S.lb[p] + at);
            nlen = ld_l2(S.ll[p] + at);
        }
        return c < runs;
    };
    bool more = fetch();
    // this lane's item of the current run: column, entries [beg, end), its first
    // chunk's position in the run, chunk number minus position
    uint32_t j = 0, beg = 0, end = 0, first = kUnset, shift = 0;
    uint32_t total = 0, g = 0, started = 0;  // the run's chunks, the next step's first, items begun
    // Issues the loads of the next step: row indices of a lane's chunk, which of
    // them belong to its column (bits of ok) and the column's label.  The raw
    // indices are kept as loaded: anything computed from them here would wait
    // for the load.  False when the level is out of runs.
    auto issue = [&](uint4& r, uint32_t& ok, uint32_t& jj) {
#pragma unroll 1
        while (g >= total) {
            ok = 0;
            if (!more) return false;
            j = nj;
            beg = nbeg;
            end = nbeg + nlen;
            const uint32_t nch = nlen ? ((nbeg & (kChunk - 1)) + nlen + kChunk - 1) / kChunk : 0u;
            t.read += nlen;
            more = fetch();
            const uint32_t incl = warp_incl_scan(nch);
            total = __shfl_sync(0xFFFFFFFFu, incl, 31);
            first = nch ? incl - nch : kUnset;
            shift = beg / kChunk - first;
            g = started = 0;
        }
        const uint32_t rel = first - g;
        const uint32_t w = __reduce_or_sync(0xFFFFFFFFu, rel < 32u ? 1u << rel : 0u);
        const uint32_t own = (started + __popc(w & le_mask) - 1u) & 31u;
        started += __popc(w);
        const uint32_t pos = (__shfl_sync(0xFFFFFFFFu, shift, own) + g + lane) * kChunk;
        const uint32_t lo = __shfl_sync(0xFFFFFFFFu, beg, own);
        const uint32_t up = __shfl_sync(0xFFFFFFFFu, end, own);
        jj = __shfl_sync(0xFFFFFFFFu, j, own);
        ok = 0;
        if (g + lane < total) {
            // entries [max(pos, lo), min(pos + 4, up)) of the chunk
            const uint32_t skip = lo > pos ? lo - pos : 0u;
            const uint32_t have = min(up - pos, kChunk);
            ok = (1u << have) - (1u << skip);
            if ((unsigned long long)pos + kChunk <= S.nnz) {
                r = ld_row4(S.rowidx + pos, 0, pol);
            } else {
                // the last chunk of the row array
                const uint32_t* const x = S.rowidx + pos;
                r.x = (ok & 1u) ? ld_ro(x) : 0u;
                r.y = (ok & 2u) ? ld_ro(x + 1) : 0u;
                r.z = (ok & 4u) ? ld_ro(x + 2) : 0u;
                r.w = 0u;
            }
        }
        g += 32;
        return true;
    };
    auto process = [&](const uint4& rr, uint32_t ok, uint32_t jj) {
        const uint32_t r[kChunk] = {rr.x, rr.y, rr.z, rr.w};
        if (KIND == kWideMulti) {
            const unsigned long long f = ok ? ld_l2(S.ms_fr[p] + jj) : 0ull;
            unsigned long long vis[kChunk];
#pragma unroll
            for (uint32_t q = 0; q < kChunk; ++q)
                vis[q] = (ok >> q) & 1u ? ld_l2(S.ms_vis + r[q]) : ~0ull;
#pragma unroll
            for (uint32_t q = 0; q < kChunk; ++q)
                if (f & ~vis[q]) red_or64(S.ms_nx + r[q], f & ~vis[q]);
            return;
        }
        uint32_t w[kChunk];
#pragma unroll
        for (uint32_t q = 0; q < kChunk; ++q)
            w[q] = (ok >> q) & 1u ? ld_frozen(bm + (r[q] >> 5)) : 0xFFFFFFFFu;
#pragma unroll
        for (uint32_t q = 0; q < kChunk; ++q) {
            if (!((w[q] >> (r[q] & 31)) & 1u)) {
                ++t.unmasked;
                red_min32(klo + 2ull * r[q], jj);
                if (KIND == kWideCounts) red_add64(S.sigma + r[q], ld_l2(S.sigma + jj));
            }
        }
    };
    // One copy of each half of the loop: it has to stay in the instruction cache
    // (with the two buffers in turn, twice the code: R-MAT-20 161 -> 168 us,
    // path counts 216 -> 250 us).
    uint4 r0 = make_uint4(0, 0, 0, 0), r1 = r0;
    uint32_t ok0 = 0, ok1 = 0, j0 = 0, j1 = 0;
    bool on = true;
#pragma unroll 1
    while (on) {  // (the first step has nothing to process: ok0 is 0)
        on = issue(r1, ok1, j1);
        process(r0, ok0, j0);
        r0 = r1;
        ok0 = ok1;
        j0 = j1;
    }
    tally_add(sm, t.read, t.unmasked);
}

// The visited bitmap (and, for the hybrid, the frontier bitmap of level k)
// from the key words, after thin levels.  Rows that no column contains count
// as visited.  A warp has the keys of kBitmapWords words in flight: with four,
// 33 MB of keys took 25 us.  Whole CTA.
constexpr int kBitmapWords = 8;

__device__ __noinline__ void sync_bitmaps(const SyncSearch& S, const Team& T, uint32_t k) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t W = T.size * kSyncWarps;
    constexpr int Q = kBitmapWords;
    const bool slow = sync_long_pass(S, T);
    for (uint32_t w0 = (warp * T.size + T.rank) * Q; w0 < S.nwords; w0 += Q * W) {
        if (slow) red_add64(&S.bar->beat, 1ull);
        uint32_t lv[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const unsigned long long v = ((unsigned long long)w0 + q) * 32 + lane;
            lv[q] = v < S.n ? (uint32_t)(ld_relaxed64(S.key + v) >> 32) : kUnset;
        }
        uint32_t vis = 0, fr = 0;  // lane q: word w0 + q
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const uint32_t a = __ballot_sync(0xFFFFFFFFu, lv[q] != kUnset);
            const uint32_t b = __ballot_sync(0xFFFFFFFFu, lv[q] == k);
            if (lane == (uint32_t)q) {
                vis = a;
                fr = b;
            }
        }
        const uint32_t w = w0 + lane;
        if (lane < (uint32_t)Q && w < S.nwords) {
            if (S.inb) vis |= ~ld_ro(S.inb + w) & word_mask(S, w);
            S.bm[w] = vis;
            if (S.bu_alpha) S.fbm[k & 1][w] = fr;
        }
    }
}

// Writes the items of this warp's columns (lane l's: [cb, cb + len), label j;
// none if empty) from position `at` of the global list on; returns their number.
// The lanes share the items: a hub's 400 written by its own lane held its warp,
// and with it the level, for 25 us.  Whole warp.
__device__ __noinline__ uint32_t list_put_long(const SyncSearch& S, uint32_t p, uint32_t at, uint32_t j,
                                               uint32_t cb, uint32_t len) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t ns = items_of(cb, len), incl = warp_incl_scan(ns);
    const uint32_t tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
#pragma unroll 1
    for (uint32_t x0 = 0; x0 < tot; x0 += 32) {
        const uint32_t x = x0 + lane;
        uint32_t own = 0;  // the first lane whose inclusive count exceeds x
#pragma unroll
        for (uint32_t d = 16; d > 0; d >>= 1)
            if (x >= __shfl_sync(0xFFFFFFFFu, incl, own + d - 1)) own += d;
        const uint32_t oj = __shfl_sync(0xFFFFFFFFu, j, own), ob = __shfl_sync(0xFFFFFFFFu, cb, own);
        const uint32_t ol = __shfl_sync(0xFFFFFFFFu, len, own);
        const uint32_t of = __shfl_sync(0xFFFFFFFFu, incl - ns, own);
        if (x < tot) {
            uint32_t b, l;
            item_at(ob, ol, x - of, b, l);
            list_put(S, p, (unsigned long long)at + x, oj, b, l);
        }
    }
    return tot;
}

// The frontier list of level k + 1.  kFromKeys: after a wide level, its new
// vertices are those outside the bitmap whose key has a parent; they get their
// level, join the bitmap (each word has one writer) and make up the frontier
// bitmap of level k + 1.  kFromBits: that bitmap is there already (after a
// bottom-up level, which counted its vertices).  kFromMasks: the vertices with
// frontier bits of a multi-source search.
//
// Two passes over a warp's words, so that the CTA meets once and reserves its
// items with one atomic: the first finds the new vertices and counts their
// items, kExtractWords words at a time in flight, the second reads the columns
// again (from L2) and writes the items in order.  One pass with a meeting and a
// reservation per 8192 vertices took 58 us for two million new vertices of
// four million, most of it waiting.  Whole CTA.
constexpr uint32_t kExtractWords = 8;

enum ExtractKind : int { kFromKeys, kFromBits, kFromMasks };

template <int KIND>
__device__ __noinline__ void sync_extract(SyncSmem& sm, const SyncSearch& S, const Team& T, uint32_t k) {
    constexpr bool FROM_KEYS = KIND == kFromKeys, MASKS = KIND == kFromMasks;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr uint32_t Q = kExtractWords;
    const uint32_t pn = (k + 1) & 1;
    const uint32_t W = T.size * kSyncWarps;
    const uint32_t g0 = (warp * T.size + T.rank) * Q;  // groups of Q words, round robin
    uint32_t* const khi = reinterpret_cast<uint32_t*>(S.key) + 1;
    uint32_t verts = 0, entries = 0, mine = 0;
    const bool slow = sync_long_pass(S, T);
    // this lane's word of the group at wb, loaded a group ahead (a batch of 128
    // graphs 608 -> 598 us)
    auto load = [&](const uint32_t* bits, uint32_t wb) {
        return lane < Q && wb < S.nwords && lane < S.nwords - wb ? ld_l2(bits + wb + lane) : 0u;
    };
    const uint32_t* const from = FROM_KEYS ? S.bm : S.fbm[pn];
    uint32_t ahead = MASKS ? 0u : load(from, g0);
#pragma unroll 1
    for (uint32_t wb = g0; wb < S.nwords; wb += Q * W) {
        if (slow) red_add64(&S.bar->beat, 1ull);
        const bool own = lane < Q && wb + lane < S.nwords;
        const uint32_t seen = ahead;
        uint32_t word = 0, add = 0;
        if (!MASKS) ahead = load(from, wb + Q * W);
        if (own) word = FROM_KEYS ? ~seen & word_mask(S, wb + lane) : MASKS ? word_mask(S, wb + lane) : seen;
        const unsigned long long v0 = (unsigned long long)wb * 32 + lane;
        bool fresh[Q];
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            const uint32_t c = __shfl_sync(0xFFFFFFFFu, word, q);
            fresh[q] = (c >> lane) & 1u;
            if (FROM_KEYS && fresh[q]) fresh[q] = (uint32_t)ld_l2(S.key + v0 + 32 * q) != kUnset;
            if (MASKS && fresh[q]) fresh[q] = ld_l2(S.ms_fr[pn] + v0 + 32 * q) != 0ull;
        }
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            if (FROM_KEYS || MASKS) {
                const uint32_t bits = __ballot_sync(0xFFFFFFFFu, fresh[q]);
                if (lane == q) add = bits;
            }
            if (fresh[q]) {
                const uint32_t cb = ld_ro(S.colptr + v0 + 32 * q);
                const uint32_t len = ld_ro(S.colptr + v0 + 32 * q + 1) - cb;
                if (FROM_KEYS) khi[2 * (v0 + 32 * q)] = k + 1;
                ++verts;
                entries += len;
                mine += items_of(cb, len);
            }
        }
        if (FROM_KEYS && own && add) S.bm[wb + lane] = seen | add;
        if ((FROM_KEYS || MASKS) && own) S.fbm[pn][wb + lane] = add;
    }
    const uint32_t wt = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0) sm.wsum[warp] = wt;
    __syncthreads();
    if (warp == 0) {
        const uint32_t x = sm.wsum[lane];
        const uint32_t incl = warp_incl_scan(x);
        uint32_t base = 0;
        if (lane == 31) {
            if (incl) base = atomicAdd(&S.bar->lcnt[pn], incl);
            sm.app[0][0] = incl;
        }
        base = __shfl_sync(0xFFFFFFFFu, base, 31);
        sm.wpre[lane] = base + incl - x;
    }
    if (KIND != kFromBits) {
        verts = __reduce_add_sync(0xFFFFFFFFu, verts);
        entries = __reduce_add_sync(0xFFFFFFFFu, entries);
        if (lane == 0 && verts) {
            atomicAdd(&sm.verts, verts);
            atomicAdd(&sm.ent, entries);
        }
    }
    __syncthreads();
    if (!wt) return;
    uint32_t at = sm.wpre[warp];
    // (this lane's own words of the first pass)
    ahead = load(S.fbm[pn], g0);
#pragma unroll 1
    for (uint32_t wb = g0; wb < S.nwords; wb += Q * W) {
        if (slow) red_add64(&S.bar->beat, 1ull);
        const uint32_t word = ahead;
        ahead = load(S.fbm[pn], wb + Q * W);
        if (!__any_sync(0xFFFFFFFFu, word != 0)) continue;
        const unsigned long long v0 = (unsigned long long)wb * 32 + lane;
        uint32_t cb[Q], len[Q];
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            const uint32_t c = __shfl_sync(0xFFFFFFFFu, word, q);
            cb[q] = len[q] = 0;
            if ((c >> lane) & 1u) {
                cb[q] = ld_ro(S.colptr + v0 + 32 * q);
                len[q] = ld_ro(S.colptr + v0 + 32 * q + 1) - cb[q];
            }
        }
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            const uint32_t ns = items_of(cb[q], len[q]);
            if (!__any_sync(0xFFFFFFFFu, ns != 0)) continue;
            const unsigned long long v = v0 + 32 * q;
            const uint32_t j = ns && S.lab ? ld_ro(S.lab + v) : (uint32_t)v;
            if (!__any_sync(0xFFFFFFFFu, ns > 1)) {
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, ns != 0);
                if (ns) list_put(S, pn, (unsigned long long)at + __popc(m & lanemask_lt()), j, cb[q], len[q]);
                at += __popc(m);
            } else {
                at += list_put_long(S, pn, at, j, cb[q], len[q]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// hybrid: bottom-up levels (direction optimisation; not the paper's method)
// ---------------------------------------------------------------------------
// As in the unit scheduler (engine_phases.cuh): an unvisited vertex scans its
// ascending column for the first vertex of the frontier bitmap, which is its
// least-index parent.  The CTAs take groups of four words in turn, a CTA's
// warps its groups as they become free.
constexpr uint32_t kBuWords = 4;

__device__ __noinline__ void sync_bottom_up(SyncSmem& sm, const SyncSearch& S, const Team& T, uint32_t k) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t p = k & 1, pn = p ^ 1;
    const uint32_t* const fbm = S.fbm[p];
    SyncTally t;
    uint32_t verts = 0, entries = 0;
#pragma unroll 1
    for (;;) {
        uint32_t x = 0;
        if (lane == 0) {
            x = atomicAdd(&sm.tick, 1u);
            sync_beat(S, x, 64);
        }
        x = __shfl_sync(0xFFFFFFFFu, x, 0);
        const unsigned long long c = ((unsigned long long)x * T.size + T.rank) * kBuWords;
        if (c >= S.nwords) break;
        const uint32_t w0 = (uint32_t)c;
        const bool own = lane < kBuWords && w0 + lane < S.nwords;
        uint32_t seen = 0, cand = 0, add = 0;
        if (own) {
            seen = ld_l2(S.bm + w0 + lane);
            cand = ~seen & word_mask(S, w0 + lane);
        }
        for (uint32_t q = 0; q < kBuWords; ++q) {
            const uint32_t cw = __shfl_sync(0xFFFFFFFFu, cand, q);
            if (!cw) continue;
            const uint32_t v = (w0 + q) * 32 + lane;
            uint32_t cb = 0, e = 0, end = 0, par = kUnset;
            if ((cw >> lane) & 1u) {
                cb = e = ld_ro(S.colptr + v);
                end = ld_ro(S.colptr + v + 1);
            }
            for (uint32_t b = 0; b < 4 && e < end; ++b) {
                uint32_t jj[4], fw[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) jj[x] = e + x < end ? ld_ro(S.rowidx + e + x) : kUnset;
#pragma unroll
                for (int x = 0; x < 4; ++x) fw[x] = jj[x] != kUnset ? ld_frozen(fbm + (jj[x] >> 5)) : 0u;
                t.read += min(4u, end - e);
#pragma unroll
                for (int x = 3; x >= 0; --x)
                    if ((fw[x] >> (jj[x] & 31)) & 1u) par = jj[x];
                e = par != kUnset ? end : e + 4;
            }
            uint32_t dm;
            bool defer = par == kUnset && e < end;
            while ((dm = __ballot_sync(0xFFFFFFFFu, defer)) != 0u) {
                const uint32_t ldr = __ffs(dm) - 1;
                const uint32_t le = __shfl_sync(0xFFFFFFFFu, e, ldr);
                const uint32_t lend = __shfl_sync(0xFFFFFFFFu, end, ldr);
                uint32_t found = kUnset;
                for (uint32_t x = le; x < lend; x += 32) {
                    if (lane == 0) sync_beat(S, (x - le) / 32, 1024);
                    const uint32_t idx = x + lane;
                    const uint32_t j = idx < lend ? ld_ro(S.rowidx + idx) : kUnset;
                    const bool hit = j != kUnset && ((ld_frozen(fbm + (j >> 5)) >> (j & 31)) & 1u);
                    const uint32_t hb = __ballot_sync(0xFFFFFFFFu, hit);
                    if (lane == 0) t.read += min(32u, lend - x);
                    if (hb) {
                        found = __shfl_sync(0xFFFFFFFFu, j, __ffs(hb) - 1);
                        break;
                    }
                }
                if (lane == ldr) {
                    par = found;
                    defer = false;
                }
            }
            const bool got = par != kUnset;
            if (got) {
                S.key[v] = (unsigned long long)(k + 1) << 32 | par;
                ++t.unmasked;
                ++verts;
                entries += end - cb;
            }
            const uint32_t bits = __ballot_sync(0xFFFFFFFFu, got);
            if (lane == q) add = bits;
        }
        if (own) {
            if (add) S.bm[w0 + lane] = seen | add;
            S.fbm[pn][w0 + lane] = add;
        }
    }
    tally_add(sm, t.read, t.unmasked);
    verts = __reduce_add_sync(0xFFFFFFFFu, verts);
    entries = __reduce_add_sync(0xFFFFFFFFu, entries);
    if (lane == 0 && verts) {
        atomicAdd(&sm.verts, verts);
        atomicAdd(&sm.ent, entries);
    }
}

}  // namespace abfs
