// Level-synchronous engine: shared state, the team barrier and the frontier
// lists.  Part of sync_engine.cu, split by topic; included in order.
//
// One search runs on a team of P CTAs that are resident together (a
// cooperative launch).  Every vertex has one 64-bit word
//     key[v] = level << 32 | parent   (all ones: not reached)
// and a level is a bulk-synchronous step between two team barriers.  Because
// the level is the high half, one atomicMin on the word masks and claims at
// once: a row reached earlier has a smaller level and keeps its word, a row of
// the next level keeps the least column index, and the returned value tells
// whether the row was new (Theorem 1's product in the (min, index) semiring
// with the mask V_{k+1} folded into the order of the keys).
#pragma once

#include "engine_common.cuh"

namespace abfs {

constexpr int kSyncThreads = 1024;
constexpr int kSyncWarps = kSyncThreads / 32;
// Columns are listed in items of at most kSeg entries (split where the row
// index is a multiple of kChunk), so that any number of warps can share a hub.
constexpr uint32_t kSeg = kSyncSeg;
// Items a CTA keeps of a thin level's frontier.  Two lists of 12-byte items
// stay under the 32 KB shared-memory split, which leaves 224 KB of L1 for the
// bitmap words of wide levels.
constexpr uint32_t kThinCap = 1024;
constexpr unsigned long long kKeyUnset = ~0ull;
// A barrier word holds the arrivals and the totals of the next level; it only
// ever grows, and what a barrier added is its difference to the barrier two
// steps back (barriers alternate between two words, so nobody can add to a
// word that a slower CTA still waits on, and no word is cleared in flight).
//   thin level:  [arrived : 8][full lists : 8][heavy lists : 8][items : 21][entries / 64 : 19]
//   otherwise:   [arrived : 8][items : 56]
// (a CTA's share of a thin word is clamped so that 240 of them fit their field;
// exact totals follow with the next barrier where they matter).  Beside it,
// for the hybrid and traces: [vertices : 31][column entries : 33].
constexpr uint32_t kArriveShift = 56, kFullShift = 48, kHeavyShift = 40, kItemShift = 19;
constexpr uint32_t kEntUnit = 64, kItemClamp = 8191;
constexpr uint32_t kAuxShift = 33;

// What a level is followed by; the team's CTAs agree on it because they decide
// from the same totals.
enum SyncAct : uint32_t {
    kActThin = 0,    // the next level is thin, the lists stay where they are
    kActEven = 1,    // thin, after the lists were evened out through the global list
    kActWide = 2,    // the next level is wide
    kActSlice = 3,   // thin, from the global list that a wide level left
    kActBottomUp = 4,
    kActDone = 5,
    kActFailed = 6,  // the bounded wait ran out, or an append failed
};

struct SyncSmem {
    // items of the current and the next thin level: column label, first row
    // index, entries
    uint32_t ij[2][kThinCap], ib[2][kThinCap], il[2][kThinCap];
    // [0] items appended to each list (may exceed kThinCap: the rest is
    // spilled), [1] column entries of their vertices
    uint32_t app[2][2];
    uint32_t verts, ent;              // wide levels: vertices this CTA reached, their entries
    uint32_t tick;                    // wide levels: runs this CTA's warps have taken
    uint32_t base;
    uint32_t at, left;                // what is left of this CTA's share of the global list
    uint32_t wsum[kSyncWarps], wpre[kSyncWarps];
    uint32_t act;                     // SyncAct after the last barrier
    uint32_t passed;                  // whether the last team_sync was passed (written there only)
    unsigned long long items;         // the next level's items
    // thread 0's state of the search
    uint32_t lim;                     // a list of more weight is heavy
    float weight;                     // of the current level's lists
    uint32_t ent_clamp;               // a CTA's largest part of a thin word's entries
    uint32_t bu;
    unsigned long long nf, entries, seen;
    unsigned long long st_read, st_unmasked, st_verts, st_ent;
    uint32_t levels;
    // multi-source searches: columns left to the whole CTA, and the masks its
    // warps found in a round
    uint32_t nlong;
    unsigned long long open;                  // entries of vertices some source has not reached
    unsigned long long wm[2][kSyncWarps];
    uint32_t step;                            // barriers passed
    unsigned long long word[2], aux[2];       // the barrier words as last seen
    unsigned long long wait_from, wait_seen;  // bar_late's clock and the progress it saw
};

// A CTA's place in its team.
struct Team {
    uint32_t rank, size;
    uint32_t expect;  // arrivals a barrier waits for (more than size only in the held tests)
};

// Counters of a thread over a whole search.
struct SyncTally {
    uint32_t read = 0, unmasked = 0, verts = 0, levels = 0;
};

// Adds a warp's counters to the CTA's.  Whole warp.
__device__ __forceinline__ void tally_add(SyncSmem& sm, uint32_t read, uint32_t unmasked) {
    read = __reduce_add_sync(0xFFFFFFFFu, read);
    unmasked = __reduce_add_sync(0xFFFFFFFFu, unmasked);
    if ((threadIdx.x & 31) == 0) {
        if (read) atomicAdd(&sm.st_read, (unsigned long long)read);
        if (unmasked) atomicAdd(&sm.st_unmasked, (unsigned long long)unmasked);
    }
}

__device__ __forceinline__ void red_add64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// The least value wins; nothing comes back.  (atomicMin with its result unused
// is compiled to an atomic that returns.)
__device__ __forceinline__ void red_min32(uint32_t* p, uint32_t v) {
    asm volatile("red.relaxed.gpu.global.min.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_or64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.relaxed.gpu.global.or.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_add_release64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Progress, for the waits of the other CTAs of the launch: in a batch a member
// may wait for one that is busy in another search, for as long as that search
// takes.  Barriers show it by themselves (bar_late reads the words of all
// searches of the launch); a step between two barriers that can outlast a
// millisecond counts its search's beat up once in a while: one lane, at each
// `every`-th (a power of two) piece of work, of which `n` counts.  Passes over
// the vertices, which the CTAs share evenly, do at each step of the team's first
// thread if a CTA has a million vertices or more.  (A count shared by a batch of
// 128, moved at every step of those passes and in every 16th thin level:
// 593 -> 606 us, 4096^2 grid 14.3 -> 14.5 ms.)
__device__ __forceinline__ void sync_beat(const SyncSearch& S, uint32_t n, uint32_t every) {
    if ((n & (every - 1)) == every - 1) red_add64(&S.bar->beat, 1ull);
}
__device__ __forceinline__ bool sync_long_pass(const SyncSearch& S, const Team& T) {
    return T.rank == 0 && threadIdx.x == 0 && (S.n >> 20) >= T.size;
}

// A CTA fails its search.  The status stands beside the barrier words and, like
// them, is cleared by the last CTA to leave, which copies it to the control
// block: a member that has waited in vain may fail before rank 0, busy in
// another search of the batch, has begun this one and cleared its control block.
__device__ __forceinline__ void sync_fail(const SyncSearch& S, uint32_t code) {
    atomicCAS(&S.bar->err, 0u, code);
}

// A waiting thread, now and then: whether its wait has run out, which fails the
// search.  The clock starts at the first look and again whenever the launch has
// made progress since the last one.
__device__ __noinline__ bool bar_late(SyncSmem& sm, const SyncSearch& S, bool first) {
    const unsigned long long now = globaltimer();
    unsigned long long seen = 0;
#pragma unroll 4
    for (uint32_t i = 0; i < S.nbars; ++i) {
        const SyncBar* const b = reinterpret_cast<const SyncBar*>(S.bars + (size_t)kBarStride * i);
        // (a sum that each new arrival and each beat changes)
        seen += ld_relaxed64(&b->word[0]) + 3 * ld_relaxed64(&b->word[1]) + 5 * ld_relaxed64(&b->beat);
    }
    if (first || seen != sm.wait_seen) {
        sm.wait_from = now;
        sm.wait_seen = seen;
    }
    if (now - sm.wait_from <= S.timeout_ns) return false;
    sync_fail(S, 5 /* ABFS_ERR_TIMEOUT */);
    return true;
}

// One thread of each CTA: adds `add` and the arrival to the barrier's word
// (bar_arrive), waits until the team has arrived and returns the totals, or ~0
// when the bounded wait ran out or, after a FULL barrier, a CTA has failed the
// search (bar_poll).  The wait itself delivers the totals: no further read
// follows unless `aux` is wanted.
//
// FULL: what the CTAs wrote before the barrier can be read after it.  Without
// it the barrier orders only the claims of a thin level: each was an atomic on
// a key word whose returned value its CTA has used before it arrived, so it
// has been performed at the L2, and everything the next level does with a key
// word is another atomic or a strong load there.  The release and the acquire
// cost 1.1 + 0.8 thousand cycles of a thin level's 8.4.  The same holds for the
// list counters lcnt: a thin level reserves in them by atomics, and whoever
// resets one does it before a FULL barrier or by an atomic whose result it has
// used.
template <bool FULL>
__device__ __forceinline__ void bar_arrive(SyncSmem& sm, const SyncSearch& S, const Team& T,
                                           unsigned long long add, unsigned long long aux) {
    if (T.expect == 1) return;
    const uint32_t b = sm.step & 1u;
    if (FULL) {
        if (aux) red_add64(&S.bar->aux[b], aux);
        red_add_release64(&S.bar->word[b], add + (1ull << kArriveShift));
    } else {
        red_add64(&S.bar->word[b], add + (1ull << kArriveShift));
    }
}
template <bool FULL>
__device__ __forceinline__ unsigned long long bar_poll(SyncSmem& sm, const SyncSearch& S, const Team& T,
                                                       unsigned long long add, unsigned long long& aux) {
    if (T.expect == 1) return add;
    const uint32_t b = sm.step & 1u;
    // (held tests: from barrier hold_from on)
    const uint32_t expect = T.expect != T.size && sm.step < S.hold_from ? T.size : T.expect;
    ++sm.step;
    unsigned long long* w = &S.bar->word[b];
    const unsigned long long before = sm.word[b];
    unsigned long long v;
    for (uint32_t spin = 0;; ++spin) {
        v = ld_relaxed64(w);
        if ((uint32_t)((v - before) >> kArriveShift) == expect) break;
        // reading %globaltimer is slow: the clock is looked at every 4096 polls
        if ((spin & 4095u) == 4095u && bar_late(sm, S, spin == 4095u)) return ~0ull;
    }
    sm.word[b] = v;
    if (FULL) {
        __threadfence();  // acquire: what the others wrote before they arrived
        const unsigned long long x = ld_relaxed64(&S.bar->aux[b]);
        const uint32_t err = ld_relaxed(&S.bar->err);
        aux = x - sm.aux[b];
        sm.aux[b] = x;
        if (err) return ~0ull;
    }
    return (v - before) & ((1ull << kArriveShift) - 1);
}
template <bool FULL>
__device__ __forceinline__ unsigned long long bar_wait(SyncSmem& sm, const SyncSearch& S, const Team& T,
                                                       unsigned long long add, unsigned long long& aux) {
    bar_arrive<FULL>(sm, S, T, add, aux);
    return bar_poll<FULL>(sm, S, T, add, aux);
}

// A plain full barrier; the sums of `add` and `ent` (thread 0's) reach sm.items
// and sm.entries.
// Returns false when the bounded wait ran out.  The verdict has a word of its
// own: callers go on to write sm.items without another __syncthreads, and every
// thread has to read the same verdict.  Whole CTA.
__device__ __forceinline__ bool team_sync(SyncSmem& sm, const SyncSearch& S, const Team& T,
                                          unsigned long long add = 0, unsigned long long ent = 0) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long tot = bar_wait<true>(sm, S, T, add, ent);
        sm.items = tot;
        sm.entries = ent;
        sm.passed = tot != ~0ull;
    }
    __syncthreads();
    return sm.passed != 0;
}

// Items of the column [beg, beg + len).
__device__ __forceinline__ uint32_t items_of(uint32_t beg, uint32_t len) {
    return len ? ((beg & (kChunk - 1)) + len + kSeg - 1) / kSeg : 0u;
}
// Item i of that column: every item but the first starts on a chunk.
__device__ __forceinline__ void item_at(uint32_t beg, uint32_t len, uint32_t i, uint32_t& b, uint32_t& l) {
    const uint32_t h = beg & (kChunk - 1);
    const uint32_t lo = i ? i * kSeg - h : 0u;
    b = beg + lo;
    l = min(len, (i + 1) * kSeg - h) - lo;
}

// Writes item (j, b, l) at position `at` of the global list of parity p.
__device__ __forceinline__ void list_put(const SyncSearch& S, uint32_t p, unsigned long long at,
                                         uint32_t j, uint32_t b, uint32_t l) {
    if (at < S.icap) {
        S.lj[p][at] = j;
        S.lb[p][at] = b;
        S.ll[p][at] = l;
    } else {
        sync_fail(S, 7 /* ABFS_ERR_DEVICE */);
    }
}

// Moves this CTA's list `q` to the global list of parity p (the spilled part
// is there already).  A team barrier follows.  Whole CTA.
__device__ __noinline__ void list_dump(SyncSmem& sm, const SyncSearch& S, uint32_t q, uint32_t p) {
    const uint32_t c = min(sm.app[q][0], kThinCap);
    __syncthreads();
    if (threadIdx.x == 0) {
        sm.base = c ? atomicAdd(&S.bar->lcnt[p], c) : 0u;
        sm.app[q][0] = sm.app[q][1] = 0;
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < c; i += kSyncThreads)
        list_put(S, p, (unsigned long long)sm.base + i, sm.ij[q][i], sm.ib[q][i], sm.il[q][i]);
}

// The next items of this CTA's share of the global list of parity p (the share:
// sm.left items from sm.at on) in its list `q`, as many as that holds.  Whole CTA.
__device__ __noinline__ void list_round(SyncSmem& sm, const SyncSearch& S, uint32_t q, uint32_t p) {
    const uint32_t at = sm.at, left = sm.left;
    const uint32_t c = min(left, kThinCap);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < c && at + i < S.icap; i += kSyncThreads) {
        sm.ij[q][i] = ld_l2(S.lj[p] + at + i);
        sm.ib[q][i] = ld_l2(S.lb[p] + at + i);
        sm.il[q][i] = ld_l2(S.ll[p] + at + i);
    }
    if (threadIdx.x == 0) {
        sync_beat(S, 0, 1);
        sm.at = at + c;
        sm.left = left - c;
        sm.app[q][0] = c;
        sm.app[q][1] = ~0u;  // entries: not known
    }
    __syncthreads();
}

// Gives this CTA its even share of the global list of parity p (`items` items),
// the first round of it in its list `q`.  Whole CTA.
__device__ __noinline__ void list_slice(SyncSmem& sm, const SyncSearch& S, const Team& T, uint32_t q,
                                        uint32_t p, unsigned long long items) {
    if (threadIdx.x == 0) {
        sm.at = (uint32_t)(items * T.rank / T.size);
        sm.left = (uint32_t)(items * (T.rank + 1) / T.size) - sm.at;
        // Every reservation in this list was made before the last barrier.  The
        // next barrier may be a thin level's, which orders no stores: the reset
        // is an atomic whose returned value this thread has stored before the
        // CTA's arrival, so it is performed before any CTA reserves again.
        if (T.rank == 0) sm.base = atomicExch(&S.bar->lcnt[p], 0u);
    }
    __syncthreads();
    list_round(sm, S, q, p);
}

}  // namespace abfs
