// Level-synchronous engine: a whole search.
// Part of sync_engine.cu, split by topic; included in order.
#pragma once

#include "sync_local.cuh"

namespace abfs {

// One trace entry (abfs_run_trace), written by the team's first thread.
__device__ __forceinline__ void sync_trace(const SyncSearch& S, const Team& T, uint32_t kind, uint32_t k,
                                           uint32_t alone, uint32_t items, uint32_t verts, uint32_t ent) {
    if (!S.trace || T.rank != 0 || threadIdx.x != 0) return;
    const uint32_t tn = ld_relaxed(&S.ctl->trace_n);
    if (tn >= S.trace_cap) return;
    const uint64_t now = globaltimer();
    S.trace[2 * tn] = make_uint4((uint32_t)now, (uint32_t)(now >> 32), (kind << 24) | (k & 0xFFFFFFu), alone);
    S.trace[2 * tn + 1] = make_uint4(items, verts, ent, 0u);
    st_relaxed(&S.ctl->trace_n, tn + 1);
}

// Clears the search's words, control block and (path counts) sums, and gives
// the source its key.  Whole team.
__device__ __forceinline__ void sync_init(const SyncSearch& S, const Team& T) {
    const uint32_t stride = T.size * kSyncThreads;
    const uint32_t t0 = T.rank * kSyncThreads + threadIdx.x;
    const bool slow = sync_long_pass(S, T);
    // two keys per 16-byte store
    ulonglong2* const k2 = reinterpret_cast<ulonglong2*>(S.key);
    for (uint32_t i = t0; i < S.n / 2; i += stride) {
        if (slow) red_add64(&S.bar->beat, 1ull);
        ulonglong2 x = make_ulonglong2(kKeyUnset, kKeyUnset);
        if (2 * i == S.src) x.x = S.src_label;
        if (2 * i + 1 == S.src) x.y = S.src_label;
        k2[i] = x;
    }
    if ((S.n & 1) && t0 == 0) S.key[S.n - 1] = S.n - 1 == S.src ? S.src_label : kKeyUnset;
    if (S.sigma)
        for (uint32_t v = t0; v < S.n; v += stride) {
            if (slow) red_add64(&S.bar->beat, 1ull);
            S.sigma[v] = v == S.src ? 1ull : 0ull;
        }
    if (T.rank == 0) {
        uint32_t* c = reinterpret_cast<uint32_t*>(S.ctl);
        for (uint32_t w = threadIdx.x; w < sizeof(InstCtl) / 4; w += kSyncThreads) c[w] = 0u;
    }
}

// The caller's level and parent of every vertex from the key words; on a
// relabelled graph, gathered in input order (vertices without edges of an
// undirected graph, from n_keep on, are known to be unreached).  Four vertices
// per thread and step, two steps in flight.  Whole team.
__device__ __noinline__ void sync_outputs(const SyncSearch& S, const Team& T) {
    const uint32_t stride = T.size * kSyncThreads;
    const uint32_t t0 = T.rank * kSyncThreads + threadIdx.x;
    const uint32_t quads = S.n / 4;
    const bool slow = sync_long_pass(S, T);
    const bool vec = ((reinterpret_cast<uintptr_t>(S.level) | reinterpret_cast<uintptr_t>(S.parent)) & 15u) == 0;
    auto key_at = [&](uint32_t o) -> unsigned long long {
        if (!S.pos) return ld_relaxed64(S.key + o);
        const uint32_t i = ld_ro(S.pos + o);
        return i < S.n_keep || i == S.src ? ld_relaxed64(S.key + i) : kKeyUnset;
    };
    auto put = [&](uint32_t q, const unsigned long long (&x)[4]) {
        const int4 lv = make_int4((int)(x[0] >> 32), (int)(x[1] >> 32), (int)(x[2] >> 32), (int)(x[3] >> 32));
        const uint4 pr = make_uint4((uint32_t)x[0], (uint32_t)x[1], (uint32_t)x[2], (uint32_t)x[3]);
        if (vec) {
            reinterpret_cast<int4*>(S.level)[q] = lv;
            reinterpret_cast<uint4*>(S.parent)[q] = pr;
        } else {
            int32_t* const l = S.level + 4ull * q;
            uint32_t* const p = S.parent + 4ull * q;
            l[0] = lv.x, l[1] = lv.y, l[2] = lv.z, l[3] = lv.w;
            p[0] = pr.x, p[1] = pr.y, p[2] = pr.z, p[3] = pr.w;
        }
    };
    for (uint32_t q = t0; q < quads; q += 2 * stride) {
        if (slow) red_add64(&S.bar->beat, 1ull);
        const bool two = q + stride < quads;
        unsigned long long a[4], b[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) a[x] = key_at(4 * q + x);
        if (two) {
#pragma unroll
            for (int x = 0; x < 4; ++x) b[x] = key_at(4 * (q + stride) + x);
        }
        put(q, a);
        if (two) put(q + stride, b);
    }
    for (uint32_t v = 4 * quads + t0; v < S.n; v += stride) {
        const unsigned long long x = key_at(v);
        S.level[v] = (int32_t)(x >> 32);
        S.parent[v] = (uint32_t)x;
    }
}

// The team's share of level 0's list: an even part of the source's column each,
// so that the rows it wins -- often hubs, on an R-MAT graph -- are spread over
// the CTAs from the start (they were one CTA's, and evened out before level 1).
__device__ __forceinline__ void sync_source(SyncSmem& sm, const SyncSearch& S, const Team& T,
                                            unsigned long long& items) {
    const uint32_t cb = ld_ro(S.colptr + S.src);
    const uint32_t len = ld_ro(S.colptr + S.src + 1) - cb;
    items = items_of(cb, len);
    // a column too long for the team's lists starts in the global list, in
    // items shared out evenly
    const bool global = items > (unsigned long long)T.size * (kThinCap - 1);
    uint32_t mine = 0;
    if (global) {
        const uint32_t ni = (uint32_t)items;  // (at most 2^24: 32 bits hold the products)
        for (uint32_t i = ni * T.rank / T.size + threadIdx.x; i < ni * (T.rank + 1) / T.size; i += kSyncThreads) {
            uint32_t b, l;
            item_at(cb, len, i, b, l);
            list_put(S, 0, i, S.src_label, b, l);
        }
    } else {
        const uint32_t per = (len + T.size - 1) / T.size;
        const uint32_t lo = min(len, per * T.rank), part = min(len - lo, per);
        mine = items_of(cb + lo, part);
        for (uint32_t i = threadIdx.x; i < mine; i += kSyncThreads) {
            uint32_t b, l;
            item_at(cb + lo, part, i, b, l);
            sm.ij[0][i] = S.src_label;
            sm.ib[0][i] = b;
            sm.il[0][i] = l;
        }
    }
    if (threadIdx.x == 0) {
        sm.step = sm.tick = 0;
        sm.left = 0;
        sm.word[0] = sm.word[1] = sm.aux[0] = sm.aux[1] = 0;
        sm.app[0][0] = mine;
        sm.app[0][1] = ~0u;  // entries: not known
        sm.app[1][0] = sm.app[1][1] = 0;
        sm.verts = sm.ent = 0;
        sm.lim = 1024;
        sm.ent_clamp = ((1u << kItemShift) - 1u) / T.size;
        sm.weight = (float)len + 4.f * (float)items + 1.f;
        sm.bu = 0;
        sm.nf = 1;
        sm.seen = sm.entries = len;
        sm.st_read = sm.st_unmasked = 0;
        sm.st_verts = T.rank == 0 ? 1 : 0;
        sm.st_ent = T.rank == 0 ? len : 0;
        sm.levels = 1;
    }
}

// A list's cost to its CTA, in entries: a claim each, and per item its append
// and look-up.  A list is heavy above what a CTA expands in about a microsecond
// and twice an even share of the next level if that grows as this one did
// (capped, so that a hub's list is noticed): evening the lists out costs 5 us.
// (Without the growth, ER 2^16 of degree 8 pays for it once more just before its
// largest level, when some lists pass the limit by chance: 52 -> 59 us.)
__device__ __forceinline__ uint32_t list_weight(uint32_t items, uint32_t ent) { return ent + 4 * items; }
__device__ __forceinline__ void heavy_limit(SyncSmem& sm, const Team& T, float items, float ent) {
    const float w = ent + 4.f * items;
    const float next = w * fminf(8.f, fmaxf(1.f, __fdividef(w, sm.weight)));
    sm.lim = 1024u + (uint32_t)__fdividef(2.f * next, (float)T.size);
    sm.weight = fmaxf(w, 1.f);
}
__device__ __forceinline__ uint32_t tot_items(unsigned long long tot) {
    return (uint32_t)(tot >> kItemShift) & ((1u << (kHeavyShift - kItemShift)) - 1u);
}
__device__ __forceinline__ uint32_t tot_ent(unsigned long long tot) {
    return ((uint32_t)tot & ((1u << kItemShift) - 1u)) * kEntUnit;
}

// Entries from which the level of a frontier of `items` items is wide.  A wide
// level costs a bitmap (8 bytes per vertex), an extraction and a barrier more
// than a thin one, about 10 us and a part in n, and saves a returned 64-bit
// atomic per entry, so the line grows with the team (a line fixed for the whole
// GPU: a batch of 32 graphs on teams of a few CTAs, 340 us instead of 317).  Those
// atomics queue where many columns share hub rows, which a frontier of columns
// well above the mean is a sign of (undirected graphs): R-MAT of scale 16, 1.2 M
// entries, 150 us with its hub levels thin, 75 us wide.  Without hubs thin levels
// stay ahead longer: ER of 150 000 vertices, degree 16, 82 us, 98 us with half
// the line.
constexpr uint32_t kWidePerCta = 10240, kHubPerCta = 1728, kRoundsPart = 4;
__device__ __forceinline__ uint32_t hub_line(const SyncSearch& S, const Team& T) {
    return kHubPerCta * T.size + S.n / 4;
}
__device__ __forceinline__ uint32_t wide_line(const SyncSearch& S, const Team& T, unsigned long long items,
                                              unsigned long long ent) {
    return ent >= S.hub_avg * items ? hub_line(S, T) : kWidePerCta * T.size + S.n;
}

// The line for a frontier whose items are counted exactly.  One that the lists do
// not hold takes rounds, each with its own chain, and pays for the spilled items:
// it stays thin only while its entries are few beside the vertices that a wide
// level passes over.  (The levels of meshes stay under n / 9.  A batch of 128 ER
// and R-MAT graphs on teams of a few CTAs, whose levels jump past the lists by a
// factor of the degree: 688 us with wide_line alone, 583 with n / 4, 593 with
// n / 8.)
__device__ __forceinline__ uint32_t list_line(const SyncSearch& S, const Team& T, unsigned long long items,
                                              unsigned long long ent) {
    const uint32_t line = wide_line(S, T, items, ent);
    return items > (unsigned long long)T.size * kThinCap ? min(line, S.n / kRoundsPart) : line;
}

// Thread 0 after the barrier that ended a thin level (tot: the barrier's
// totals): the next level's kind.  The first tests are the usual case.
__device__ __forceinline__ uint32_t thin_next(SyncSmem& sm, const SyncSearch& S, const Team& T,
                                              unsigned long long tot, unsigned long long aux, bool want_aux) {
    const uint32_t flags = (uint32_t)(tot >> kHeavyShift);
    const uint32_t items = tot_items(tot), ent = tot_ent(tot);
    sm.items = items;
    if (items == 0) return kActDone;
    if (flags == 0 && ent < hub_line(S, T) && !want_aux) return kActThin;
    if (tot == ~0ull) return kActFailed;
    if (want_aux) {
        sm.nf = items;
        sm.entries = aux;
        sm.seen += aux;
        if (S.bu_alpha) {
            const unsigned long long mu = S.nnz > sm.seen ? S.nnz - sm.seen : 0ull;
            sm.bu = aux * S.bu_alpha > mu;
            if (sm.bu) return kActBottomUp;
        }
    }
    if (ent >= wide_line(S, T, items, ent)) return kActWide;
    // a list is full, or a few CTAs hold much more than the others
    const uint32_t heavy = flags & 0xFFu;
    if ((flags >> 8) || (heavy && 2 * heavy <= T.size)) {
        heavy_limit(sm, T, (float)items, (float)ent);
        return kActEven;
    }
    return kActThin;
}

// Runs thin levels from level k on until another kind of level follows
// (sm.act); returns that level's number.  A function of its own, so that the
// loop that long searches spend their time in has its own registers.
//
// The first level may take several rounds, where the lists do not hold it
// (list_slice).  As a wide level it would cost, besides its entries, something
// for every unvisited vertex, which a mesh of 10^8 vertices pays hundreds of
// times and a small team on a small mesh all the same; in rounds the cost follows
// the frontier (464^3: 98 -> 30 ms, on the unit scheduler 42; 152 searches of
// 64^3 in a batch 13.9 -> 5.8 ms).  The test costs a thin level 2 %; rounds in a
// function of their own cost the others their registers (R-MAT-20 182 -> 190 us).
// Whole CTA.
template <bool SIG>
__device__ __noinline__ uint32_t thin_run(SyncSmem& sm, const SyncSearch& S, const Team& team, uint32_t k) {
    const Team T = team;
    // the barrier and the decision fall to the warp that has work of its own
    // only when all of them have
    const bool lead = threadIdx.x == kSyncThreads - 32;
    const bool want_aux = S.bu_alpha != 0 || S.trace != nullptr;
    SyncTally t;
    ThinStage st;
    uint32_t act = kActThin;
    bool staged = false;
    __syncthreads();
    do {
        if (!staged) thin_stage(sm, S, k & 1, st);
        if (S.trace) sync_trace(S, T, kPhLevel, k, 4u, (uint32_t)sm.items, (uint32_t)sm.nf, (uint32_t)sm.entries);
        thin_claims<SIG>(sm, S, k, st, t);
        const bool more = sm.left != 0;
        __syncthreads();
        if (more) {
            list_round(sm, S, k & 1, k & 1);
            staged = false;
            continue;
        }
        const uint32_t cur = k & 1;
        unsigned long long add = 0, aux = 0;
        if (lead) {
            const uint32_t c = sm.app[cur ^ 1][0], e = sm.app[cur ^ 1][1];
            add = (unsigned long long)min(c, kItemClamp) << kItemShift | min(e / kEntUnit, sm.ent_clamp);
            if (list_weight(c, e) > sm.lim) add += 1ull << kHeavyShift;
            if (c > kThinCap) add += 1ull << kFullShift;
            aux = e;
            if (SIG || want_aux) bar_arrive<true>(sm, S, T, add, aux);
            else bar_arrive<false>(sm, S, T, add, aux);
            sm.app[cur][0] = sm.app[cur][1] = 0;
            sm.st_ent += e;
        }
        __syncwarp();
        staged = sm.app[cur ^ 1][1] <= kThinAhead;
        if (staged) thin_stage(sm, S, cur ^ 1, st);
        unsigned long long tot = 0;
        if (lead) {
            tot = SIG || want_aux ? bar_poll<true>(sm, S, T, add, aux) : bar_poll<false>(sm, S, T, add, aux);
            sm.act = thin_next(sm, S, T, tot, aux, want_aux);
        }
        __syncthreads();
        ++k;
        act = sm.act;
        if (lead && act == kActThin) heavy_limit(sm, T, (float)tot_items(tot), (float)tot_ent(tot));
    } while (act == kActThin);
    tally_add(sm, t.read, t.unmasked);
    t.verts = __reduce_add_sync(0xFFFFFFFFu, t.verts);
    t.levels = __reduce_max_sync(0xFFFFFFFFu, t.levels);
    if ((threadIdx.x & 31) == 0 && t.verts) {
        atomicAdd(&sm.st_verts, (unsigned long long)t.verts);
        atomicMax(&sm.levels, t.levels);
    }
    __syncthreads();
    return k;
}

// Thread 0 after the barrier that ended a wide or a bottom-up level.
__device__ __forceinline__ uint32_t wide_next(SyncSmem& sm, const SyncSearch& S, const Team& T, bool bottom_up,
                                              unsigned long long tot, unsigned long long aux) {
    if (tot == ~0ull) return kActFailed;
    sm.items = tot;
    sm.nf = aux >> kAuxShift;
    sm.entries = aux & ((1ull << kAuxShift) - 1);
    sm.seen += sm.entries;
    if (bottom_up ? sm.nf == 0 : tot == 0) return kActDone;
    if (S.bu_alpha) {
        // the direction, as the unit scheduler chooses it (decide_next)
        const unsigned long long mu = S.nnz > sm.seen ? S.nnz - sm.seen : 0ull;
        sm.bu = sm.bu ? sm.nf * S.bu_beta >= S.n : sm.entries * S.bu_alpha > mu;
        if (sm.bu) return kActBottomUp;
    }
    if (bottom_up || sm.entries >= list_line(S, T, tot, sm.entries) / 2) return kActWide;
    heavy_limit(sm, T, (float)tot, (float)sm.entries);
    return kActSlice;
}

// Thread 0 of a CTA that is done with a search: the last one to leave sets the
// status, clears the barrier's words for the next search and returns true.
__device__ __forceinline__ bool sync_leave(const SyncSearch& S, const Team& T) {
    __threadfence();
    if (atomicInc(&S.bar->exited, T.size - 1) != T.size - 1) return false;
    __threadfence();
    for (int b = 0; b < 2; ++b) {
        S.bar->word[b] = S.bar->aux[b] = 0;
        S.bar->lcnt[b] = 0;
    }
    const uint32_t err = ld_relaxed(&S.bar->err);
    S.bar->err = 0;
    S.ctl->err = err;
    S.ctl->status = err ? kFailed : kDone;
    return true;
}

// Runs one search on this team.  The outputs and the control block are written
// when it returns (to be read after the kernel).
//
// Thin levels hold while the frontier's entries stay below wide_line; wide levels
// until they are fewer than half of that (each thin -> wide switch rebuilds the
// bitmap, 8 bytes per vertex).
// After a barrier thread 0 alone decides what follows: the same decision made
// by every thread took 1.3 us a level on 32 warps.
// Returns, in thread 0, whether this CTA was the last to leave.
template <bool SIG>
__device__ __forceinline__ bool sync_search(SyncSmem& sm, const SyncSearch& S, const Team& T) {
    const bool lead = threadIdx.x == 0;
    if (!SIG && S.local && T.expect == 1) {
        local_search(sm, S);
        return lead && sync_leave(S, T);
    }
    unsigned long long items;
    uint32_t k = 0, wide_levels = 0, act = kActThin;
    sync_init(S, T);
    sync_source(sm, S, T, items);
    if (!team_sync(sm, S, T)) act = kActFailed;
    else if (items == 0) act = kActDone;
    else if (items > (unsigned long long)T.size * (kThinCap - 1)) {
        sync_bitmaps(S, T, 0);
        act = team_sync(sm, S, T) ? kActWide : kActFailed;
        if (lead) sm.items = items;
        __syncthreads();
    }
    sync_trace(S, T, 0xFEu, 0, 0, 0, 1, 0);
    while (act < kActDone) {
        if (act == kActThin) {
            k = thin_run<SIG>(sm, S, T, k);
            act = sm.act;
            const uint32_t p = k & 1;
            if (act == kActEven || act == kActWide) {
                const uint32_t mine = sm.app[p][0], ent = sm.app[p][1];
                list_dump(sm, S, p, p);
                if (act == kActWide) sync_bitmaps(S, T, k);
                if (!team_sync(sm, S, T, mine, ent)) {
                    act = kActFailed;
                } else if (act == kActEven) {
                    // exact totals now: the thin level's were clamped per CTA
                    const unsigned long long all = sm.items, entries = sm.entries;
                    if (entries < list_line(S, T, all, entries)) {
                        list_slice(sm, S, T, p, p, all);
                        // a failed append leaves the list incomplete
                        if (lead) sm.act = ld_relaxed(&S.bar->err) ? kActFailed : kActThin;
                        __syncthreads();
                        act = sm.act;
                    } else {
                        sync_bitmaps(S, T, k);
                        act = team_sync(sm, S, T) ? kActWide : kActFailed;
                        if (lead) {
                            sm.items = all;
                            sm.entries = entries;
                        }
                        __syncthreads();
                    }
                }
            } else if (act == kActBottomUp) {
                sync_trace(S, T, kPhBuPrep, k, 0u, 0u, 0u, 0u);
                sync_bitmaps(S, T, k);
                if (lead) {
                    sm.app[p][0] = sm.app[p][1] = 0;
                    if (T.rank == 0) st_relaxed(&S.bar->lcnt[p], 0u);
                }
                if (!team_sync(sm, S, T)) act = kActFailed;
            }
        } else if (act == kActSlice) {
            list_slice(sm, S, T, k & 1, k & 1, sm.items);
            act = kActThin;
        } else {
            const bool up = act == kActBottomUp;
            // read by nobody any more, and used again at the next level
            if (T.rank == 0 && lead) st_relaxed(&S.bar->lcnt[k & 1], 0u);
            if (S.trace)
                sync_trace(S, T, up ? kPhBottomUp : kPhLevelScan, k, 0u, (uint32_t)sm.items, (uint32_t)sm.nf,
                           (uint32_t)sm.entries);
            ++wide_levels;
            if (up) {
                sync_bottom_up(sm, S, T, k);
            } else {
                constexpr int kind = SIG ? kWideCounts : kWidePlain;
                if (S.n <= kBitsN) wide_expand<kind, true>(sm, S, T, k, sm.items);
                else wide_expand<kind, false>(sm, S, T, k, sm.items);
                if (!team_sync(sm, S, T)) {
                    act = kActFailed;
                    break;
                }
                sync_trace(S, T, kPhExtract, k, 0u, 0u, 0u, 0u);
                sync_extract<kFromKeys>(sm, S, T, k);
            }
            __syncthreads();
            if (lead) {
                const uint32_t c = sm.app[0][0], v = sm.verts, e = sm.ent;
                sm.app[0][0] = 0;
                sm.verts = sm.ent = sm.tick = 0;
                if (v) sm.levels = k + 2;
                sm.st_verts += v;
                sm.st_ent += e;
                unsigned long long aux = (unsigned long long)v << kAuxShift | e;
                const unsigned long long tot = bar_wait<true>(sm, S, T, c, aux);
                sm.act = wide_next(sm, S, T, up, tot, aux);
                // a failed append leaves a list incomplete: nothing reads it
                if (sm.act < kActDone && T.expect == 1 && ld_relaxed(&S.bar->err)) sm.act = kActFailed;
            }
            __syncthreads();
            ++k;
            act = sm.act;
            if (up && act == kActWide) {
                // back to top-down levels: the list of the frontier bitmap
                sync_extract<kFromBits>(sm, S, T, k - 1);
                __syncthreads();
                const uint32_t c = sm.app[0][0];
                if (!team_sync(sm, S, T, c)) act = kActFailed;
                else if (sm.items == 0) act = kActDone;
                if (lead) sm.app[0][0] = 0;
                __syncthreads();
            }
        }
    }
    sync_trace(S, T, 0xFFu, k, 0u, 0u, 0u, 0u);
    if (act == kActDone) sync_outputs(S, T);
    __syncthreads();
    if (lead) {
        InstCtl* c = S.ctl;
        if (sm.st_read) atomicAdd(&c->entries_read, sm.st_read);
        if (sm.st_unmasked) {
            atomicAdd(&c->entries_unmasked, sm.st_unmasked);
            atomicAdd(&c->claims, sm.st_unmasked);
        }
        if (sm.st_ent) atomicAdd(&c->nnz_reached, sm.st_ent);
        if (sm.st_verts) atomicAdd(&c->reached, (uint32_t)sm.st_verts);
        atomicMax(&c->levels, sm.levels);
        if (T.rank == 0 && wide_levels) atomicAdd(&c->wide_levels, wide_levels);
        return sync_leave(S, T);
    }
    return false;
}

}  // namespace abfs
