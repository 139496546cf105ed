// Serving on the level-synchronous engine: how the CTAs that come free agree on
// the team of a query.  The protocol is one word per slot; it is written over a
// policy of word accesses, so that it also runs on the host.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define ABFS_TEAM_FN __device__ __forceinline__
#else
#define ABFS_TEAM_FN inline
#endif

namespace abfs {

// The word: [sequence : 32][open : 1 at bit 16][wanted : 8][joined : 8].  A CTA
// joins by a compare-and-swap that adds 1 to an open word with room; its rank is
// the count before.
constexpr unsigned long long kJoinOpen = 1ull << 16;
ABFS_TEAM_FN uint32_t join_count(unsigned long long w) { return (uint32_t)w & 0xFFu; }
ABFS_TEAM_FN uint32_t join_wanted(unsigned long long w) { return (uint32_t)(w >> 8) & 0xFFu; }
ABFS_TEAM_FN bool join_room(unsigned long long w) { return (w & kJoinOpen) && join_count(w) < join_wanted(w); }
// The word of a team just opened by its leader (rank 0) for `size` CTAs.
ABFS_TEAM_FN unsigned long long join_opened(unsigned long long before, uint32_t size) {
    return ((before >> 32) + 1) << 32 | kJoinOpen | (unsigned long long)size << 8 | 1ull;
}

// One thread of a CTA that has opened or joined a team: waits until the team is
// closed and returns its size, the same in every CTA of the team.  The leader
// closes it when it is full or after wait_ns, but while fewer than half of the
// wanted CTAs have joined not before few_ns divided by their number.  A member whose own, much longer
// wait runs out (the leader was not running meanwhile) closes it itself: the
// size is the count in the word at the moment it was closed, whoever did that,
// since nobody joins a closed team.  The word is not reused before this CTA
// has left the search.
template <class Io>
ABFS_TEAM_FN uint32_t team_form(Io& io, bool leader, unsigned long long wait_ns, unsigned long long few_ns = 0) {
    const unsigned long long t0 = io.now();
    for (;;) {
        const unsigned long long w = io.load();
        if (!(w & kJoinOpen)) return join_count(w);
        unsigned long long limit = wait_ns;
        if (leader && 2 * join_count(w) < join_wanted(w) && few_ns / join_count(w) > limit)
            limit = few_ns / join_count(w);
        if ((leader && !join_room(w)) || io.now() - t0 > limit) return join_count(io.close());
    }
}

}  // namespace abfs
