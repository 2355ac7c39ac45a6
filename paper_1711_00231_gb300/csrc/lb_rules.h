// Rules of the query loops that are plain arithmetic: shared by the host, the
// whole-query kernel and the serving kernel, and compiled alone by the tests.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define LB_HD __host__ __device__
#else
#define LB_HD
#endif

namespace lbk {

// Worklist iterations an SSSP with a distance threshold may take: those of an
// interval add up to at most its vertices and one more.  n < 2^31.
LB_HD inline uint32_t threshold_levels(int64_t n) {
    const uint64_t k = 2u * (uint64_t)n + 66u;
    return k < 0xFFFFFFF0ull ? (uint32_t)k : 0xFFFFFFF0u;
}

// How a query goes on when the next iteration would be number `level`: it has
// a list, or a pull of far vertices is due, or neither.  Work left at the cap
// is an error, whichever kind it is.
enum : int { kGoesOn = 0, kIsDone = 1, kIsCut = 2 };
LB_HD inline int level_end(bool list, bool pull, uint32_t level, uint32_t cap) {
    if (!list && !pull) return kIsDone;
    return level <= cap ? kGoesOn : kIsCut;
}

// Iterations so far, after a list of `entries` entries.
LB_HD inline uint32_t level_after(uint32_t level, uint32_t entries) { return level + (entries > 0u ? 1u : 0u); }

// Serving: whether a list of E edges, the last of `lists` lists with `edges`
// edges, is one of a growing front.  After its largest lists a random graph's
// query has a tail of short ones that a distance threshold only lengthens:
// lone SSSP on 2^20 vertices and 2^21 edges 2.09 ms with it, 1.36 without.
LB_HD inline bool front_grows(uint64_t E, uint32_t lists, uint64_t edges) { return E * lists >= edges; }

}  // namespace lbk
