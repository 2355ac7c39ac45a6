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

// Serving: width of the next interval of an SSSP with a distance threshold,
// after one whose `lists` lists (> 0) had `edges` edges and whose pull cost
// `reads` reads of 32 distances by one warp.  Intervals widen
//   while their lists average fewer than list / 8 edges (list: the longest
//   list one CTA takes),
//   while they have fewer than `least` edges, and
//   while the pull costs as much as the lists: the CTA reads about 64 x 32
//   distances in a microsecond and takes 4 to 12 us for a list, so beyond a
//   few hundred reads per list.  A far set that a few heavy edges spread over
//   the graph keeps thousands of blocks alive, and its intervals stayed eight
//   lists long: lone SSSP on a 1024^2 grid with weights 1 and 1% of 10^6,
//   kPullReads 256 / 512 / 1024 / 2048 / without: 15.2 / 15.0 / 15.1-18.5 /
//   18.4-21 / 42 ms (without a threshold 26.2); 64 mixed queries 12.8 / 12.7 /
//   12.6 / 11.9 / 12.1 ms, hence 2048.
// They narrow while lists average over list / 2 edges and neither of the
// other two would soon widen them again.
constexpr uint64_t kPullReads = 2048;
LB_HD inline uint32_t next_width(uint32_t delta, uint64_t reads, uint32_t lists, uint64_t edges, uint64_t least,
                                 uint32_t list, uint32_t max_delta) {
    const uint64_t avg = edges / lists, costly = kPullReads * lists;
    if (edges < least || reads > costly || avg < list / 8u) return delta < max_delta ? delta * 2u : delta;
    if (avg > list / 2u && edges > 4u * least && 4u * reads < costly) return delta / 2u > 1u ? delta / 2u : 1u;
    return delta;
}

}  // namespace lbk
