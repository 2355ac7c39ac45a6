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

}  // namespace lbk
