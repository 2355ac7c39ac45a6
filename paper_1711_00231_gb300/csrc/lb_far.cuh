// The far set of an SSSP with a distance threshold (described in
// lb_query_wd.cu): the parts the whole-query kernel and the serving kernel
// share.
#pragma once

#include "lb_device.cuh"

namespace lbk {

constexpr uint32_t kFarMaxDelta = 1u << 30;

// T + delta, or "no threshold" when that passes the largest distance.
__device__ __forceinline__ uint32_t far_add(uint32_t t, uint32_t delta) {
    const uint64_t x = (uint64_t)t + delta;
    return x >= kSat ? kInf : (uint32_t)x;
}

// Loop state of a CTA.  `u` is the same in every CTA of a step: each of them
// updates it from the step's published counts alone.
struct QueryState {
    QueryLoop u;
    FarSet far;  // far.T == u.T
    uint32_t ok, rank;            // rank: this CTA in the team (kNoRank: outside); 0 leads
    uint32_t full, team, resume;  // barriers and publications so far
    uint32_t grid_steps, team_steps;  // regular steps of the whole grid / of the team so far
    uint32_t fmin;                // a pull's smallest distance left
    uint32_t maxdeg;              // largest degree this CTA listed in the level
    uint32_t trace;               // leader: records written
    uint64_t deadline, t0, pushes;
    // fast levels: exchanges and conversions so far, what the last exchange
    // said, the segments' first positions, this CTA's pushes of the level
    uint32_t fast_epoch, fast_conv, fast_n, fast_e, fast_maxdeg, fast_late;
    uint32_t fast_pre[kFastTeam + 1];
    uint32_t out_n, out_e, out_maxdeg;
};

// Calls take(v, d) for 32 consecutive vertices at a time of this warp's
// share of the far set's blocks, with d their distances (kInf past the end),
// and clears the bits of the blocks in which no lane's keep(d) held.  A lane
// holds one word of the bitmap (one load for up to 1024 blocks per warp),
// and eight blocks' distances are in flight at once: a wave on a grid sets
// one bit in each of thousands of words.
template <class Take, class Keep>
__device__ __forceinline__ void far_blocks(const uint32_t *status, int64_t n, const FarSet &far, uint32_t me,
                                           uint32_t ctas, bool clear, Take take, Keep keep) {
    constexpr int kB = 8;
    const uint32_t lane = lane_id();
    const uint32_t words = (uint32_t)(((n - 1) >> far.shift) >> 5) + 1u;
    const uint32_t warps = ctas * kWarps;
    const int32_t chunks = 1 << (far.shift - 5);  // of 32 vertices per block
    for (uint32_t w0 = me + ctas * (threadIdx.x >> 5); w0 < words; w0 += 32u * warps) {  // warp-uniform
        uint32_t my = w0 + lane * warps < words ? __ldcg(far.bits + w0 + lane * warps) : 0u;
        unsigned nz = __ballot_sync(kFull, my != 0u);
        while (nz) {
            uint32_t blk[kB], left = 0u;  // block numbers (kInf: none), bit r: block r keeps its bit
#pragma unroll
            for (int r = 0; r < kB; ++r) {
                blk[r] = kInf;
                if (nz) {  // warp-uniform
                    const int l = __ffs(nz) - 1;
                    const int b = __ffs(__shfl_sync(kFull, my, l)) - 1;
                    blk[r] = (w0 + (uint32_t)l * warps) * 32u + (uint32_t)b;
                    if ((int)lane == l) my &= my - 1u;
                    nz = __ballot_sync(kFull, my != 0u);
                }
            }
            for (int32_t c = 0; c < chunks; ++c) {
                uint32_t d[kB];
#pragma unroll
                for (int r = 0; r < kB; ++r) {
                    const int64_t v = ((int64_t)blk[r] << far.shift) + 32 * c + lane;
                    d[r] = blk[r] != kInf && v < n ? __ldcg(status + v) : kInf;
                }
#pragma unroll
                for (int r = 0; r < kB; ++r) {
                    if (__any_sync(kFull, keep(d[r]))) left |= 1u << r;
                    take((int32_t)(((int64_t)blk[r] << far.shift) + 32 * c + lane), d[r]);
                }
            }
            if (clear && lane == 0)
#pragma unroll
                for (int r = 0; r < kB; ++r)
                    if (blk[r] != kInf && !((left >> r) & 1u)) atomicAnd(far.bits + (blk[r] >> 5), ~(1u << (blk[r] & 31u)));
        }
    }
}

}  // namespace lbk
