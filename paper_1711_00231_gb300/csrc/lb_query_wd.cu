// A whole WD query (workload decomposition, Sec. III-A) in one cooperative
// launch: set-up, every worklist iteration and the overflow check.
//
// What bounds it: on small and high-diameter graphs nothing but the chain
// of iterations, so what a level costs beyond its edges is what counts.  A
// launch per level inside a CUDA-graph WHILE node cost 14-16 us for a list
// of one edge (kernel drain, last-CTA finalisation, condition, relaunch),
// beside the set-up and check launches of every query.  Here the grid stays
// resident and a level ends with one grid barrier; every CTA then reads the
// output list's packed size and goes on by itself.
//
// Levels with lists of at most small_edges edges run on a team of CTAs with
// a barrier of its own, while the others wait (with sleeps) for the team to
// publish that a list has grown or the query has ended: a barrier over the
// whole grid costs more than such a level's work.
//
// Worklists are read with plain loads (kLdPlain): a barrier's acquire drops
// the SM's L1 lines, so a level sees everything earlier levels wrote, and
// the L1 still caches the visited bits and distances within a level, as in
// a launch of its own.
//
// SSSP takes a distance threshold once its lists get long: see "far set".
#include "lb_far.cuh"
#include "lb_launch.h"
#include "lb_steps.cuh"

namespace lbk {

// Resident CTAs per SM (the register budget).  BFS runs at 5 (48 registers):
// at 6 (40) the loop state beside the walk spills.  Measured, 6 / 5 / 4 CTAs:
// R-MAT scale 20 BFS 141.9 / 129.8 / 127.3 us, scale 24 1754 / 1681 / 1798 us;
// SSSP at 4 / 5 CTAs, scale 24: 5.61 / 5.95 ms.
#ifndef LB_QUERY_MIN_BLOCKS
#define LB_QUERY_MIN_BLOCKS 5
#endif
#ifndef LB_QUERY_MIN_BLOCKS_SSSP
#define LB_QUERY_MIN_BLOCKS_SSSP LB_WD_MIN_BLOCKS_SSSP
#endif

constexpr uint32_t kResumeAbort = 0xFFFFFFFFu;
// A CTA waits this long for the whole grid or the team at a barrier, then
// records kErrDeadline and leaves: every wait ends.
constexpr uint64_t kQueryBarrierNs = 2000000000ull;

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t add_acq_rel(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Waits until *p - want >= 0 (wrapping); false when `limit` ns have passed
// or *p became kResumeAbort.  `idle`: sleep between the polls, an eighth of
// the time waited so far (0.2 to 8 us), for the CTAs outside a long-running
// team.
__device__ __forceinline__ bool wait_for(const uint32_t *p, uint32_t want, uint64_t limit, bool idle) {
    if ((int32_t)(ld_acquire(p) - want) >= 0) return true;
    const uint64_t t0 = global_ns();
    for (;;) {
        const uint32_t v = ld_acquire(p);
        if (v == kResumeAbort) return false;
        if ((int32_t)(v - want) >= 0) return true;
        const uint64_t t = global_ns() - t0;
        if (t > limit) return false;
        if (idle) __nanosleep(t < 1600u ? 200u : t > 64000u ? 8000u : (uint32_t)t / 8u);
    }
}

// One thread's arrival at a barrier of `size` CTAs; `round` counts the
// barriers of this kind so far (this one included).  The whole grid waits
// on a word of its own, released by the last arrival, so that the pollers
// do not hold up the arrivals; the team waits on the arrival count itself,
// one hop less.
__device__ __forceinline__ bool arrive_full(QuerySync *s, uint32_t size, uint32_t round) {
    fence_acq_rel();
    const uint32_t old = add_acq_rel(&s->full_arrive, 1u);
    if (old + 1u == size * round) {
        st_release(&s->full_release, round);
        return true;
    }
    return wait_for(&s->full_release, round, kQueryBarrierNs, false);
}
__device__ __forceinline__ bool arrive_team(QuerySync *s, uint32_t size, uint32_t round) {
    fence_acq_rel();
    const uint32_t old = add_acq_rel(&s->team_arrive, 1u);
    if (old + 1u == size * round) return true;
    return wait_for(&s->team_arrive, size * round, kQueryBarrierNs, false);
}

// ---- SSSP: the far set -----------------------------------------------------
// Relaxing every improved vertex in the next iteration (Bellman-Ford order)
// relaxes an edge again each time its source improves: 203 times on a
// 4096^2 grid, 3 times on a uniform random graph.  Once a query shows that
// shape (below) a threshold T holds back the rest: a vertex improved to a
// distance >= T is not queued, and when the list runs empty T moves up by
// delta and the vertices in [old T, new T) are pulled.
//
// The far set needs no list: every reached vertex below T has been expanded
// with its final distance when the list is empty, so the vertices waiting
// are exactly those at T or above.  A bit per block of 2^far_shift (32 up to 2^24)
// vertices, set when one is held back, keeps a pull from scanning all
// distances: it reads the blocks with a set bit, queues what lies below the
// new T, and clears the bits of blocks with nothing left.
//
// When: Bellman-Ford order is the faster one while a list's work is hidden
// by the iteration's latency, and on skewed low-diameter graphs, whose few
// iterations relax most edges once or twice (an extra pull and a longer
// chain of iterations cost more).  So T is set at the first list of at
// least kFarEdges edges that comes after kFarLevels iterations with fewer
// than a quarter of the graph's edges listed so far, or after kFarLate
// iterations.  delta starts at 32 * mean weight / mean degree and doubles
// (halves) after an interval whose lists averaged fewer than kFarLow (more
// than kFarHigh) edges.
//
// Measured: 4096^2 grid 334 -> 96 ms (list edges 203 -> 8 per edge), with
// the fast levels below 53 ms; uniform graph of 8.4M vertices and 33.5M edges
// 2.93 -> 1.6 ms (3.0 -> 1.3).  First width 8 / 16 / 32 / 64 * weight / degree:
// uniform graph 2.14 / 1.73 / 1.67 / 3.17 ms.  kFarHigh 131072 / 65536 / 32768
// / 24576: grid 75.4 / 65.8 / 62.4 / 62.5 ms.  On R-MAT
// graphs no width pays (a model of scale 21: 1.58 -> 1.42 relaxations per
// edge for 3 times the iterations), and the rule never sets T there.
#ifndef LB_FAR_EDGES
#define LB_FAR_EDGES 16384
#endif
#ifndef LB_FAR_MULT
#define LB_FAR_MULT 32
#endif
#ifndef LB_FAR_LOW
#define LB_FAR_LOW 4096
#endif
#ifndef LB_FAR_HIGH
#define LB_FAR_HIGH 32768
#endif
#ifndef LB_FAR_MINDIV
#define LB_FAR_MINDIV 4
#endif
constexpr uint32_t kFarEdges = LB_FAR_EDGES;
constexpr uint32_t kFarLevels = 6, kFarLate = 32;
constexpr uint64_t kFarLow = LB_FAR_LOW, kFarHigh = LB_FAR_HIGH;

// Thread 0, the same in every CTA: whether a list of E edges (iteration
// u.iters) makes the threshold rule above hold.
__device__ __forceinline__ void far_engage(QueryState &q, uint32_t E, int64_t m) {
    ++q.u.int_lists;
    q.u.int_edges += E;
    q.u.int_max = max(q.u.int_max, E);
    if (q.u.engaged || E < kFarEdges) return;
    if (!((q.u.iters >= kFarLevels && q.u.relaxed + E < (uint64_t)m / 4) || q.u.iters >= kFarLate)) return;
    q.u.engaged = 1u;
    q.u.T = q.far.T = far_add(0u, q.u.delta);
    q.u.int_lists = q.u.int_max = 0u;
    q.u.int_edges = 0ull;
}

// Thread 0, the same in every CTA: the next step pulls [u.T, from + delta).
// u.edges becomes the size of list to expect (whether the team runs it), and
// the interval's lists decide the next width.
__device__ __forceinline__ void far_start_pull(QueryState &q, uint32_t from) {
    q.u.done = 0u;
    q.u.pull = 1u;
    q.u.T0 = q.u.T;
    q.u.T = q.far.T = far_add(from, q.u.delta);
    q.u.edges = q.u.int_max;
    if (q.u.int_lists > 0u) {
        const uint64_t avg = q.u.int_edges / q.u.int_lists;
        if (avg < kFarLow && q.u.delta < kFarMaxDelta) q.u.delta *= 2u;
        if (avg > kFarHigh) q.u.delta = max(q.u.delta / 2u, q.u.delta_min);
    }
    q.u.int_lists = q.u.int_max = 0u;
    q.u.int_edges = 0ull;
}

// One pull: queues the vertices of the far set in [T0, T1), clears the bits
// of the blocks that hold no vertex at T1 or above, and lowers *fmin (shared
// memory) to the smallest of those that are left.  Nothing sets bits
// meanwhile.
template <class WB, class WS, class FO>
__device__ __forceinline__ void far_pull(const uint32_t *status, int64_t n, const FarSet &far, uint32_t T0,
                                         uint32_t T1, uint32_t me, uint32_t ctas, uint32_t *fmin, WB &wb, WS &ws,
                                         uint32_t &cnt, const FO &o) {
    uint32_t mn = kInf;
    far_blocks(
        status, n, far, me, ctas, true,
        [&](int32_t v, uint32_t d) {
            const bool want = d >= T0 && d < T1;  // kInf is never below T1
            if (__any_sync(kFull, want)) {
                wpush(wb, cnt, want, v, 0, 0u);
                if (cnt > (uint32_t)(WB::kCap - 32)) wflush<kOutNode, true>(wb, ws, cnt, o);
            }
        },
        [&](uint32_t d) {
            const bool k = d != kInf && d >= T1;
            if (k) mn = min(mn, d);
            return k;
        });
    wflush<kOutNode, true>(wb, ws, cnt, o);
    mn = __reduce_min_sync(kFull, mn);
    if (lane_id() == 0 && mn != kInf) atomicMin(fmin, mn);
}

// Picks the SMs of the small-list team, once per workspace.  The L2 is in two
// halves, each by one die's SMs, and what another SM has just written costs
// an SM of the other half 600-690 cycles instead of 260-330 (a dependent
// atomic; a line that stays unwritten is read in 230-310 from either).  A
// fast level's exchange waits for the slowest CTA's word to reach the
// slowest reader, so the team is the kFastTeam SMs nearest to the words:
// every CTA times atomics on them, and the last one ranks the SMs.
// Teams from both halves: 3.4 us per level of the 1000 x 1537 grid's BFS, and
// 7.0 to 8.9 ms per query by where the words lay.
__global__ void __launch_bounds__(kBlock) k_team_pick(Ctl *ctl) {
    __shared__ alignas(16) uint32_t s_lat[kMaxSms];
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        uint32_t sm, best = kNoRank;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
        // CTAs spread over the words: queueing at one would hide the distance
        unsigned long long *const w = fast_words(ctl) + (blockIdx.x * 5u) % (2u * kFastTeam);
        for (int r = 0; r < 3; ++r) {
            unsigned long long x = 0ull;
            const long long t0 = clock64();
#pragma unroll 1
            for (int k = 0; k < 6; ++k) x = atomicAdd(w + x, 0ull);  // the words are zero: a dependent chain
            const long long t1 = clock64() + (long long)x;
            best = min(best, (uint32_t)(t1 - t0));
        }
        if (sm < kMaxSms) ctl->sm_rank[sm] = best;  // zero: no CTA ran there
        __threadfence();
        s_last = atomicAdd(&ctl->team_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (uint32_t k = threadIdx.x; k < kMaxSms; k += kBlock) {
        const uint32_t l = __ldcg(&ctl->sm_rank[k]);
        s_lat[k] = l ? min(l, kNoRank >> 10) << 9 | k : kNoRank;  // ordered by latency, then SM
    }
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < kMaxSms; k += kBlock) {
        const uint32_t mine = s_lat[k];
        uint32_t rank = 0;
        for (uint32_t j = 0; j < kMaxSms / 4; ++j) {
            const uint4 x = reinterpret_cast<const uint4 *>(s_lat)[j];
            rank += (x.x < mine) + (x.y < mine) + (x.z < mine) + (x.w < mine);
        }
        ctl->sm_rank[k] = mine != kNoRank && rank < (uint32_t)kFastTeam ? rank : kNoRank;
    }
}

cudaError_t launch_team_pick(Ctl *ctl, int sms, cudaStream_t st) {
    // one CTA per SM (shared memory)
    constexpr int kSmem = 160 * 1024;
    cudaError_t e = cudaFuncSetAttribute(k_team_pick, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    k_team_pick<<<sms, kBlock, kSmem, st>>>(ctl);
    return cudaGetLastError();
}

// The counters of this step (ahead 0) or of the next one of its kind (1).
__device__ __forceinline__ QuerySync::Step *step_counters(QuerySync *sync, const QueryState &q, bool team, uint32_t ahead) {
    return team ? sync->team_step + (q.team_steps + ahead) % 3u : sync->grid_step + (q.grid_steps + ahead) % 3u;
}

// The leader's thread 0: the state the CTAs outside the team go on from.
__device__ __forceinline__ void publish(QuerySync *sync, QueryState &q) {
    sync->loop = q.u;
    st_release(&sync->resume, ++q.resume);
}

// ---- fast levels -------------------------------------------------------------
// A high-diameter graph spends thousands of levels on lists of a few
// thousand short entries, and such a level is a chain of dependent L2 and
// DRAM trips of 0.6-0.9 us each, whatever its size.  The walk's chain has
// about eleven (tile start, list window, columns, check, claim, offsets,
// list reservation, fence, barrier arrival, release, list size).  A fast
// level has six: entry, columns, claim beside the claimed vertex's offsets,
// fence, and the exchange of the CTAs' counts, which is the barrier too.
//
// Lists: each of the kFastTeam CTAs appends to a segment of its own, a
// 16-byte record {vertex, first edge, degree} per entry, two buffers.  A
// level ends when every CTA has published one word (entries, edges, largest
// degree, stamped with the number of the exchange) and warp 0 has read the
// words of all of them.  The counts' prefix sums turn a list position into a
// segment and a slot.
// Work: four lanes per entry, two entries per lane group and two edges of
// each per lane in flight; entry k goes to CTA k % kFastTeam, so a level
// spreads over the team and a CTA takes at most ceil(N / kFastRound) * 64
// entries.  A level runs here only while that times the largest degree is
// at most the segment's size (it cannot overflow), no entry has more than
// kFastMaxDeg edges (no lane loops long) and the list has at most
// LB_FAST_LIMIT * small_edges edges.
// Measured, per level: grid BFS (4000-8000 edges) 7.7 -> 3.0 us, grid SSSP
// 9 -> 4.6 us, with 16384-32768 edges 10.2 -> 5.6 us, 32768-65536 edges
// 10.2 -> 8.3 us (above that the whole grid is as fast, hence LB_FAST_LIMIT).
// Teams of 32 / 64 / 128 CTAs on both halves of the L2: grid BFS 3.9 / 3.3 /
// 5.6 us (the words of 128 CTAs take longer to collect).
constexpr int kFastLanes = 4;
constexpr int kFastWords = kFastTeam / 32;  // CTAs' words a lane of warp 0 reads
static_assert(kFastWords % 2 == 0, "words are read in pairs");
constexpr uint32_t kFastGroups = kBlock / kFastLanes;     // entries a CTA takes at once
constexpr uint32_t kFastRound = kFastGroups * kFastTeam;  // entries the team takes at once
constexpr uint32_t kFastMaxDeg = kFastSeg / kFastGroups;  // the longest entry
#ifndef LB_FAST_LIMIT
#define LB_FAST_LIMIT 4
#endif
constexpr uint32_t kFastMaxEdges = 1u << 24;

// Largest list (edges) of a fast level.
__device__ __forceinline__ uint32_t fast_limit(int32_t small_edges) {
    return (uint32_t)min((int64_t)small_edges * LB_FAST_LIMIT, (int64_t)kFastMaxEdges);
}
__device__ __forceinline__ bool fast_fits(const QueryArgs &a, uint32_t n, uint32_t e, uint32_t maxdeg, uint32_t lim) {
    return e <= lim && maxdeg <= kFastMaxDeg &&
           (n + kFastRound - 1u) / kFastRound * maxdeg * kFastGroups <= (uint32_t)a.seg_cap;
}

// Whether a regular list is taken to the fast levels, and whether the team
// runs it (the same in every CTA).
__device__ __forceinline__ bool fast_takes(const StepParams &p, const QueryArgs &a, const QueryLoop &u) {
    return a.fast_seg && u.pull == 0u && u.cnt > 0u && u.maxdeg > 0u &&
           fast_fits(a, u.cnt, u.edges, u.maxdeg, fast_limit(p.small_edges));
}
__device__ __forceinline__ bool team_runs(const StepParams &p, const QueryArgs &a, const QueryLoop &u) {
    return p.small_edges > 0 && (u.edges <= (uint32_t)p.small_edges || fast_takes(p, a, u));
}

// One CTA's word of an exchange: stamp 16 | time limit passed 1 | largest
// degree 7 | entries 12 | edges 28; degree and edges saturate (a saturated
// value never fits, and what leaves the fast levels is counted anew).
__device__ __forceinline__ unsigned long long fast_word(uint32_t epoch, bool late, uint32_t maxdeg, uint32_t n,
                                                        uint32_t e) {
    return (unsigned long long)(epoch & 0xFFFFu) << 48 | (unsigned long long)(late ? 1u : 0u) << 47 |
           (unsigned long long)min(maxdeg, 127u) << 40 | (unsigned long long)n << 28 |
           (unsigned long long)min(e, (1u << 28) - 1u);
}

// Publishes this CTA's pushes and waits for everyone's (every thread calls
// it).  False when a CTA's word did not come within the barrier limit.
__device__ __forceinline__ bool fast_exchange(Ctl *ctl, QueryState &q) {
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t lane = threadIdx.x;
        const uint32_t epoch = q.fast_epoch + 1u;
        unsigned long long *const all = fast_words(ctl) + (epoch & 1u) * kFastTeam;
        if (lane == 0) {
            fence_acq_rel();
            *(volatile unsigned long long *)(all + q.rank) =
                fast_word(epoch, q.rank == 0u && global_ns() > q.deadline, q.out_maxdeg, q.out_n, q.out_e);
        }
        const unsigned long long *const words = all + kFastWords * lane;
        const uint64_t t0 = global_ns();
        unsigned long long w[kFastWords];
        bool ok = true;
        for (;;) {
            bool have = true;
#pragma unroll
            for (int j = 0; j < kFastWords; j += 2)
                asm volatile("ld.acquire.gpu.global.v2.u64 {%0, %1}, [%2];"
                             : "=l"(w[j]), "=l"(w[j + 1]) : "l"(words + j) : "memory");
#pragma unroll
            for (int j = 0; j < kFastWords; ++j) have = have && (uint32_t)(w[j] >> 48) == (epoch & 0xFFFFu);
            if (__all_sync(kFull, have)) break;
            if (__any_sync(kFull, global_ns() - t0 > kQueryBarrierNs)) {
                ok = false;
                break;
            }
        }
        uint32_t in = 0, e = 0, md = 0, late = 0;
#pragma unroll
        for (int j = 0; j < kFastWords; ++j) {
            in += (uint32_t)(w[j] >> 28) & 0xFFFu;
            // up to 2^26 / kFastWords each (the sum of all fits 32 bits): that never fits a fast level
            e += min((uint32_t)w[j] & ((1u << 28) - 1u), (1u << 26) / kFastWords);
            md = max(md, (uint32_t)(w[j] >> 40) & 127u);
            late |= (uint32_t)(w[j] >> 47) & 1u;
        }
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
            const uint32_t t = __shfl_up_sync(kFull, in, k);
            if ((int)lane >= k) in += t;
        }
        const uint32_t tot = __shfl_sync(kFull, in, 31);
#pragma unroll
        for (int j = kFastWords - 1; j >= 0; --j) {
            q.fast_pre[kFastWords * lane + j + 1] = in;
            in -= (uint32_t)(w[j] >> 28) & 0xFFFu;
        }
        e = __reduce_add_sync(kFull, e);
        md = __reduce_max_sync(kFull, md);
        late = __reduce_or_sync(kFull, late);
        if (lane == 0) {
            q.fast_pre[0] = 0;
            q.fast_n = tot;
            q.fast_e = e;
            q.fast_maxdeg = md;
            q.fast_late = late;
            q.fast_epoch = epoch;
            q.ok = ok ? 1u : 0u;
            q.out_n = q.out_e = q.out_maxdeg = 0u;
        }
    }
    __syncthreads();
    return q.ok != 0u;
}

// Appends the lanes' entries (those with want set) to this CTA's segment.
__device__ __forceinline__ void fast_push(int4 *seg, int32_t cap, QueryState &q, bool want, int32_t v, int32_t beg, int32_t deg) {
    const unsigned m = __ballot_sync(kFull, want);
    if (!m) return;
    const uint32_t lane = lane_id();
    const uint32_t e = __reduce_add_sync(kFull, want ? (uint32_t)deg : 0u);
    const uint32_t md = __reduce_max_sync(kFull, want ? (uint32_t)deg : 0u);
    uint32_t base = 0;
    if (lane == 0) {
        base = atomicAdd(&q.out_n, (uint32_t)__popc(m));
        atomicAdd(&q.out_e, e);
        atomicMax(&q.out_maxdeg, md);
    }
    base = __shfl_sync(kFull, base, 0);
    const uint32_t slot = base + __popc(m & lanemask_lt());
    if (want && slot < (uint32_t)cap) seg[slot] = make_int4(v, beg, deg, 0);
}

// Segment holding list position i.
__device__ __forceinline__ uint32_t fast_segment(const uint32_t *pre, uint32_t i) {
    uint32_t lo = 0;
#pragma unroll
    for (int k = kFastTeam / 2; k > 0; k >>= 1)
        if (pre[lo + k] <= i) lo += k;
    return lo;
}

// Runs levels on the team's segments from the regular list lists[u.par], and
// leaves a regular list (or an empty one) and the loop state behind.  Every
// thread of every team CTA calls it with the same state.  False: a wait ran
// out.
template <bool SSSP>
__device__ __forceinline__ bool fast_levels(const StepParams &p, const QueryArgs &a, QuerySync *sync, QueryState &q,
                                            WarpBufT<SSSP ? LB_KWB_WD_SSSP : LB_KWB_WD_BFS> &wb) {
    constexpr int kE = 2, kU = 2, kI = kE * kU;  // entries of a lane group, edges per lane of each, at once
    Ctl *const ctl = p.ctl;
    const uint32_t tid = threadIdx.x, rank = q.rank;
    const uint32_t lim = fast_limit(p.small_edges);
    const uint32_t conv = q.fast_conv & 1u;
    int4 *const mine = a.fast_seg + (size_t)rank * a.seg_cap;  // this CTA's segment of buffer 0
    const size_t seg_buf = (size_t)kFastTeam * a.seg_cap;
    // the regular list into segment buffer 0
    {
        const NodeList in = p.lists[q.u.par];
        const uint32_t n = q.u.cnt;
        // last used two conversions back: every CTA has read it since
        if (rank == 0 && tid == 0) sync->fast_pack[conv] = 0ull;
        for (uint32_t i0 = 0; i0 < n; i0 += kBlock * kFastTeam) {
            const uint32_t i = i0 + tid * kFastTeam + rank;
            int32_t v = 0, beg = 0, deg = 0;
            if (i < n) {
                v = in.v[i];
                beg = in.beg[i];
                deg = (i + 1 < n ? in.scan[i + 1] : (int32_t)q.u.edges) - in.scan[i];
                if (beg < 0 || deg < 0 || (int64_t)beg + deg > p.g.m || v < 0 || (int64_t)v >= p.g.n) {
                    atomicOr(&ctl->error, kErrBounds);
                    v = beg = deg = 0;
                }
            }
            // fast levels set no queued bits: drop the ones of this list
            if (SSSP && i < n) {
                uint32_t *const qn = queued_half(p.bitmap, p.bm_words, q.u.level + 1u);
                atomicAnd(qn + ((uint32_t)v >> 5), ~(1u << ((uint32_t)v & 31u)));
            }
            fast_push(mine, a.seg_cap, q, i < n && deg > 0, v, beg, deg);
        }
        if (!fast_exchange(ctl, q)) return false;
        if (tid == 0) ++q.fast_conv;
    }
    uint32_t buf = 0, err = 0;
    for (;;) {
        const uint32_t n = q.fast_n, e = q.fast_e, level = q.u.level;
        if (err || n == 0u || !fast_fits(a, n, e, q.fast_maxdeg, lim)) break;
        const int4 *const in = a.fast_seg + buf * seg_buf;
        int4 *const out = mine + (buf ^ 1u) * seg_buf;
        const int32_t r = (int32_t)(tid % kFastLanes);
        for (uint32_t i0 = 0; i0 < n; i0 += kE * kFastRound) {
            int4 x[kE];
            uint32_t du[kE];
            int32_t maxdeg = 0;
#pragma unroll
            for (int g = 0; g < kE; ++g) {
                const uint32_t i = i0 + g * kFastRound + (tid / kFastLanes) * kFastTeam + rank;
                x[g] = make_int4(0, 0, 0, 0);
                du[g] = 0u;
                if (i < n) {
                    const uint32_t sg = fast_segment(q.fast_pre, i);
                    x[g] = __ldcg(in + (size_t)sg * a.seg_cap + (i - q.fast_pre[sg]));
                }
            }
#pragma unroll
            for (int g = 0; g < kE; ++g) {
                maxdeg = max(maxdeg, x[g].z);
                if (SSSP && x[g].z > 0) du[g] = __ldcg(a.status + x[g].x);
            }
            for (int32_t k = r; __any_sync(kFull, k < maxdeg); k += kFastLanes * kU) {
                int32_t c[kI], b0[kI], b1[kI];
                uint32_t w[kI], old[kI];
#pragma unroll
                for (int j = 0; j < kI; ++j) {
                    const int32_t kk = k + kFastLanes * (j % kU);
                    const int4 &y = x[j / kU];
                    c[j] = kk < y.z ? __ldg(p.g.col + y.y + kk) : -1;
                    w[j] = SSSP && kk < y.z ? __ldg(p.g.w + y.y + kk) : 0u;
                }
                // the claim and the offsets of the vertex in one round trip
#pragma unroll
                for (int j = 0; j < kI; ++j) {
                    old[j] = SSSP ? 0u : kInf;
                    b0[j] = b1[j] = 0;
                    if (SSSP) {
                        // du is finite: the entry was reached
                        const uint32_t s32 = du[j / kU] + w[j];
                        w[j] = (s32 < w[j] || s32 >= kSat) ? kSat : s32;
                    }
                    if (c[j] >= 0) {
                        if (SSSP) old[j] = atomicMin(a.status + c[j], w[j]);
                        else old[j] = atomicOr(p.bitmap + ((uint32_t)c[j] >> 5), 1u << ((uint32_t)c[j] & 31u));
                        b0[j] = (int32_t)__ldg(p.g.off + c[j]);
                        b1[j] = (int32_t)__ldg(p.g.off + c[j] + 1);
                    }
                }
#pragma unroll
                for (int j = 0; j < kI; ++j) {
                    bool want;
                    if (SSSP) {
                        // a vertex improved k times in a level is listed k
                        // times: the repeats relax nothing, and a queued bit
                        // would be one more round trip per level
                        want = w[j] < old[j];
                        if (want && w[j] == kSat) atomicOr(&ctl->error, kErrSaturated);
                        if (want && w[j] >= q.u.T) {
                            const uint32_t blk = (uint32_t)c[j] >> q.far.shift;
                            atomicOr(q.far.bits + (blk >> 5), 1u << (blk & 31u));  // no result: nothing waits for it
                            want = false;
                        }
                    } else {
                        want = !((old[j] >> ((uint32_t)c[j] & 31u)) & 1u);
                        if (want) a.status[c[j]] = level + 1u;
                    }
                    fast_push(out, a.seg_cap, q, want && b1[j] > b0[j], c[j], b0[j], b1[j] - b0[j]);
                }
            }
        }
        if (!fast_exchange(ctl, q)) return false;
        if (tid == 0) {
            if (rank == 0) {
                if (q.trace < (uint32_t)kTraceMax) {
                    TraceRec *t = &ctl->trace[q.trace];
                    t->level = (int32_t)q.u.iters;
                    t->mode = kModeSmall;
                    t->list_size = n;
                    t->edges = e;
                    t->t_ns = (int64_t)(global_ns() - q.t0);
                    ++q.trace;
                }
                q.pushes += q.fast_n;
            }
            if (SSSP) far_engage(q, e, p.g.m);
            q.u.relaxed += e;
            q.u.iters += 1u;
            q.u.level = level + 1u;
        }
        buf ^= 1u;
        __syncthreads();
        if (q.fast_n > 0u) {
            if (q.u.iters >= a.max_levels) err = kErrIterCap;
            else if (q.fast_late) err = kErrDeadline;
        }
    }
    const uint32_t n = q.fast_n;
    if (err || n == 0u) {
        if (tid == 0) {
            if (err) atomicOr(&ctl->error, err);
            q.u.cnt = n;
            q.u.edges = 0;
            q.u.done = 1u;
            if (SSSP && !err && q.u.T != kInf) far_start_pull(q, q.u.T);
        }
        __syncthreads();
        return true;
    }
    // back to a regular list in lists[u.par], whose entries have all been read
    {
        const int4 *const in = a.fast_seg + buf * seg_buf;
        FlushOut o;
        o.list = p.lists[q.u.par];
        o.elist = nullptr;
        o.pack = &sync->fast_pack[conv];
        o.err = &ctl->error;
        o.pushes = nullptr;
        o.child_first = nullptr;
        o.cap = p.list_cap;
        o.tile_cap = p.tile_cap;
        o.tile = (int32_t)kTileGrain;
        o.mdt = p.mdt;
        NoScratch ns;
        uint32_t cnt = 0;
        for (uint32_t i0 = 0; i0 < n; i0 += kBlock * kFastTeam) {
            const uint32_t i = i0 + tid * kFastTeam + rank;
            int4 x = make_int4(0, 0, 0, 0);
            if (i < n) {
                const uint32_t sg = fast_segment(q.fast_pre, i);
                x = __ldcg(in + (size_t)sg * a.seg_cap + (i - q.fast_pre[sg]));
            }
            bool want = i < n;
            if (SSSP && want) {
                // each vertex once, with the queued bit of the level before
                uint32_t *const qb = queued_half(p.bitmap, p.bm_words, q.u.level + 1u);
                const uint32_t bit = 1u << ((uint32_t)x.x & 31u);
                want = !(atomicOr(qb + ((uint32_t)x.x >> 5), bit) & bit);
            }
            wpush(wb, cnt, want, x.x, x.y, (uint32_t)x.z);
            if (cnt > (uint32_t)(WarpBufT<SSSP ? LB_KWB_WD_SSSP : LB_KWB_WD_BFS>::kCap - 32))
                wflush<kOutNode, true>(wb, ns, cnt, o);
        }
        wflush_block<kOutNode, true>(wb, ns, cnt, o);
        __syncthreads();
        if (tid == 0) {
            q.ok = arrive_team(sync, kFastTeam, ++q.team) ? 1u : 0u;
            const unsigned long long x = __ldcg(&sync->fast_pack[conv]);
            q.u.cnt = (uint32_t)(x >> 32);
            q.u.edges = (uint32_t)x;
            q.u.maxdeg = 0u;  // it did not fit: a regular level is next
        }
        __syncthreads();
    }
    return q.ok != 0u;
}

// A pull step up to its barrier, out of line: its registers are not the
// walk's.
template <class WB>
__device__ __noinline__ void pull_level(const StepParams &p, const QueryArgs &a, QuerySync::Step *step, QueryState &q,
                                        WB &wb, uint32_t me, uint32_t ctas) {
    NoScratch ns;
    FlushOutT<1> o;
    o.list = p.lists[q.u.par ^ 1u];
    o.elist = nullptr;
    o.pack = &step->v;
    o.cap = p.list_cap;
    o.tile_cap = p.tile_cap;
    o.tile = (int32_t)kTileGrain;
    o.mdt = p.mdt;
    o.err = &p.ctl->error;
    o.pushes = nullptr;
    o.child_first = nullptr;
    o.off = p.g.off;
    o.maxdeg = &q.maxdeg;
    uint32_t cnt = 0;
    far_pull(a.status, p.g.n, q.far, q.u.T0, q.u.T, me, ctas, &q.fmin, wb, ns, cnt, o);
}

// One regular level up to its barrier: the walk over the list's tiles and
// the flushes.
// Long lists are walked in slices that the warps claim one by one, in list
// order, instead of two tiles per CTA laid down ahead.  A warp's time per
// edge depends on what it finds (candidates, flushes, hubs, the die its
// lines live on): with the fixed split the grid waited 50-155 us per level
// of 0.8-1.75 ms at scale 24 for its last CTA (measured with per-CTA
// clocks), and a 4096-edge slice starts 4x less often than a 1024-edge one
// (a start is a chain of ~5 dependent loads, ~1.8 us).  R-MAT edge factor
// 32, highest-degree source, fixed -> claimed: BFS scale 21 294 -> 284, 22
// 500 -> 476, 23 891 -> 836, 24 1706 -> 1601 us; SSSP 1228 -> 1217, 1994
// -> 1950, 3367 -> 3135, 5466 -> 5060 us.
//
// A slice is wd_tile edges (BFS) or half of that (SSSP: list order keeps
// the distances fresher; 4096 against 8192 / 16384 edges: 5.06 / 5.35 / 5.67
// ms), at most half a warp's share; when less than two such rounds are left,
// slices halve from half of what is left down to LB_SLICE_LOW grains (1 / 2
// / 4 grains: BFS 1613 / 1607 / 1617, SSSP 5111 / 5094 / 5122 us).  A claim is one
// atomic on one word, made while the warp walks the slice before: 2048-edge
// slices (BFS 1645 us) and 1024-edge slices (1803 us) pay for the starts and
// the claims.
//
// Lists of fewer than LB_CLAIM_SHARE grains per warp keep the fixed split:
// there the claimed slices become so short that their starts cost what the
// balance gains (scale 20, edge factor 16, 6-12 grains per warp: BFS 134 ->
// 138, SSSP 471 -> 476 us; a line at 8 / 16 / 32 at scale 21: BFS 284 / 284 /
// 289 us).
#ifndef LB_CLAIM_SHARE
#define LB_CLAIM_SHARE 16
#endif
#ifndef LB_SLICE_LOW
#define LB_SLICE_LOW 2
#endif

// Grains of a full slice; share: grains per warp, at least 2.
template <bool SSSP>
__device__ __forceinline__ uint32_t full_slice(uint32_t share, uint32_t tile) {
    return min(max(tile / (uint32_t)(SSSP ? 2 * kTileGrain : kTileGrain), 1u), share / 2u);
}

// Slice k of a list claimed in slices: its first edge and its edges.  Slices
// follow one another without gaps for every k; the first past the list's end
// tells a warp that it is done (k stays below the list's grains + warps).
template <bool SSSP>
__device__ __forceinline__ void claimed_slice(uint32_t k, uint32_t share, uint32_t tile, uint32_t warps, uint32_t &w0,
                                              uint32_t &len) {
    uint32_t s = full_slice<SSSP>(share, tile);
    const uint32_t full = (share - s) / s;  // rounds of the grid in slices of s grains
    uint32_t pos = 0;
    if (k >= full * warps) {
        k -= full * warps;
        pos = full * warps * s;
        uint32_t r = share - full * s;  // grains left per warp
        s = max(r / 2u, (uint32_t)LB_SLICE_LOW);
        while (s > (uint32_t)LB_SLICE_LOW && k >= warps) {
            pos += warps * s;
            k -= warps;
            r -= s;
            s = max(r / 2u, (uint32_t)LB_SLICE_LOW);
        }
    }
    w0 = (pos + k * s) * (uint32_t)kTileGrain;
    len = s * (uint32_t)kTileGrain;
}

template <bool SSSP, int ITEMS>
__device__ __forceinline__ void regular_level(const StepParams &p, const QueryArgs &a, QuerySync::Step *step, QueryState &q,
                                           WarpBufT<SSSP ? LB_KWB_WD_SSSP : LB_KWB_WD_BFS> &wb, uint32_t me,
                                           uint32_t ctas, bool team_mode) {
    Ctl *const ctl = p.ctl;
    uint32_t *const status = a.status;
    NoScratch ns;
    const uint32_t level = q.u.level, par = q.u.par, in_cnt = q.u.cnt, E = q.u.edges;
    uint32_t *const qcur = queued_half(p.bitmap, p.bm_words, level);
    const NodeList in = p.lists[par];
    if (SSSP) {
        // the other half holds the bits of the previous level, whose
        // queued vertices with out-edges are exactly this level's entries
        // (bits of vertices without out-edges are never read): clear
        // those, or sweep the half when the list is long
        if (!team_mode && (int64_t)in_cnt > p.bm_words / 8) {
            clear_next_queued(p.bitmap, p.bm_words, level);
        } else {
            uint32_t *qn = queued_half(p.bitmap, p.bm_words, level + 1u);
            for (uint32_t k = me * kBlock + threadIdx.x; k < in_cnt; k += ctas * kBlock) {
                const int32_t u = in.v[k];
                if (u >= 0 && (int64_t)u < p.g.n) atomicAnd(&qn[(uint32_t)u >> 5], ~(1u << ((uint32_t)u & 31u)));
            }
        }
    }
    FlushOutT<SSSP ? 3 : 2> o;
    o.list = p.lists[par ^ 1u];
    o.elist = nullptr;
    o.pack = &step->v;
    o.cap = p.list_cap;
    o.tile_cap = p.tile_cap;
    o.tile = (int32_t)kTileGrain;
    o.mdt = p.mdt;
    o.err = &ctl->error;
    o.pushes = nullptr;
    o.child_first = nullptr;
    o.off = p.g.off;
    o.maxdeg = &q.maxdeg;
    if (SSSP) o.far = &q.far;
    o.claim_bitmap = SSSP ? qcur : p.bitmap;
    o.claim_status = status;
    o.claim_level = level;
    uint32_t cnt = 0;
    const uint32_t warp = threadIdx.x >> 5, warps = ctas * kWarps;
    const uint32_t share = E / ((uint32_t)kTileGrain * warps);  // grains per warp
    const bool claims = share >= (uint32_t)LB_CLAIM_SHARE;  // a team's lists are far shorter
    const uint32_t T = (uint32_t)iteration_tile(E, ctas, p.tile);
    uint32_t len = claims ? full_slice<SSSP>(share, (uint32_t)p.tile) * (uint32_t)kTileGrain : T / kWarps;
    uint32_t w0 = (me * kWarps + warp) * len;
    while (w0 < E) {  // warp-uniform
        uint32_t k = 0;  // the next slice, claimed ahead
        if (claims && lane_id() == 0) k = atomicAdd(&step->next, 1u);
        wd_walk_slice<SSSP, ITEMS, kLdPlain>(p.g, in, (int32_t)in_cnt, E, w0, min(w0 + len, E), p.bitmap, qcur, status,
                                             level, &ctl->error, wb, ns, cnt, o);
        if (claims) claimed_slice<SSSP>(warps + __shfl_sync(kFull, k, 0), share, (uint32_t)p.tile, warps, w0, len);
        else w0 += warps * len;
    }
    wflush_block<kOutNode, true>(wb, ns, cnt, o);
}

template <bool SSSP, int ITEMS>
__global__ void __launch_bounds__(kBlock, SSSP ? LB_QUERY_MIN_BLOCKS_SSSP : LB_QUERY_MIN_BLOCKS)
    k_query_wd(const __grid_constant__ StepParams p, const __grid_constant__ QueryArgs a) {
    __shared__ WarpBufT<SSSP ? LB_KWB_WD_SSSP : LB_KWB_WD_BFS> s_wb[kWarps];
    __shared__ QueryState q;  // in shared memory: the registers belong to the walk
    Ctl *ctl = p.ctl;
    QuerySync *const sync = &ctl->qsync[a.number & 1u];
    uint32_t *const status = a.status;

    // ---- set-up -----------------------------------------------------------
    {
        const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        const int64_t stride = (int64_t)gridDim.x * blockDim.x;
        const int32_t src = a.src;
        const int64_t n = p.g.n;
        const int64_t beg = p.g.off[src];
        const int64_t deg = p.g.off[src + 1] - beg;
        unsigned long long wsum = 0;  // SSSP, CTA 0: weights sampled by this thread
        if (SSSP && blockIdx.x == 0 && p.g.m > 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) wsum += __ldg(p.g.w + (((int64_t)threadIdx.x * 4 + k) * p.g.m >> 10));
        }
        if (((uintptr_t)status & 15u) == 0) {
            uint4 *s4 = reinterpret_cast<uint4 *>(status);
            const int64_t n4 = n / 4;
            for (int64_t i = tid; i < n4; i += stride) {
                uint4 x = make_uint4(kInf, kInf, kInf, kInf);
                if (i == src / 4) {
                    const int32_t k = src % 4;
                    if (k == 0) x.x = 0u;
                    else if (k == 1) x.y = 0u;
                    else if (k == 2) x.z = 0u;
                    else x.w = 0u;
                }
                s4[i] = x;
            }
            for (int64_t i = 4 * n4 + tid; i < n; i += stride) status[i] = i == src ? 0u : kInf;
        } else {
            for (int64_t i = tid; i < n; i += stride) status[i] = i == src ? 0u : kInf;
        }
        // BFS: the visited bits, the source already visited; SSSP: both
        // queued halves empty
        const int64_t words = SSSP ? 2 * p.bm_words : (n + 31) / 32;
        for (int64_t w = tid; w < words; w += stride)
            p.bitmap[w] = (!SSSP && w == (src >> 5)) ? (1u << (src & 31)) : 0u;
        if (SSSP)
            for (int64_t w = tid; w < kFarWords; w += stride) ctl->far_bits[w] = 0u;
        const NodeList L = p.lists[0];
        if (L.tstart != nullptr) {
            const int64_t grains = (deg + kTileGrain - 1) / kTileGrain;
            for (int64_t k = tid; k < grains && k < p.tile_cap; k += stride) L.tstart[k] = 0;
        }
        if (threadIdx.x == 0) {
            for (uint32_t k = 0; k < sizeof(QueryState) / 4; ++k) reinterpret_cast<uint32_t *>(&q)[k] = 0u;
            q.u.cnt = deg > 0 ? 1u : 0u;
            q.u.edges = q.u.maxdeg = (uint32_t)deg;
            q.u.T = q.far.T = kInf;
            q.far.shift = a.far_shift;
            q.far.bits = ctl->far_bits;
            q.fmin = kInf;
            q.t0 = global_ns();
            q.deadline = q.t0 + a.time_limit_ns;
            // The team is the first CTA on each of the SMs that k_team_pick
            // gave a rank.
            uint32_t sm;
            asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
            q.rank = kNoRank;
            if (sm < kMaxSms && atomicAdd(&sync->sm_ctas[sm], 1u) == 0u) {
                q.rank = ctl->sm_rank[sm];
                if (q.rank != kNoRank) atomicAdd(&sync->team_here, 1u);
            }
            if (blockIdx.x == 0) {
                L.v[0] = src;
                L.beg[0] = (int32_t)beg;
                L.scan[0] = 0;
                L.scan[deg > 0 ? 1 : 0] = (int32_t)deg;
                ctl->status = status;
                ctl->src = src;
                ctl->kind = SSSP ? 1 : 0;
                if (a.prev_error) *a.prev_error = ctl->error;
                ctl->error = 0;
                ctl->t_start = q.t0;
                // what a query that ends at a wait's limit reports
                ctl->level = ctl->trace_len = ctl->in_cnt = 0u;
                ctl->step = ctl->in_edges = 0u;
                ctl->relaxed = ctl->pushes = 0ull;
            }
        }
        if (blockIdx.x == 0) {
            uint32_t *const nx = reinterpret_cast<uint32_t *>(&ctl->qsync[(a.number + 1u) & 1u]);
            for (uint32_t k = threadIdx.x; k < sizeof(QuerySync) / 4; k += kBlock) nx[k] = 0u;
            for (uint32_t k = threadIdx.x; k < 2 * kFastTeam; k += kBlock) fast_words(ctl)[k] = 0ull;
            if (SSSP) {
                // mean weight of 1024 evenly spaced edges -> first interval width
                __shared__ unsigned long long s_w;
                if (threadIdx.x == 0) s_w = 0ull;
                __syncthreads();
#pragma unroll
                for (int k = 16; k > 0; k >>= 1) wsum += __shfl_xor_sync(kFull, wsum, k);
                if (lane_id() == 0) atomicAdd(&s_w, wsum);
                __syncthreads();
                if (threadIdx.x == 0) {
                    const double d = (double)LB_FAR_MULT * ((double)s_w / 1024.0) * (double)n /
                                     (double)(p.g.m > 0 ? p.g.m : 1);
                    sync->delta0 = d < 1.0 ? 1u : d > (double)kFarMaxDelta ? kFarMaxDelta : (uint32_t)d;
                }
            }
        }
        // test hook: a CTA that never arrives makes the others' waits run out
        if (p.test_barrier_skip == kTestSkip && blockIdx.x == 1) return;
        __syncthreads();
        if (threadIdx.x == 0) {
            q.full = 1;
            q.ok = arrive_full(sync, gridDim.x, 1u) ? 1u : 0u;
            // not every SM of the team holds a CTA: the first CTAs are the team
            if (__ldcg(&sync->team_here) != (uint32_t)a.team)
                q.rank = blockIdx.x < (uint32_t)a.team ? blockIdx.x : kNoRank;
            if (SSSP) q.u.delta = __ldcg(&sync->delta0);
            q.u.delta_min = max(q.u.delta / LB_FAR_MINDIV, 1u);
        }
        __syncthreads();
    }

    // ---- worklist iterations ------------------------------------------------
    bool team_mode = false;
    bool failed = q.ok == 0u;
    while (!failed && !q.u.done) {
        const uint32_t E = q.u.edges;
        const bool small = team_runs(p, a, q.u);
        if (small && !team_mode) {
            team_mode = true;
            if (q.rank == kNoRank) {
                // wait until the team publishes the state it stopped at (every
                // thread has read the loop state before it is replaced)
                __syncthreads();
                if (threadIdx.x == 0)
                    q.ok = wait_for(&sync->resume, ++q.resume, a.time_limit_ns + 2 * kQueryBarrierNs, true) ? 1u : 0u;
                __syncthreads();
                if (threadIdx.x < sizeof(QueryLoop) / 4)
                    reinterpret_cast<uint32_t *>(&q.u)[threadIdx.x] =
                        __ldcg(reinterpret_cast<const uint32_t *>(&sync->loop) + threadIdx.x);
                __syncthreads();
                if (threadIdx.x == 0) q.far.T = q.u.T;
                __syncthreads();
                failed = q.ok == 0u;
                team_mode = false;
                continue;
            }
        } else if (!small) {
            team_mode = false;
        }
        const bool fast = team_mode && fast_takes(p, a, q.u);
        if (p.test_barrier_skip >= kTestTeamSkip && team_mode &&
            (p.test_barrier_skip == kTestTeamGone || (q.rank == 1u && p.test_barrier_skip == (fast ? kTestFastSkip : kTestTeamSkip))))
            return;
        if (fast) {
            // uniform over the team: every CTA has the same state
            failed = !fast_levels<SSSP>(p, a, sync, q, s_wb[threadIdx.x >> 5]);
            // the team hands over, as after a regular level
            if (!failed && q.rank == 0u && threadIdx.x == 0 && (q.u.done || !team_runs(p, a, q.u))) publish(sync, q);
            continue;
        }
        const uint32_t ctas = team_mode ? (uint32_t)a.team : gridDim.x;
        const uint32_t me = team_mode ? q.rank : blockIdx.x;
        const uint32_t level = q.u.level, par = q.u.par;
        const uint32_t in_cnt = q.u.cnt;
        const bool pull = SSSP && q.u.pull != 0u;
        // the next step of this kind finds its counters cleared
        if (q.rank == 0u && threadIdx.x == 0) {
            QuerySync::Step *const nx = step_counters(sync, q, team_mode, 1u);
            nx->v = 0ull;
            nx->far_left = 0u;
            nx->maxdeg = 0u;
            nx->next = 0u;
        }
        if (SSSP && pull) pull_level(p, a, step_counters(sync, q, team_mode, 0u), q, s_wb[threadIdx.x >> 5], me, ctas);
        else regular_level<SSSP, ITEMS>(p, a, step_counters(sync, q, team_mode, 0u), q, s_wb[threadIdx.x >> 5], me, ctas, team_mode);
        __syncthreads();
        if (threadIdx.x == 0) {
            QuerySync::Step *const step = step_counters(sync, q, team_mode, 0u);
            if (SSSP && pull && q.fmin != kInf) {
                atomicMax(&step->far_left, ~q.fmin);
                q.fmin = kInf;
            }
            if (q.maxdeg > 0u) {
                atomicMax(&step->maxdeg, q.maxdeg);
                q.maxdeg = 0u;
            }
            if (q.rank == 0u && global_ns() > q.deadline) atomicOr(&step->v, 1ull << 63);
            q.ok = (team_mode ? arrive_team(sync, ctas, ++q.team) : arrive_full(sync, ctas, ++q.full)) ? 1u : 0u;
            // test hook: the team is far ahead when these CTAs read
            if (p.test_barrier_skip == kTestLateReads && q.rank == kNoRank)
                for (const uint64_t t = global_ns(); global_ns() - t < 200000u;) __nanosleep(1000);
            const unsigned long long x = __ldcg(&step->v);
            q.u.maxdeg = __ldcg(&step->maxdeg);
            const uint32_t fmin = SSSP && pull ? ~__ldcg(&step->far_left) : 0u;
            ++(team_mode ? q.team_steps : q.grid_steps);
            uint32_t ncnt = (uint32_t)(x >> 32) & 0x7FFFFFFFu;
            uint32_t err = 0;
            if ((int64_t)ncnt > p.list_cap) {
                err |= kErrCapacity;
                ncnt = (uint32_t)p.list_cap;
            }
            if (q.rank == 0u) {
                if (!pull && q.trace < (uint32_t)kTraceMax) {
                    TraceRec *r = &ctl->trace[q.trace];
                    r->level = (int32_t)q.u.iters;
                    r->mode = team_mode ? kModeSmall : kModeRelax;
                    r->list_size = in_cnt;
                    r->edges = E;
                    r->t_ns = (int64_t)(global_ns() - q.t0);
                    ++q.trace;
                }
                q.pushes += ncnt;
            }
            q.u.level = level + 1u;
            q.u.par = par ^ 1u;
            q.u.cnt = ncnt;
            q.u.edges = (uint32_t)x;
            q.u.pull = 0u;
            if (!pull) {
                if (SSSP) far_engage(q, E, p.g.m);
                q.u.iters += 1u;
                q.u.relaxed += E;
            }
            bool more = ncnt > 0;
            // the list is empty: pull the next interval, unless no threshold
            // is in force or nothing was left at the last pull
            if (SSSP && !more && q.u.T != kInf && !(pull && fmin == kInf)) {
                more = true;
                far_start_pull(q, pull ? fmin : q.u.T);
            }
            if (more && q.u.iters >= a.max_levels) {
                err |= kErrIterCap;
                more = false;
            }
            if (more && (x >> 63) != 0ull) {
                err |= kErrDeadline;
                more = false;
            }
            if (err) atomicOr(&ctl->error, err);
            q.u.done = more ? 0u : 1u;
            // the team hands over: the list has grown, or the query ends
            if (q.rank == 0u && team_mode && q.ok && (q.u.done || !team_runs(p, a, q.u))) publish(sync, q);
        }
        __syncthreads();
        failed = q.ok == 0u;
    }
    if (failed) {
        if (threadIdx.x == 0) {
            atomicOr(&ctl->error, kErrDeadline);
            atomicExch(&sync->resume, kResumeAbort);
            ctl->active = 0u;
        }
        return;
    }

    // ---- tear-down ----------------------------------------------------------
    if (SSSP && (__ldcg(&ctl->error) & kErrSaturated)) {
        // some relaxation saturated: overflow iff a final distance still does
        const int64_t stride = (int64_t)gridDim.x * blockDim.x;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p.g.n; i += stride)
            if (__ldcg(status + i) == kSat) {
                atomicOr(&ctl->error, kErrOverflow);
                break;
            }
    }
    if (q.rank == 0u && threadIdx.x == 0) {
        p.lists[q.u.par].scan[q.u.cnt] = (int32_t)q.u.edges;
        ctl->level = q.u.iters;
        ctl->step = q.u.iters;
        ctl->par = q.u.par;
        ctl->in_cnt = q.u.cnt;
        ctl->in_edges = q.u.edges;
        ctl->active = 0u;
        ctl->relaxed = q.u.relaxed;
        ctl->pushes = q.pushes;
        ctl->trace_len = q.trace;
    }
}

cudaError_t launch_query_wd(bool sssp, const StepParams &p, const QueryArgs &a, int grid, cudaStream_t st) {
    // cooperative: the CTAs wait on one another at grid barriers, so all of
    // them must be resident at once
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kBlock);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return sssp ? cudaLaunchKernelEx(&cfg, k_query_wd<true, kItemsWdSssp>, p, a)
                : cudaLaunchKernelEx(&cfg, k_query_wd<false, kItemsWdBfs>, p, a);
}

// Resident CTAs per SM; also sets the kernels' shared-memory carve-out (see
// launch_step_wd): 25% selects the 64 KB configuration, which holds the
// resident CTAs' push buffers and leaves the rest to the L1.
int query_wd_blocks_per_sm(bool sssp) {
    int nb = 0;
    cudaError_t e;
    if (sssp) {
        e = cudaFuncSetAttribute(k_query_wd<true, kItemsWdSssp>, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_query_wd<true, kItemsWdSssp>, kBlock, 0);
    } else {
        e = cudaFuncSetAttribute(k_query_wd<false, kItemsWdBfs>, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_query_wd<false, kItemsWdBfs>, kBlock, 0);
    }
    return (e == cudaSuccess && nb > 0) ? nb : 1;
}

}  // namespace lbk
