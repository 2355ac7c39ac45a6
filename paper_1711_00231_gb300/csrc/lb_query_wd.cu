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
// or *p became kResumeAbort.
__device__ __forceinline__ bool wait_for(const uint32_t *p, uint32_t want, uint64_t limit, uint32_t sleep_ns) {
    if ((int32_t)(ld_acquire(p) - want) >= 0) return true;
    const uint64_t t0 = global_ns();
    for (;;) {
        const uint32_t v = ld_acquire(p);
        if (v == kResumeAbort) return false;
        if ((int32_t)(v - want) >= 0) return true;
        if (global_ns() - t0 > limit) return false;
        if (sleep_ns) __nanosleep(sleep_ns);
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
    return wait_for(&s->full_release, round, kQueryBarrierNs, 32);
}
__device__ __forceinline__ bool arrive_team(QuerySync *s, uint32_t size, uint32_t round) {
    fence_acq_rel();
    const uint32_t old = add_acq_rel(&s->team_arrive, 1u);
    if (old + 1u == size * round) return true;
    return wait_for(&s->team_arrive, size * round, kQueryBarrierNs, 0);
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
// are exactly those at T or above.  A bit per block of 2^far_shift (>= 128)
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
// Measured: 4096^2 grid 334 -> 96 ms (list edges 203 -> 8 per edge), uniform
// graph of 8.4M vertices and 33.5M edges 2.93 -> 1.67 ms (3.0 -> 1.3).
// First width 8 / 16 / 32 / 64 * weight / degree: uniform graph 2.14 / 1.73
// / 1.67 / 3.17 ms; kFarEdges 8192 / 32768: grid 97.4 / 96.2 ms.  On R-MAT
// graphs no width pays (a model of scale 21: 1.58 -> 1.42 relaxations per
// edge for 3 times the iterations), and the rule never sets T there.
#ifndef LB_FAR_EDGES
#define LB_FAR_EDGES 32768
#endif
#ifndef LB_FAR_MULT
#define LB_FAR_MULT 32
#endif
#ifndef LB_FAR_LOW
#define LB_FAR_LOW 8192
#endif
#ifndef LB_FAR_HIGH
#define LB_FAR_HIGH 131072
#endif
#ifndef LB_FAR_MINDIV
#define LB_FAR_MINDIV 4
#endif
constexpr int64_t kFarEdges = LB_FAR_EDGES;
constexpr uint32_t kFarLevels = 6, kFarLate = 32;
constexpr uint64_t kFarLow = LB_FAR_LOW, kFarHigh = LB_FAR_HIGH;

// T + delta, or "no threshold" when that passes the largest distance.
__device__ __forceinline__ uint32_t far_add(uint32_t t, uint32_t delta) {
    const uint64_t x = (uint64_t)t + delta;
    return x >= kSat ? kInf : (uint32_t)x;
}

// One pull: queues the vertices of the far set in [T0, T1), keeps the bits
// of the blocks that still hold vertices at T1 or above, and lowers *fmin
// (shared memory) to the smallest of those.  A warp owns a word of the
// bitmap: nothing else touches the bits during a pull.
template <class WB, class WS, class FO>
__device__ __forceinline__ void far_pull(const uint32_t *status, int64_t n, uint32_t *far_bits, int32_t shift,
                                         uint32_t T0, uint32_t T1, uint32_t ctas, uint32_t *fmin, WB &wb, WS &ws,
                                         uint32_t &cnt, const FO &o) {
    const uint32_t lane = lane_id();
    const int32_t words = (int32_t)((((n - 1) >> shift) >> 5) + 1);
    const int32_t stride = (int32_t)ctas * kWarps;
    uint32_t mn = kInf;
    for (int32_t w = (int32_t)blockIdx.x + (int32_t)ctas * (int32_t)(threadIdx.x >> 5); w < words; w += stride) {
        uint32_t bits = __ldcg(far_bits + w);
        uint32_t keep = 0;
        const uint32_t had = bits;
        while (bits) {  // warp-uniform
            const int b = __ffs(bits) - 1;
            bits &= bits - 1;
            const int64_t v0 = ((int64_t)w * 32 + b) << shift;
            const int64_t v1 = min(v0 + ((int64_t)1 << shift), n);
            bool left = false;
            for (int64_t v = v0 + lane; v < v1 + lane; v += 128) {  // warp-uniform trip count
                uint32_t d[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) d[r] = v + 32 * r < v1 ? __ldcg(status + v + 32 * r) : kInf;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (d[r] != kInf && d[r] >= T1) {
                        left = true;
                        mn = min(mn, d[r]);
                    }
                    const bool take = d[r] >= T0 && d[r] < T1;  // kInf is never below T1
                    if (__any_sync(kFull, take)) {
                        wpush(wb, cnt, take, (int32_t)(v + 32 * r), 0, 0u);
                        if (cnt > (uint32_t)(WB::kCap - 32)) wflush<kOutNode, true>(wb, ws, cnt, o);
                    }
                }
            }
            if (__any_sync(kFull, left)) keep |= 1u << b;
        }
        if (lane == 0 && keep != had) far_bits[w] = keep;
    }
    wflush<kOutNode, true>(wb, ws, cnt, o);
    mn = __reduce_min_sync(kFull, mn);
    if (lane == 0 && mn != kInf) atomicMin(fmin, mn);
}

template <bool SSSP, int ITEMS>
__global__ void __launch_bounds__(kBlock, SSSP ? LB_QUERY_MIN_BLOCKS_SSSP : LB_QUERY_MIN_BLOCKS)
    k_query_wd(StepParams p, QueryArgs a) {
    __shared__ WarpBufT<SSSP ? LB_KWB_WD_SSSP : LB_KWB_WD_BFS> s_wb[kWarps];
    // loop state, kept in shared memory (registers belong to the walk)
    __shared__ uint32_t s_ok, s_level, s_par, s_cnt, s_done, s_full, s_team, s_resume;
    __shared__ uint64_t s_edges, s_deadline, s_t0;
    __shared__ uint32_t s_trace;               // CTA 0
    __shared__ unsigned long long s_relaxed, s_pushes;
    // SSSP threshold: in force (s_far.T), the interval of a pull step [s_T0,
    // s_far.T), whether the next step is a pull, a pull's smallest distance left
    __shared__ FarSet s_far;
    __shared__ uint32_t s_iters, s_T0, s_pull, s_fmin;
    // CTA 0's decisions: width of the next interval and its smallest value,
    // lists and edges of the current interval
    __shared__ uint32_t s_delta, s_delta_min, s_int_lists;
    __shared__ uint64_t s_int_edges, s_int_max;
    NoScratch ns;
    Ctl *ctl = p.ctl;
    QuerySync *const sync = &ctl->qsync[a.number & 1u];
    uint32_t *const status = a.status;
    const int64_t lim = p.small_edges;

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
        const NodeList L = p.lists[0];
        if (L.tstart != nullptr) {
            const int64_t grains = (deg + kTileGrain - 1) / kTileGrain;
            for (int64_t k = tid; k < grains && k < p.tile_cap; k += stride) L.tstart[k] = 0;
        }
        if (threadIdx.x == 0) {
            s_level = 0;
            s_par = 0;
            s_cnt = deg > 0 ? 1u : 0u;
            s_edges = (uint64_t)deg;
            s_done = 0;
            s_full = s_team = s_resume = 0;
            s_trace = 0;
            s_iters = 0;
            s_far.T = kInf;
            s_far.shift = a.far_shift;
            s_far.bits = ctl->far_bits;
            s_T0 = s_pull = 0;
            s_fmin = kInf;
            s_delta = 0;
            s_int_lists = 0;
            s_int_edges = s_int_max = 0;
            s_relaxed = s_pushes = 0ull;
            s_t0 = global_ns();
            s_deadline = s_t0 + a.time_limit_ns;
            if (blockIdx.x == 0) {
                L.v[0] = src;
                L.beg[0] = (int32_t)beg;
                L.scan[0] = 0;
                L.scan[deg > 0 ? 1 : 0] = (int32_t)deg;
                ctl->status = status;
                ctl->src = src;
                ctl->kind = SSSP ? 1 : 0;
                ctl->error = 0;
                ctl->t_start = s_t0;
                QuerySync *const nx = &ctl->qsync[(a.number + 1u) & 1u];
                nx->full_arrive = nx->full_release = nx->team_arrive = nx->resume = 0u;
                for (int k = 0; k < 3; ++k) nx->pack[k].v = 0ull;
            }
        }
        if (SSSP) {
            for (int64_t w = tid; w < kFarWords; w += stride) ctl->far_bits[w] = 0u;
            if (blockIdx.x == 0) {
                // mean weight of 1024 evenly spaced edges -> first interval width
                __shared__ unsigned long long s_w;
                if (threadIdx.x == 0) s_w = 0ull;
                __syncthreads();
#pragma unroll
                for (int k = 16; k > 0; k >>= 1) wsum += __shfl_xor_sync(kFull, wsum, k);
                if (lane_id() == 0) atomicAdd(&s_w, wsum);
                __syncthreads();
                if (threadIdx.x == 0 && p.g.m > 0) {
                    const double d = (double)LB_FAR_MULT * ((double)s_w / 1024.0) * (double)n / (double)p.g.m;
                    s_delta = d < 1.0 ? 1u : d > 1073741824.0 ? (1u << 30) : (uint32_t)d;
                    s_delta_min = s_delta / LB_FAR_MINDIV > 0 ? s_delta / LB_FAR_MINDIV : 1u;
                }
            }
        }
        // test hook: a CTA that never arrives makes the others' waits run out
        if (p.test_barrier_skip && blockIdx.x == 1) return;
        __syncthreads();
        if (threadIdx.x == 0) {
            s_full = 1;
            s_ok = arrive_full(sync, gridDim.x, 1u) ? 1u : 0u;
        }
        __syncthreads();
    }

    // ---- worklist iterations ------------------------------------------------
    bool team_mode = false;
    bool failed = s_ok == 0u;
    while (!failed && !s_done) {
        const int64_t E = (int64_t)s_edges;
        const bool small = lim > 0 && E <= lim;
        if (small && !team_mode) {
            team_mode = true;
            if (blockIdx.x >= (uint32_t)a.team) {
                // wait until the team publishes the state it stopped at (every
                // thread has read the loop state before it is replaced)
                __syncthreads();
                if (threadIdx.x == 0) {
                    const uint32_t want = ++s_resume;
                    s_ok = wait_for(&sync->resume, want, a.time_limit_ns + 2 * kQueryBarrierNs, 1000) ? 1u : 0u;
                    s_level = __ldcg(&sync->r_level);
                    s_par = __ldcg(&sync->r_par);
                    s_cnt = __ldcg(&sync->r_cnt);
                    s_edges = __ldcg(&sync->r_edges);
                    s_done = __ldcg(&sync->r_done);
                    s_iters = __ldcg(&sync->r_iters);
                    s_pull = __ldcg(&sync->r_pull);
                    s_T0 = __ldcg(&sync->r_T0);
                    s_far.T = __ldcg(&sync->r_T);
                }
                __syncthreads();
                failed = s_ok == 0u;
                team_mode = false;
                continue;
            }
        } else if (!small) {
            team_mode = false;
        }
        const uint32_t ctas = team_mode ? (uint32_t)a.team : gridDim.x;
        const uint32_t level = s_level, par = s_par;
        const int64_t in_cnt = s_cnt;
        const bool pull = SSSP && s_pull != 0u;
        uint32_t *const qcur = queued_half(p.bitmap, p.bm_words, level);
        const NodeList in = p.lists[par];
        if (SSSP && !pull) {
            // the other half holds the bits of the previous level, whose
            // queued vertices with out-edges are exactly this level's entries
            // (bits of vertices without out-edges are never read): clear
            // those, or sweep the half when the list is long
            uint32_t *qn = queued_half(p.bitmap, p.bm_words, level + 1u);
            const int64_t stride = (int64_t)ctas * blockDim.x;
            const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
            if (!team_mode && in_cnt > p.bm_words / 8) {
                clear_next_queued(p.bitmap, p.bm_words, level);
            } else {
                for (int64_t k = tid; k < in_cnt; k += stride) {
                    const int32_t u = in.v[k];
                    if (u >= 0 && (int64_t)u < p.g.n) atomicAnd(&qn[(uint32_t)u >> 5], ~(1u << ((uint32_t)u & 31u)));
                }
            }
        }
        // the next level's output counter (its last reads were before the
        // barrier that ended the previous level)
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            QuerySync::Pack *const nx = &sync->pack[(level + 1u) % 3u];
            nx->v = 0ull;
            if (SSSP) {
                uint32_t T = s_far.T;
                if (pull) {
                    // an interval has ended: its lists decide the next width
                    if (s_int_lists > 0) {
                        const uint64_t avg = s_int_edges / s_int_lists;
                        if (avg < kFarLow && s_delta < (1u << 30)) s_delta *= 2u;
                        if (avg > kFarHigh) s_delta = max(s_delta / 2u, s_delta_min);
                    }
                    s_int_lists = 0;
                    s_int_edges = s_int_max = 0;
                } else {
                    ++s_int_lists;
                    s_int_edges += (uint64_t)E;
                    s_int_max = max(s_int_max, (uint64_t)E);
                    if (T == kInf && s_T0 == 0u && E >= kFarEdges &&
                        ((s_iters >= kFarLevels && s_relaxed + (uint64_t)E < (uint64_t)p.g.m / 4) ||
                         s_iters >= kFarLate)) {
                        T = far_add(0u, s_delta);
                        s_T0 = 1u;  // set once
                        s_int_lists = 0;
                        s_int_edges = s_int_max = 0;
                    }
                }
                nx->far_min = kInf;
                nx->T = T;
                nx->delta = s_delta;
                nx->pull_size = (uint32_t)(s_int_max > 0x7FFFFFFFull ? 0x7FFFFFFFull : s_int_max);
            }
        }
        FlushOutT<SSSP ? 3 : 2> o;
        o.list = p.lists[par ^ 1u];
        o.elist = nullptr;
        o.pack = &sync->pack[level % 3u].v;
        o.cap = p.list_cap;
        o.tile_cap = p.tile_cap;
        o.tile = (int32_t)kTileGrain;
        o.mdt = p.mdt;
        o.err = &ctl->error;
        o.pushes = nullptr;
        o.child_first = nullptr;
        o.off = p.g.off;
        if (SSSP) o.far = &s_far;
        o.claim_bitmap = SSSP ? qcur : p.bitmap;
        o.claim_status = status;
        o.claim_level = level;
        uint32_t cnt = 0;
        const uint32_t warp = threadIdx.x >> 5;
        const uint32_t T = (uint32_t)iteration_tile(E, ctas, p.tile);
        const uint32_t ntiles = pull ? 0u : ((uint32_t)E + T - 1u) / T;
        if (SSSP && pull) {
            FlushOutT<1> op;
            static_cast<FlushOut &>(op) = o;
            far_pull(status, p.g.n, ctl->far_bits, a.far_shift, s_T0, s_far.T, ctas, &s_fmin, s_wb[warp], ns, cnt, op);
        }
        for (uint32_t t = blockIdx.x; t < ntiles; t += ctas)
            wd_walk_tile<SSSP, ITEMS, kLdPlain>(p.g, in, (int32_t)in_cnt, (uint32_t)E, T, t, p.bitmap, qcur, status, level, &ctl->error,
                                                s_wb[warp], ns, cnt, o);
        wflush_block<kOutNode, true>(s_wb[warp], ns, cnt, o);
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long *const pk = &sync->pack[level % 3u].v;
            QuerySync::Pack *const nx = &sync->pack[(level + 1u) % 3u];
            if (SSSP && pull && s_fmin != kInf) {
                atomicMin(&sync->pack[level % 3u].far_min, s_fmin);
                s_fmin = kInf;
            }
            if (blockIdx.x == 0 && global_ns() > s_deadline) atomicOr(pk, 1ull << 63);
            s_ok = (team_mode ? arrive_team(sync, ctas, ++s_team) : arrive_full(sync, ctas, ++s_full)) ? 1u : 0u;
            const unsigned long long x = __ldcg(pk);
            const bool late = (x >> 63) != 0ull;
            int64_t ncnt = (int64_t)((x >> 32) & 0x7FFFFFFFull);
            uint32_t nedges = (uint32_t)x;
            uint32_t err = 0;
            if (ncnt > p.list_cap) {
                err |= kErrCapacity;
                ncnt = p.list_cap;
            }
            bool more = ncnt > 0;
            const uint32_t iters = s_iters + (pull ? 0u : 1u);
            uint32_t npull = 0, nT = kInf, nT0 = 0;
            if (SSSP) {
                const uint32_t fmin = pull ? __ldcg(&sync->pack[level % 3u].far_min) : 0u;
                const uint32_t delta = __ldcg(&nx->delta), hint = __ldcg(&nx->pull_size);
                nT = pull ? s_far.T : __ldcg(&nx->T);
                nT0 = s_T0;
                // the list is empty: pull the next interval, unless no
                // threshold is in force or nothing was left at the last pull
                if (!more && nT != kInf && !(pull && fmin == kInf)) {
                    npull = 1u;
                    more = true;
                    nT0 = nT;
                    nT = far_add(pull ? fmin : nT, delta);
                    nedges = hint;
                }
            }
            if (more && iters >= a.max_levels) {
                err |= kErrIterCap;
                more = false;
            }
            if (more && late) {
                err |= kErrDeadline;
                more = false;
            }
            if (err) atomicOr(&ctl->error, err);
            if (blockIdx.x == 0) {
                const uint32_t tl = s_trace;
                if (!pull && tl < (uint32_t)kTraceMax) {
                    TraceRec *r = &ctl->trace[tl];
                    r->level = (int32_t)s_iters;
                    r->mode = team_mode ? kModeSmall : kModeRelax;
                    r->list_size = in_cnt;
                    r->edges = E;
                    r->t_ns = (int64_t)(global_ns() - s_t0);
                    s_trace = tl + 1u;
                }
                if (!pull) s_relaxed += (unsigned long long)E;
                s_pushes += (unsigned long long)ncnt;
                // the team hands over: the list has grown, or the query ends
                if (team_mode && s_ok && (!more || (int64_t)nedges > lim)) {
                    sync->r_level = level + 1u;
                    sync->r_par = par ^ 1u;
                    sync->r_cnt = (uint32_t)ncnt;
                    sync->r_edges = nedges;
                    sync->r_done = more ? 0u : 1u;
                    sync->r_iters = iters;
                    sync->r_pull = npull;
                    sync->r_T0 = nT0;
                    sync->r_T = nT;
                    st_release(&sync->resume, ++s_resume);
                }
            }
            s_level = level + 1u;
            s_par = par ^ 1u;
            s_cnt = (uint32_t)ncnt;
            s_edges = nedges;
            s_done = more ? 0u : 1u;
            s_iters = iters;
            if (SSSP) {
                s_pull = npull;
                s_T0 = nT0;
                s_far.T = nT;
            }
        }
        __syncthreads();
        failed = s_ok == 0u;
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
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint32_t par = s_par;
        p.lists[par].scan[s_cnt] = (int32_t)s_edges;
        ctl->level = s_iters;
        ctl->step = s_iters;
        ctl->par = par;
        ctl->in_cnt = s_cnt;
        ctl->in_edges = s_edges;
        ctl->active = 0u;
        ctl->relaxed = s_relaxed;
        ctl->pushes = s_pushes;
        ctl->trace_len = s_trace;
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
