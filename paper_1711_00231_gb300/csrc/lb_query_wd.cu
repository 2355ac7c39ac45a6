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

template <bool SSSP, int ITEMS>
__global__ void __launch_bounds__(kBlock, SSSP ? LB_QUERY_MIN_BLOCKS_SSSP : LB_QUERY_MIN_BLOCKS)
    k_query_wd(StepParams p, QueryArgs a) {
    __shared__ WarpBufT<SSSP ? LB_KWB_WD_SSSP : LB_KWB_WD_BFS> s_wb[kWarps];
    // loop state, kept in shared memory (registers belong to the walk)
    __shared__ uint32_t s_ok, s_level, s_par, s_cnt, s_done, s_full, s_team, s_resume;
    __shared__ uint64_t s_edges, s_deadline, s_t0;
    __shared__ uint32_t s_trace;               // CTA 0
    __shared__ unsigned long long s_relaxed, s_pushes;
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
        uint32_t *const qcur = queued_half(p.bitmap, p.bm_words, level);
        const NodeList in = p.lists[par];
        if (SSSP) {
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
        if (blockIdx.x == 0 && threadIdx.x == 0) sync->pack[(level + 1u) % 3u].v = 0ull;
        FlushOut o;
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
        o.defer = SSSP ? 3 : 2;
        o.claim_bitmap = SSSP ? qcur : p.bitmap;
        o.claim_status = status;
        o.claim_level = level;
        uint32_t cnt = 0;
        const uint32_t warp = threadIdx.x >> 5;
        const int64_t T = iteration_tile(E, ctas, p.tile);
        const int64_t ntiles = (E + T - 1) / T;
        for (int64_t t = blockIdx.x; t < ntiles; t += ctas)
            wd_walk_tile<SSSP, ITEMS, kLdPlain>(p.g, in, in_cnt, E, T, t, p.bitmap, qcur, status, level, &ctl->error,
                                                s_wb[warp], ns, cnt, o);
        wflush_block<kOutNode, true>(s_wb[warp], ns, cnt, o);
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long *const pk = &sync->pack[level % 3u].v;
            if (blockIdx.x == 0 && global_ns() > s_deadline) atomicOr(pk, 1ull << 63);
            s_ok = (team_mode ? arrive_team(sync, ctas, ++s_team) : arrive_full(sync, ctas, ++s_full)) ? 1u : 0u;
            const unsigned long long x = __ldcg(pk);
            const bool late = (x >> 63) != 0ull;
            int64_t ncnt = (int64_t)((x >> 32) & 0x7FFFFFFFull);
            const uint32_t nedges = (uint32_t)x;
            uint32_t err = 0;
            if (ncnt > p.list_cap) {
                err |= kErrCapacity;
                ncnt = p.list_cap;
            }
            bool more = ncnt > 0;
            if (more && level + 1u >= a.max_levels) {
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
                if (tl < (uint32_t)kTraceMax) {
                    TraceRec *r = &ctl->trace[tl];
                    r->level = (int32_t)level;
                    r->mode = team_mode ? kModeSmall : kModeRelax;
                    r->list_size = in_cnt;
                    r->edges = E;
                    r->t_ns = (int64_t)(global_ns() - s_t0);
                    s_trace = tl + 1u;
                }
                s_relaxed += (unsigned long long)E;
                s_pushes += (unsigned long long)ncnt;
                // the team hands over: the list has grown, or the query ends
                if (team_mode && s_ok && (!more || (int64_t)nedges > lim)) {
                    sync->r_level = level + 1u;
                    sync->r_par = par ^ 1u;
                    sync->r_cnt = (uint32_t)ncnt;
                    sync->r_edges = nedges;
                    sync->r_done = more ? 0u : 1u;
                    st_release(&sync->resume, ++s_resume);
                }
            }
            s_level = level + 1u;
            s_par = par ^ 1u;
            s_cnt = (uint32_t)ncnt;
            s_edges = nedges;
            s_done = more ? 0u : 1u;
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
        ctl->level = s_level;
        ctl->step = s_level;
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
