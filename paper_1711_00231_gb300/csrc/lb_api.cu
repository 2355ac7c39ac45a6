// Host implementation of the C ABI declared in include/lb.h.
#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "lb_internal.cuh"

using namespace lbk;

namespace {

thread_local std::string t_err;

std::mutex g_alloc_mu;
void *(*g_alloc_fn)(size_t, void *) = nullptr;
void (*g_free_fn)(void *, void *) = nullptr;
void *g_alloc_ctx = nullptr;

lb_status fail(lb_status s, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    t_err = buf;
    return s;
}

#define LB_CU(call)                                                                                      \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess)                                                                           \
            return fail(e_ == cudaErrorMemoryAllocation ? LB_ERR_OOM : LB_ERR_CUDA, "%s failed: %s (%s:%d)", \
                        #call, cudaGetErrorString(e_), __FILE__, __LINE__);                              \
    } while (0)

#define LB_TRY(expr)                \
    do {                            \
        lb_status s_ = (expr);      \
        if (s_ != LB_OK) return s_; \
    } while (0)

struct Allocator {
    void *(*alloc_fn)(size_t, void *) = nullptr;
    void (*free_fn)(void *, void *) = nullptr;
    void *ctx = nullptr;

    cudaError_t alloc(void **p, size_t bytes) const {
        if (bytes == 0) bytes = 16;
        if (alloc_fn) {
            *p = alloc_fn(bytes, ctx);
            return *p ? cudaSuccess : cudaErrorMemoryAllocation;
        }
        return cudaMalloc(p, bytes);
    }
    void release(void *p) const {
        if (!p) return;
        if (free_fn) free_fn(p, ctx);
        else cudaFree(p);
    }
};

// Restores the caller's current device on scope exit.
struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

constexpr int kStrategies = 7;
// WD, fast levels: entries per CTA segment (lists of small graphs are short:
// less to allocate in the first query), and 16-byte list entries in all, one
// of them to align the rest (a custom allocator may return any address)
int32_t fast_seg_cap(int64_t n) { return n <= 32768 ? 256 : kFastSeg; }
int64_t fast_entries(int64_t n) { return 2 * (int64_t)kFastTeam * fast_seg_cap(n) + 1; }

// Default small_edges.
#ifndef LB_SMALL_EDGES_DEFAULT
#define LB_SMALL_EDGES_DEFAULT 16384
#endif

constexpr int32_t LB_TUNE_BOTH = 2;  // lb_autotune: time a BFS and an SSSP per source

bool is_ep(int s) { return s == LB_EP || s == LB_EP_NOCHUNK; }

// tile-start entries a list needs: one per kTileGrain worklist edges
int64_t round_tiles(int64_t m) { return m / kTileGrain + 2; }

// words of one half of the visited / queued bitmap: one bit per vertex,
// rounded up to whole 16-byte groups
int64_t bitmap_words(int64_t n) { return ((n + 31) / 32 + 3) / 4 * 4; }

// Bitmap placements (lb_options::bitmap_place): the bitmap starts
// place * step words into its allocation, step = min(1 MiB, one half
// rounded up to 4 KiB), and the allocation carries kBitmapPlaces - 1 steps
// of slack.  The bitmap is read at random by every SM; measured on GB300,
// R-MAT scale 24 BFS takes 1.80 to 1.94 ms per query depending only on
// where it starts, so the autotuner times the placements.
constexpr int32_t kBitmapPlaces = 8;
int64_t bitmap_step_words(int64_t n) {
    const int64_t half4k = (bitmap_words(n) + 1023) / 1024 * 1024;
    return half4k < (int64_t)(1 << 18) ? half4k : (int64_t)(1 << 18);
}
int64_t bitmap_alloc_words(int64_t n) { return 2 * bitmap_words(n) + (kBitmapPlaces - 1) * bitmap_step_words(n); }

}  // namespace

struct lb_graph {
    int device = 0;
    int sms = 0;
    int64_t n = 0, m = 0;
    bool weighted = false;
    bool zero_weight = false;
    int64_t max_degree = 0;
    Allocator al;
    std::mutex mu;
    lb_options opt{};
    int64_t resident = 0;

    // CSR
    int64_t *off = nullptr;
    int32_t *col = nullptr;
    uint32_t *w = nullptr;

    // workspace (lazily allocated)
    Ctl *ctl = nullptr;
    uint32_t *bitmap = nullptr;  // bitmap_alloc_words(n): two halves (BFS visited bits / SSSP queued bits) + placement slack
    int4 *fast_seg = nullptr;    // WD: list segments of the fast levels (fast_entries)
    uint32_t *out_internal = nullptr;  // result buffer of host-output queries
    int32_t *par_internal = nullptr;
    NodeList lists[2]{};
    NodeList subs[2]{};
    int64_t lists_bytes = 0, subs_bytes = 0;  // of the two pairs' allocations
    int64_t list_cap = 0;
    int64_t tile_cap = 0;
    bool have_tiles = false;
    bool have_subs = false;
    int32_t *elist[2]{};
    int64_t elist_cap = 0;
    int32_t *coo_src = nullptr;
    int32_t *child_first = nullptr;         // NS_PHYS split map (n)
    int32_t *parent_of = nullptr;           // NS_PHYS (children)
    uint32_t *child_dist = nullptr;         // NS_PHYS (children)
    unsigned long long *ns_sums = nullptr;  // NS_PHYS build scratch (n / 1024 + 1)
    int64_t phys_mdt = -1;                  // MDT the split map was built for
    int64_t phys_children = 0;
    unsigned long long *scratch = nullptr;  // MDT histogram / counters (4097 words)
    int64_t *dres = nullptr;                // device results (4 words)
    int64_t *hres = nullptr;                // pinned host mirror
    uint32_t *hflag = nullptr;              // pinned host word for the host loop

    int64_t mdt = -1;          // computed with opt.hist_bins (or override)
    int64_t mdt_bins = -1;
    int64_t mdt_maxdeg = 0;
    int32_t mdt_bin = 0;
    int64_t ns_children = -1;  // at mdt

    cudaGraphExec_t exec[kStrategies][2]{};
    int grid[kStrategies][2]{};
    int query_grid[2]{};        // whole-query WD launch (0: not yet computed)
    uint32_t query_number = 0;  // whole-query WD launches so far
    bool team_picked = false;   // the SMs of its small-list team are chosen

    // batched host-output queries: the second result buffer, one error
    // word per query, the copy stream and the events that order each
    // buffer's copy against its next query
    uint32_t *out_internal2 = nullptr;
    uint32_t *batch_err = nullptr;
    int64_t batch_err_cap = 0;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_comp[2]{}, ev_copy[2]{};

    cudaStream_t stream = nullptr;  // capture stream and host-output query stream
    cudaEvent_t ev_start = nullptr, ev_stop = nullptr, ev_done = nullptr;
    cudaStream_t last_stream = nullptr;
    bool has_last = false;
    int last_strategy = -1;

    template <class T>
    lb_status alloc(T **p, int64_t count) {
        void *q = nullptr;
        const size_t bytes = (size_t)(count > 0 ? count : 1) * sizeof(T);
        cudaError_t e = al.alloc(&q, bytes);
        if (e != cudaSuccess)
            return fail(LB_ERR_OOM, "device allocation of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
        *p = (T *)q;
        resident += (int64_t)bytes;
        return LB_OK;
    }
    template <class T>
    void release(T *&p, int64_t count) {
        if (!p) return;
        al.release((void *)p);
        resident -= (int64_t)((size_t)(count > 0 ? count : 1) * sizeof(T));
        p = nullptr;
    }
};

namespace {

lb_options default_options() {
    lb_options o;
    memset(&o, 0, sizeof(o));
    o.hist_bins = 10;
    o.mdt_override = 0;
    o.hp_threshold = 1024;
    o.hp_mode = 0;
    o.hp_warp_max = 4096;
    o.ns_mode = 0;
    o.thread_max = 32;
    o.hp_depth = 1;
    o.small_edges = LB_SMALL_EDGES_DEFAULT;
    o.loop_mode = 0;
    o.wd_tile = 8192;
    o.ctas_per_sm = 0;
    return o;
}

lb_status normalise_options(const lb_options *in, lb_options *out) {
    lb_options d = default_options();
    lb_options o = *in;
    if (o.hist_bins == 0) o.hist_bins = d.hist_bins;
    if (o.hp_threshold == 0) o.hp_threshold = d.hp_threshold;
    if (o.hp_warp_max == 0) o.hp_warp_max = d.hp_warp_max;
    if (o.hp_mode != 0 && o.hp_mode != 1) return fail(LB_ERR_ARG, "hp_mode must be 0 or 1");
    if (o.hp_warp_max < 32) return fail(LB_ERR_ARG, "hp_warp_max must be >= 32");
    if (o.thread_max == 0) o.thread_max = d.thread_max;
    if (o.hp_depth == 0) o.hp_depth = d.hp_depth;
    if (o.ns_mode != 0 && o.ns_mode != 1) return fail(LB_ERR_ARG, "ns_mode must be 0 or 1");
    if (o.thread_max < 1 || o.thread_max > 1024) return fail(LB_ERR_ARG, "thread_max must be in [1, 1024]");
    if (o.hp_depth < 1 || o.hp_depth > 8) return fail(LB_ERR_ARG, "hp_depth must be in [1, 8]");
    if (o.small_edges < 0 || o.small_edges > (1 << 24)) return fail(LB_ERR_ARG, "small_edges must be in [0, 2^24]");
    if (o.test_barrier_skip < 0 || o.test_barrier_skip > kTestMax) return fail(LB_ERR_ARG, "test_barrier_skip must be 0..%d", kTestMax);
    if (o.bitmap_place < 0 || o.bitmap_place >= kBitmapPlaces) return fail(LB_ERR_ARG, "bitmap_place must be in [0, 7]");
    for (int i = 0; i < 2; ++i)
        if (o.reserved[i] != 0) return fail(LB_ERR_ARG, "reserved option fields must be 0");
    if (o.wd_tile == 0) o.wd_tile = d.wd_tile;
    if (o.hist_bins < 1 || o.hist_bins > 4096) return fail(LB_ERR_ARG, "hist_bins must be in [1, 4096]");
    if (o.mdt_override < 0) return fail(LB_ERR_ARG, "mdt_override must be >= 0");
    if (o.loop_mode != 0 && o.loop_mode != 1) return fail(LB_ERR_ARG, "loop_mode must be 0 or 1");
    if (o.wd_tile < 256 || o.wd_tile > 32768 || o.wd_tile % 256) return fail(LB_ERR_ARG, "wd_tile must be a multiple of 256 in [256, 32768]");
    if (o.ctas_per_sm < 0 || o.ctas_per_sm > 32) return fail(LB_ERR_ARG, "ctas_per_sm must be in [0, 32]");
    *out = o;
    return LB_OK;
}

// Waits for the last query so buffers can be freed or reallocated safely.
void quiesce(lb_graph *g) {
    if (g->has_last) cudaEventSynchronize(g->ev_done);
    cudaStreamSynchronize(g->stream);
}

void drop_execs(lb_graph *g) {
    for (int s = 0; s < kStrategies; ++s)
        for (int k = 0; k < 2; ++k)
            if (g->exec[s][k]) {
                cudaGraphExecDestroy(g->exec[s][k]);
                g->exec[s][k] = nullptr;
            }
}

// Both buffers of a worklist live in one allocation, each piece on a
// 256-byte step of it: cudaMalloc takes about 30 us from 1 MiB up, and a
// first query would make eight of them per pair.
int64_t step256(int64_t bytes) { return (bytes + 255) / 256 * 256; }

void free_lists(lb_graph *g, NodeList *L, int64_t &bytes) {
    unsigned char *block = (unsigned char *)L[0].v;
    g->release(block, bytes);
    L[0] = L[1] = NodeList{};
    bytes = 0;
}

lb_status alloc_lists(lb_graph *g, NodeList *L, int64_t &bytes, int64_t cap, int64_t tcap, bool tiles) {
    const int64_t entry = step256(4 * (cap > 0 ? cap : 1)), scan = step256(4 * (cap + 1));
    const int64_t ts = tiles ? step256(4 * tcap) : 0, one = 2 * entry + scan + ts;
    unsigned char *block = nullptr;
    LB_TRY(g->alloc(&block, 2 * one));
    bytes = 2 * one;
    for (int b = 0; b < 2; ++b) {
        unsigned char *q = block + b * one;
        L[b].v = (int32_t *)q;
        L[b].beg = (int32_t *)(q + entry);
        L[b].scan = (int32_t *)(q + 2 * entry);
        L[b].tstart = tiles ? (int32_t *)(q + 2 * entry + scan) : nullptr;
    }
    return LB_OK;
}

void free_workspace(lb_graph *g) {
    drop_execs(g);
    g->release(g->ctl, 1);
    g->team_picked = false;
    g->release(g->bitmap, bitmap_alloc_words(g->n));
    g->release(g->fast_seg, fast_entries(g->n));
    g->release(g->out_internal, g->n);
    g->release(g->out_internal2, g->n);
    g->release(g->batch_err, g->batch_err_cap);
    g->batch_err_cap = 0;
    g->release(g->par_internal, g->n);
    free_lists(g, g->lists, g->lists_bytes);
    free_lists(g, g->subs, g->subs_bytes);
    g->list_cap = 0;
    g->have_tiles = false;
    g->have_subs = false;
    for (int b = 0; b < 2; ++b) g->release(g->elist[b], g->elist_cap);
    g->elist_cap = 0;
    g->release(g->coo_src, g->m);
    g->release(g->child_first, g->n);
    g->release(g->parent_of, g->phys_children);
    g->release(g->child_dist, g->phys_children);
    g->release(g->ns_sums, g->n / 1024 + 1);
    g->phys_mdt = -1;
    g->phys_children = 0;
}

// MDT with the graph's options (histogram on the device, cached).
lb_status ensure_mdt(lb_graph *g) {
    const int64_t bins = g->opt.hist_bins;
    if (g->opt.mdt_override > 0) {
        if (g->mdt != g->opt.mdt_override) {
            g->mdt = g->opt.mdt_override;
            g->mdt_bins = -1;
            g->ns_children = -1;
        }
    } else if (g->mdt < 0 || g->mdt_bins != bins) {
        GraphDev gd{g->off, g->col, g->w, g->n, g->m};
        LB_CU(launch_mdt(gd, (int32_t)bins, g->scratch, g->dres, g->stream));
        LB_CU(cudaMemcpyAsync(g->hres, g->dres, 3 * sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream));
        LB_CU(cudaStreamSynchronize(g->stream));
        g->mdt = g->hres[0] > 0 ? g->hres[0] : 1;
        g->mdt_maxdeg = g->hres[1];
        g->mdt_bin = (int32_t)g->hres[2];
        g->mdt_bins = bins;
        g->ns_children = -1;
    }
    if (g->ns_children < 0) {
        GraphDev gd{g->off, g->col, g->w, g->n, g->m};
        LB_CU(launch_ns_count(gd, (int32_t)g->mdt, g->scratch, g->stream));
        LB_CU(cudaMemcpyAsync(g->hres, g->scratch, sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream));
        LB_CU(cudaStreamSynchronize(g->stream));
        g->ns_children = g->hres[0];
    }
    return LB_OK;
}

int64_t node_list_cap(const lb_graph *g, int s) {
    return (s == LB_NS || s == LB_NS_PHYS) ? g->n + (g->ns_children > 0 ? g->ns_children : 0) : g->n;
}

// Allocates what strategy s needs; any reallocation invalidates the cached
// device loops (their kernel parameters hold the pointers).
lb_status ensure_workspace(lb_graph *g, int s) {
    // each piece on its own, so an attempt after a failed allocation
    // completes what the earlier one left
    if (!g->ctl) {
        LB_TRY(g->alloc(&g->ctl, 1));
        LB_CU(cudaMemsetAsync(g->ctl, 0, sizeof(Ctl), g->stream));
    }
    if (!g->bitmap) LB_TRY(g->alloc(&g->bitmap, bitmap_alloc_words(g->n)));
    if (s == LB_NS || s == LB_NS_PHYS || s == LB_HP) LB_TRY(ensure_mdt(g));
    if (s == LB_NS_PHYS && g->phys_mdt != g->mdt) {
        quiesce(g);
        drop_execs(g);
        g->release(g->child_first, g->n);
        g->release(g->parent_of, g->phys_children);
        g->release(g->child_dist, g->phys_children);
        g->phys_children = g->ns_children;
        LB_TRY(g->alloc(&g->child_first, g->n));
        LB_TRY(g->alloc(&g->parent_of, g->phys_children));
        LB_TRY(g->alloc(&g->child_dist, g->phys_children));
        if (!g->ns_sums) LB_TRY(g->alloc(&g->ns_sums, g->n / 1024 + 1));
        GraphDev gd{g->off, g->col, g->w, g->n, g->m};
        LB_CU(launch_ns_phys_build(gd, (int32_t)g->mdt, g->child_first, g->parent_of, g->ns_sums, g->stream));
        g->phys_mdt = g->mdt;
    }
    if (is_ep(s)) {
        if (!g->coo_src) {
            LB_TRY(g->alloc(&g->coo_src, g->m));
            GraphDev gd{g->off, g->col, g->w, g->n, g->m};
            LB_CU(launch_coo_build(gd, g->coo_src, g->stream));
        }
        if (g->elist_cap < g->m || !g->elist[0] || !g->elist[1]) {
            quiesce(g);
            drop_execs(g);
            for (int b = 0; b < 2; ++b) g->release(g->elist[b], g->elist_cap);
            g->elist_cap = g->m > 0 ? g->m : 1;
            for (int b = 0; b < 2; ++b) LB_TRY(g->alloc(&g->elist[b], g->elist_cap));
        }
        return LB_OK;
    }
    const int64_t cap = node_list_cap(g, s);
    const bool tiles = (s == LB_WD || s == LB_HP);
    const int64_t tcap = round_tiles(g->m);
    if (g->list_cap < cap || (tiles && (!g->have_tiles || g->tile_cap != tcap))) {
        quiesce(g);
        drop_execs(g);
        free_lists(g, g->lists, g->lists_bytes);
        const int64_t newcap = cap > g->list_cap ? cap : g->list_cap;
        const bool want_tiles = tiles || g->have_tiles;
        if (g->have_subs) {
            free_lists(g, g->subs, g->subs_bytes);
            g->have_subs = false;
        }
        g->list_cap = 0;
        g->have_tiles = false;
        g->tile_cap = tcap;
        LB_TRY(alloc_lists(g, g->lists, g->lists_bytes, newcap, tcap, want_tiles));
        g->list_cap = newcap;
        g->have_tiles = want_tiles;
    }
    if (s == LB_WD && !g->fast_seg) LB_TRY(g->alloc(&g->fast_seg, fast_entries(g->n)));
    // only the whole-query launch has a team (its pick takes an idle GPU: a
    // CTA with 160 KB of shared memory per SM)
    if (s == LB_WD && g->opt.loop_mode == 0 && !g->team_picked) {
        LB_CU(launch_team_pick(g->ctl, g->sms, g->stream));
        g->team_picked = true;
    }
    if (s == LB_HP && !g->have_subs) {
        quiesce(g);
        drop_execs(g);
        free_lists(g, g->subs, g->subs_bytes);
        LB_TRY(alloc_lists(g, g->subs, g->subs_bytes, g->n, g->tile_cap, true));
        g->have_subs = true;
    }
    return LB_OK;
}

StepParams make_params(const lb_graph *g, int s) {
    StepParams p;
    memset(&p, 0, sizeof(p));
    p.g = GraphDev{g->off, g->col, g->w, g->n, g->m};
    p.ctl = g->ctl;
    for (int b = 0; b < 2; ++b) {
        p.lists[b] = g->lists[b];
        p.subs[b] = g->subs[b];
        p.elist[b] = g->elist[b];
    }
    p.coo_src = g->coo_src;
    p.child_first = g->child_first;
    p.parent_of = g->parent_of;
    p.child_dist = g->child_dist;
    p.n_children = g->phys_children;
    p.bitmap = g->bitmap + (int64_t)g->opt.bitmap_place * bitmap_step_words(g->n);
    p.bm_words = bitmap_words(g->n);
    p.list_cap = s == LB_HP ? (g->list_cap < g->n ? g->list_cap : g->n) : g->list_cap;
    p.tile_cap = g->tile_cap;
    p.elist_cap = g->elist_cap;
    p.tile = g->opt.wd_tile;
    p.mdt = (int32_t)(g->mdt > 0 ? g->mdt : 1);
    p.hp_threshold = g->opt.hp_threshold;
    p.hp_mode = g->opt.hp_mode;
    p.hp_warp_max = g->opt.hp_warp_max;
    p.thread_max = g->opt.thread_max;
    p.ns_mode = g->opt.ns_mode;
    p.hp_depth = g->opt.hp_depth;
    p.hist_bins = g->opt.hist_bins;
    p.small_edges = s == LB_WD ? g->opt.small_edges : 0;
    p.test_barrier_skip = g->opt.test_barrier_skip;
    p.strategy = s;
    p.use_cond = 0;
    return p;
}

int step_grid(lb_graph *g, int s, bool sssp) {
    int &gr = g->grid[s][sssp ? 1 : 0];
    if (gr == 0) {
        int occ = step_blocks_per_sm(s, sssp, g->opt.ns_mode);
        if (g->opt.ctas_per_sm > 0 && g->opt.ctas_per_sm < occ) occ = g->opt.ctas_per_sm;
        gr = occ * g->sms;
    }
    return gr;
}

// Grid of the whole-query WD launch: every CTA resident (a cooperative
// launch), at most ctas_per_sm per SM.  BFS on a small graph is launches,
// barriers and list ends more than edges, and these get cheaper with fewer
// CTAs: 5 / 4 / 3 per SM took, at 64K edges (R-MAT scale 12) 48.2 / 46.7 /
// 46.7 us, 400K (Erdos-Renyi) 94.8 / 89.5 / 87.7, 2M (R-MAT 17) 73.2 / 72.0 /
// 69.3, 2M (Erdos-Renyi) 132 / 127 / 130, 4M (R-MAT 18) 90.6 / 85.3 / 82.7, 4M
// (Erdos-Renyi) 164 / 164 / 171, 8M 125 / 125 / 128, 16M (R-MAT 20) 134 / 137 /
// 156 us.  SSSP (4 per SM) gained nothing from 3.
int query_grid(lb_graph *g, bool sssp) {
    int &gr = g->query_grid[sssp ? 1 : 0];
    if (gr == 0) {
        int occ = query_wd_blocks_per_sm(sssp);
        const int want = sssp || g->m > (1 << 23) ? occ : g->m > (1 << 21) ? 4 : 3;
        if (g->opt.ctas_per_sm == 0 && want < occ) occ = want;
        if (g->opt.ctas_per_sm > 0 && g->opt.ctas_per_sm < occ) occ = g->opt.ctas_per_sm;
        gr = occ * g->sms;
    }
    return gr;
}

// CTAs of the persistent small-list launch (all resident: a cooperative launch).
int small_grid(const lb_graph *g) { return g->sms * small_ctas_per_sm(); }

// HP with a hierarchy deeper than one list runs k_hp_mdt before every step.
bool hp_needs_mdt_kernel(const lb_graph *g, int s) { return s == LB_HP && g->opt.hp_depth > 1; }

// Captures one step launch into the body of a conditional WHILE node.
lb_status build_exec(lb_graph *g, int s, bool sssp, cudaGraphExec_t *out) {
    cudaGraph_t graph = nullptr;
    LB_CU(cudaGraphCreate(&graph, 0));
    cudaGraphConditionalHandle h;
    cudaError_t e = cudaGraphConditionalHandleCreate(&h, graph, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) {
        cudaGraphDestroy(graph);
        return fail(LB_ERR_CUDA, "cudaGraphConditionalHandleCreate: %s", cudaGetErrorString(e));
    }
    // cudaGraphNodeParams holds a union with a deleted default constructor:
    // build it in zeroed raw storage.
    alignas(cudaGraphNodeParams) unsigned char cp_store[sizeof(cudaGraphNodeParams)];
    memset(cp_store, 0, sizeof(cp_store));
    cudaGraphNodeParams &cp = *reinterpret_cast<cudaGraphNodeParams *>(cp_store);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &cp);
    if (e != cudaSuccess) {
        cudaGraphDestroy(graph);
        return fail(LB_ERR_CUDA, "cudaGraphAddNode(conditional): %s", cudaGetErrorString(e));
    }
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    StepParams p = make_params(g, s);
    p.use_cond = 1;
    p.cond = h;
    const int grid = step_grid(g, s, sssp);
    e = cudaStreamBeginCaptureToGraph(g->stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaError_t le = cudaSuccess;
        if (hp_needs_mdt_kernel(g, s)) le = launch_hp_mdt(p, 2 * g->sms, g->stream);
        if (le == cudaSuccess) le = launch_step(s, sssp, p, grid, g->stream);
        cudaGraph_t captured = nullptr;
        e = cudaStreamEndCapture(g->stream, &captured);
        if (le != cudaSuccess) e = le;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(out, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, "building the device loop failed: %s", cudaGetErrorString(e));
    return LB_OK;
}

lb_status status_from_error(uint32_t e) {
    if (e & (kErrCapacity | kErrShape | kErrBounds))
        return fail(LB_ERR_INTERNAL, "device consistency check failed (0x%x)", e);
    if (e & (kErrIterCap | kErrDeadline)) return fail(LB_ERR_TIMEOUT, "iteration cap or time limit reached (0x%x)", e);
    if (e & kErrOverflow) return fail(LB_ERR_OVERFLOW, "a shortest distance does not fit in 32 bits");
    return LB_OK;
}

// One launch runs the whole query (WD, device loop).
bool whole_query(const lb_graph *g, int s) { return g->opt.loop_mode == 0 && (s == LB_WD || s == LB_AUTO); }

lb_status run_query(lb_graph *g, int kind, int s, int32_t src, void *out_dev, int32_t *parents_dev,
                    cudaStream_t st, uint32_t *prev_error = nullptr) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    if (src < 0 || (int64_t)src >= g->n) return fail(LB_ERR_ARG, "source %d out of range [0, %lld)", src, (long long)g->n);
    if (s == LB_AUTO) s = LB_WD;
    if (s < 0 || s >= kStrategies) return fail(LB_ERR_ARG, "unknown strategy %d", s);
    if (kind == LB_KIND_SSSP && !g->weighted) return fail(LB_ERR_UNSUPPORTED, "SSSP needs a weighted graph");
    if (!out_dev) return fail(LB_ERR_ARG, "output buffer is NULL");
    if (parents_dev && kind == LB_KIND_SSSP && g->zero_weight)
        return fail(LB_ERR_UNSUPPORTED, "parents for graphs with zero-weight edges are not supported");
    const bool sssp = kind == LB_KIND_SSSP;
    LB_TRY(ensure_workspace(g, s));
    if (g->has_last && g->last_stream != st) LB_CU(cudaStreamWaitEvent(st, g->ev_done, 0));
    if (st != g->stream) {  // workspace set-up ran on g->stream
        LB_CU(cudaEventRecord(g->ev_done, g->stream));
        LB_CU(cudaStreamWaitEvent(st, g->ev_done, 0));
    }
    StepParams p = make_params(g, s);
    const uint32_t max_levels = (uint32_t)(g->n + 1 < 0xFFFFFFF0ll ? g->n + 1 : 0xFFFFFFF0ll);
    const uint64_t max_steps = (uint64_t)1 << 40;
    const uint64_t time_limit_ns = (uint64_t)120 * 1000000000ull;  // safety net; no query comes close
    const bool whole = whole_query(g, s);
    const int grid = whole ? query_grid(g, sssp) : step_grid(g, s, sssp);
    LB_CU(cudaEventRecord(g->ev_start, st));
    if (whole) {
        QueryArgs a;
        a.status = (uint32_t *)out_dev;
        a.src = src;
        a.max_levels = sssp ? threshold_levels(g->n) : max_levels;
        a.time_limit_ns = p.test_barrier_skip == kTestTeamGone ? 0 : time_limit_ns;
        a.number = g->query_number;
        a.seg_cap = fast_seg_cap(g->n);
        a.far_shift = far_shift(g->n);
        a.prev_error = prev_error;
        a.team = kFastTeam < grid ? kFastTeam : grid;
        a.fast_seg = a.team == kFastTeam ? (int4 *)(((uintptr_t)g->fast_seg + 15u) & ~(uintptr_t)15u) : nullptr;
        LB_CU(launch_query_wd(sssp, p, a, grid, st));
        ++g->query_number;
        if (parents_dev) LB_CU(launch_parents(p, sssp, parents_dev, st));
        LB_CU(cudaEventRecord(g->ev_stop, st));
        LB_CU(cudaEventRecord(g->ev_done, st));
        g->last_stream = st;
        g->has_last = true;
        g->last_strategy = s;
        return LB_OK;
    }
    LB_CU(launch_init(p, src, (uint32_t *)out_dev, kind, max_levels, max_steps, time_limit_ns, grid, st));
    if (g->opt.loop_mode == 0) {
        cudaGraphExec_t &ex = g->exec[s][sssp ? 1 : 0];
        if (!ex) LB_TRY(build_exec(g, s, sssp, &ex));
        LB_CU(cudaGraphLaunch(ex, st));
    } else {
        for (;;) {
            if (hp_needs_mdt_kernel(g, s)) LB_CU(launch_hp_mdt(p, 2 * g->sms, st));
            if (p.small_edges > 0) LB_CU(launch_small_levels(sssp, p, small_grid(g), st));
            LB_CU(launch_step(s, sssp, p, grid, st));
            LB_CU(cudaMemcpyAsync(g->hflag, &g->ctl->active, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
            LB_CU(cudaStreamSynchronize(st));
            if (!*g->hflag) break;
        }
    }
    if (sssp) LB_CU(launch_finish_query(p, st));
    if (parents_dev) LB_CU(launch_parents(p, sssp, parents_dev, st));
    LB_CU(cudaEventRecord(g->ev_stop, st));
    LB_CU(cudaEventRecord(g->ev_done, st));
    g->last_stream = st;
    g->has_last = true;
    g->last_strategy = s;
    return LB_OK;
}

lb_status read_ctl(lb_graph *g, Ctl *h) {
    LB_CU(cudaEventSynchronize(g->ev_done));
    LB_CU(cudaMemcpy(h, g->ctl, offsetof(Ctl, trace), cudaMemcpyDeviceToHost));
    return LB_OK;
}

lb_status host_query(lb_graph *g, int kind, lb_strategy s, int32_t src, void *host_out) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    if (!host_out) return fail(LB_ERR_ARG, "output buffer is NULL");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    if (!g->out_internal) LB_TRY(g->alloc(&g->out_internal, g->n));
    LB_TRY(run_query(g, kind, s, src, g->out_internal, nullptr, g->stream));
    LB_CU(cudaMemcpyAsync(host_out, g->out_internal, sizeof(uint32_t) * (size_t)g->n, cudaMemcpyDeviceToHost,
                          g->stream));
    LB_CU(cudaStreamSynchronize(g->stream));
    Ctl h;
    LB_TRY(read_ctl(g, &h));
    return status_from_error(h.error);
}

// k host-output queries with the copy of query i's result overlapping query
// i + 1: results alternate between two device buffers; query i's copy runs
// on copy_stream after query i (ev_comp), and query i + 2, which reuses the
// buffer, waits for that copy (ev_copy).  Each query's error word is kept
// on the device (by the next query's set-up where one launch runs a query,
// else and for the last query by a copy) and read once at the end.  Every copy has
// finished before the call returns, on success or error.
lb_status host_query_batch(lb_graph *g, int kind, lb_strategy s, const int32_t *srcs, int64_t k, void *host_out) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    if (k < 0) return fail(LB_ERR_ARG, "query count %lld is negative", (long long)k);
    if (k == 0) return LB_OK;
    if (!srcs || !host_out) return fail(LB_ERR_ARG, "NULL argument");
    for (int64_t i = 0; i < k; ++i)
        if (srcs[i] < 0 || (int64_t)srcs[i] >= g->n)
            return fail(LB_ERR_ARG, "source %d of query %lld out of range [0, %lld)", srcs[i], (long long)i,
                        (long long)g->n);
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    if (!g->out_internal) LB_TRY(g->alloc(&g->out_internal, g->n));
    if (!g->out_internal2) LB_TRY(g->alloc(&g->out_internal2, g->n));
    if (g->batch_err_cap < k) {
        g->release(g->batch_err, g->batch_err_cap);
        g->batch_err_cap = 0;
        const int64_t cap = (k + 1023) / 1024 * 1024;
        LB_TRY(g->alloc(&g->batch_err, cap));
        g->batch_err_cap = cap;
    }
    if (!g->copy_stream) LB_CU(cudaStreamCreateWithFlags(&g->copy_stream, cudaStreamNonBlocking));
    for (int b = 0; b < 2; ++b) {
        if (!g->ev_comp[b]) LB_CU(cudaEventCreateWithFlags(&g->ev_comp[b], cudaEventDisableTiming));
        if (!g->ev_copy[b]) LB_CU(cudaEventCreateWithFlags(&g->ev_copy[b], cudaEventDisableTiming));
    }
    uint32_t *buf[2] = {g->out_internal, g->out_internal2};
    const size_t bytes = sizeof(uint32_t) * (size_t)g->n;
    lb_status st = LB_OK;
    cudaError_t e = cudaSuccess;
    for (int64_t i = 0; i < k && st == LB_OK && e == cudaSuccess; ++i) {
        const int b = (int)(i & 1);
        if (i >= 2) e = cudaStreamWaitEvent(g->stream, g->ev_copy[b], 0);
        if (e != cudaSuccess) break;
        st = run_query(g, kind, s, srcs[i], buf[b], nullptr, g->stream, i > 0 ? g->batch_err + i - 1 : nullptr);
        if (st != LB_OK) break;
        if (!whole_query(g, s) || i == k - 1)
            e = cudaMemcpyAsync(g->batch_err + i, &g->ctl->error, sizeof(uint32_t), cudaMemcpyDeviceToDevice, g->stream);
        if (e == cudaSuccess) e = cudaEventRecord(g->ev_comp[b], g->stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(g->copy_stream, g->ev_comp[b], 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync((char *)host_out + (size_t)i * bytes, buf[b], bytes, cudaMemcpyDeviceToHost,
                                g->copy_stream);
        if (e == cudaSuccess) e = cudaEventRecord(g->ev_copy[b], g->copy_stream);
    }
    const cudaError_t e1 = cudaStreamSynchronize(g->copy_stream);
    const cudaError_t e2 = cudaStreamSynchronize(g->stream);
    if (st != LB_OK) return st;
    if (e == cudaSuccess) e = e1 != cudaSuccess ? e1 : e2;
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, "batched query failed: %s", cudaGetErrorString(e));
    std::vector<uint32_t> errs((size_t)k);
    LB_CU(cudaMemcpy(errs.data(), g->batch_err, sizeof(uint32_t) * (size_t)k, cudaMemcpyDeviceToHost));
    for (int64_t i = 0; i < k; ++i) {
        if (!errs[(size_t)i]) continue;
        const lb_status q = status_from_error(errs[(size_t)i]);
        if (q != LB_OK) {
            const std::string msg = lb_last_error();
            return fail(q, "query %lld (source %d): %s", (long long)i, srcs[i], msg.c_str());
        }
    }
    return LB_OK;
}

lb_status create_common(lb_graph *g) {
    LB_CU(cudaGetDevice(&g->device));
    LB_CU(cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, g->device));
    LB_CU(cudaStreamCreateWithFlags(&g->stream, cudaStreamNonBlocking));
    LB_CU(cudaEventCreate(&g->ev_start));
    LB_CU(cudaEventCreate(&g->ev_stop));
    LB_CU(cudaEventCreateWithFlags(&g->ev_done, cudaEventDisableTiming));
    LB_CU(cudaMallocHost((void **)&g->hres, 8 * sizeof(int64_t)));
    LB_CU(cudaMallocHost((void **)&g->hflag, sizeof(uint32_t)));
    LB_TRY(g->alloc(&g->scratch, 4097));
    LB_TRY(g->alloc(&g->dres, 4));
    return LB_OK;
}

void destroy_graph(lb_graph *g) {
    if (!g) return;
    DeviceGuard dg(g->device);
    if (g->stream) cudaStreamSynchronize(g->stream);
    if (g->has_last) cudaEventSynchronize(g->ev_done);
    free_workspace(g);
    g->release(g->scratch, 4097);
    g->release(g->dres, 4);
    g->release(g->off, g->n + 1);
    g->release(g->col, g->m);
    g->release(g->w, g->m);
    if (g->hres) cudaFreeHost(g->hres);
    if (g->hflag) cudaFreeHost(g->hflag);
    if (g->ev_start) cudaEventDestroy(g->ev_start);
    if (g->ev_stop) cudaEventDestroy(g->ev_stop);
    if (g->ev_done) cudaEventDestroy(g->ev_done);
    for (int b = 0; b < 2; ++b) {
        if (g->ev_comp[b]) cudaEventDestroy(g->ev_comp[b]);
        if (g->ev_copy[b]) cudaEventDestroy(g->ev_copy[b]);
    }
    if (g->copy_stream) cudaStreamDestroy(g->copy_stream);
    if (g->stream) cudaStreamDestroy(g->stream);
    delete g;
}

lb_graph *new_graph(int64_t n, int64_t m, bool weighted) {
    lb_graph *g = new (std::nothrow) lb_graph();
    if (!g) return nullptr;
    g->n = n;
    g->m = m;
    g->weighted = weighted;
    g->opt = default_options();
    std::lock_guard<std::mutex> lk(g_alloc_mu);
    g->al.alloc_fn = g_alloc_fn;
    g->al.free_fn = g_free_fn;
    g->al.ctx = g_alloc_ctx;
    return g;
}

}  // namespace

void lbk::set_last_error(const char *msg) { t_err = msg; }

void lbk::graph_device_arrays(const lb_graph *g, const int64_t **off, const int32_t **col, const uint32_t **w) {
    *off = g->off;
    *col = g->col;
    *w = g->w;
}

extern "C" {

const char *lb_last_error(void) { return t_err.c_str(); }

const char *lb_version(void) { return "lb 1.0 (sm_103a)"; }

lb_status lb_set_allocator(void *(*alloc_fn)(size_t, void *), void (*free_fn)(void *, void *), void *ctx) {
    if ((alloc_fn == nullptr) != (free_fn == nullptr)) return fail(LB_ERR_ARG, "give both allocator functions or neither");
    std::lock_guard<std::mutex> lk(g_alloc_mu);
    g_alloc_fn = alloc_fn;
    g_free_fn = free_fn;
    g_alloc_ctx = ctx;
    return LB_OK;
}

lb_status lb_graph_create(const int64_t *offsets, const int32_t *cols, const uint32_t *weights, int64_t n, int64_t m,
                          lb_graph **out) {
    if (!out) return fail(LB_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!offsets || (m > 0 && !cols)) return fail(LB_ERR_ARG, "offsets / cols is NULL");
    if (n < 1 || n >= ((int64_t)1 << 31)) return fail(LB_ERR_ARG, "n must be in [1, 2^31)");
    if (m < 0 || m >= ((int64_t)1 << 31)) return fail(LB_ERR_ARG, "m must be in [0, 2^31)");
    if (offsets[0] != 0) return fail(LB_ERR_ARG, "offsets[0] must be 0");
    if (offsets[n] != m) return fail(LB_ERR_ARG, "offsets[n] = %lld but m = %lld", (long long)offsets[n], (long long)m);
    int64_t maxdeg = 0;
    for (int64_t u = 0; u < n; ++u) {
        const int64_t d = offsets[u + 1] - offsets[u];
        if (d < 0) return fail(LB_ERR_ARG, "offsets decrease at %lld", (long long)u);
        if (d > maxdeg) maxdeg = d;
    }
    for (int64_t e = 0; e < m; ++e)
        if (cols[e] < 0 || (int64_t)cols[e] >= n) return fail(LB_ERR_ARG, "cols[%lld] = %d out of range", (long long)e, cols[e]);
    bool zero = false;
    if (weights)
        for (int64_t e = 0; e < m && !zero; ++e) zero = weights[e] == 0;
    lb_graph *g = new_graph(n, m, weights != nullptr);
    if (!g) return fail(LB_ERR_OOM, "host allocation failed");
    g->zero_weight = zero;
    g->max_degree = maxdeg;
    lb_status s = create_common(g);
    if (s == LB_OK) s = g->alloc(&g->off, n + 1);
    if (s == LB_OK) s = g->alloc(&g->col, m);
    if (s == LB_OK && weights) s = g->alloc(&g->w, m);
    if (s == LB_OK) {
        cudaError_t e = cudaMemcpy(g->off, offsets, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && m > 0) e = cudaMemcpy(g->col, cols, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice);
        if (e == cudaSuccess && weights && m > 0)
            e = cudaMemcpy(g->w, weights, sizeof(uint32_t) * (size_t)m, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) s = fail(LB_ERR_CUDA, "upload failed: %s", cudaGetErrorString(e));
    }
    if (s != LB_OK) {
        destroy_graph(g);
        return s;
    }
    *out = g;
    return LB_OK;
}

lb_status lb_graph_create_dev(const int64_t *offsets_dev, const int32_t *cols_dev, const uint32_t *weights_dev,
                              int64_t n, int64_t m, lb_graph **out) {
    if (!out) return fail(LB_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!offsets_dev || (m > 0 && !cols_dev)) return fail(LB_ERR_ARG, "offsets / cols is NULL");
    if (n < 1 || n >= ((int64_t)1 << 31)) return fail(LB_ERR_ARG, "n must be in [1, 2^31)");
    if (m < 0 || m >= ((int64_t)1 << 31)) return fail(LB_ERR_ARG, "m must be in [0, 2^31)");
    lb_graph *g = new_graph(n, m, weights_dev != nullptr);
    if (!g) return fail(LB_ERR_OOM, "host allocation failed");
    lb_status s = create_common(g);
    if (s == LB_OK) s = g->alloc(&g->off, n + 1);
    if (s == LB_OK) s = g->alloc(&g->col, m);
    if (s == LB_OK && weights_dev) s = g->alloc(&g->w, m);
    if (s == LB_OK) {
        cudaError_t e = cudaMemcpyAsync(g->off, offsets_dev, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyDeviceToDevice, g->stream);
        if (e == cudaSuccess && m > 0)
            e = cudaMemcpyAsync(g->col, cols_dev, sizeof(int32_t) * (size_t)m, cudaMemcpyDeviceToDevice, g->stream);
        if (e == cudaSuccess && weights_dev && m > 0)
            e = cudaMemcpyAsync(g->w, weights_dev, sizeof(uint32_t) * (size_t)m, cudaMemcpyDeviceToDevice, g->stream);
        uint32_t *derr = (uint32_t *)g->dres;
        if (e == cudaSuccess) e = cudaMemsetAsync(derr, 0, sizeof(uint32_t), g->stream);
        GraphDev gd{g->off, g->col, g->w, n, m};
        if (e == cudaSuccess) e = launch_validate(gd, derr, g->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(g->hres, derr, sizeof(uint32_t), cudaMemcpyDeviceToHost, g->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
        if (e != cudaSuccess) s = fail(LB_ERR_CUDA, "device graph set-up failed: %s", cudaGetErrorString(e));
        else if (*(uint32_t *)g->hres & kErrShape) s = fail(LB_ERR_ARG, "malformed CSR (offsets or cols)");
    }
    if (s == LB_OK && weights_dev) g->zero_weight = (*(uint32_t *)g->hres & kErrZeroWeight) != 0;
    if (s != LB_OK) {
        destroy_graph(g);
        return s;
    }
    *out = g;
    return LB_OK;
}

lb_status lb_graph_destroy(lb_graph *g) {
    destroy_graph(g);
    return LB_OK;
}

lb_status lb_graph_info(const lb_graph *g, int64_t *n, int64_t *m, int32_t *weighted, int32_t *device) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    if (n) *n = g->n;
    if (m) *m = g->m;
    if (weighted) *weighted = g->weighted ? 1 : 0;
    if (device) *device = g->device;
    return LB_OK;
}

lb_status lb_set_options(lb_graph *g, const lb_options *o) {
    if (!g || !o) return fail(LB_ERR_ARG, "NULL argument");
    lb_options n;
    LB_TRY(normalise_options(o, &n));
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    if (g->has_last) cudaEventSynchronize(g->ev_done);
    drop_execs(g);
    memset(g->grid, 0, sizeof(g->grid));
    memset(g->query_grid, 0, sizeof(g->query_grid));
    if (n.hist_bins != g->opt.hist_bins || n.mdt_override != g->opt.mdt_override) {
        g->mdt = -1;
        g->ns_children = -1;
    }
    g->opt = n;
    return LB_OK;
}

lb_status lb_get_options(const lb_graph *g, lb_options *o) {
    if (!g || !o) return fail(LB_ERR_ARG, "NULL argument");
    *o = g->opt;
    return LB_OK;
}

lb_status lb_bfs(lb_graph *g, int32_t src, lb_strategy s, int32_t *levels_out) {
    return host_query(g, LB_KIND_BFS, s, src, levels_out);
}

lb_status lb_sssp(lb_graph *g, int32_t src, lb_strategy s, uint32_t *dist_out) {
    return host_query(g, LB_KIND_SSSP, s, src, dist_out);
}

lb_status lb_bfs_batch(lb_graph *g, const int32_t *srcs, int64_t k, lb_strategy s, int32_t *levels_out) {
    return host_query_batch(g, LB_KIND_BFS, s, srcs, k, levels_out);
}

lb_status lb_sssp_batch(lb_graph *g, const int32_t *srcs, int64_t k, lb_strategy s, uint32_t *dist_out) {
    if (g && !g->weighted) return fail(LB_ERR_UNSUPPORTED, "SSSP needs a weighted graph");
    return host_query_batch(g, LB_KIND_SSSP, s, srcs, k, dist_out);
}

lb_status lb_bfs_dev(lb_graph *g, int32_t src, lb_strategy s, int32_t *out_dev, int32_t *parents_dev, void *stream) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    return run_query(g, LB_KIND_BFS, s, src, out_dev, parents_dev, (cudaStream_t)stream);
}

lb_status lb_sssp_dev(lb_graph *g, int32_t src, lb_strategy s, uint32_t *out_dev, int32_t *parents_dev,
                      void *stream) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    return run_query(g, LB_KIND_SSSP, s, src, out_dev, parents_dev, (cudaStream_t)stream);
}

lb_status lb_last_stats(lb_graph *g, lb_query_stats *out) {
    if (!g || !out) return fail(LB_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    memset(out, 0, sizeof(*out));
    if (!g->has_last) return fail(LB_ERR_ARG, "no query has run on this graph");
    Ctl h;
    LB_TRY(read_ctl(g, &h));
    float ms = 0.f;
    LB_CU(cudaEventElapsedTime(&ms, g->ev_start, g->ev_stop));
    out->iterations = h.level;
    out->steps = (int64_t)h.step;
    out->edges_relaxed = (int64_t)h.relaxed;
    out->pushes = (int64_t)h.pushes;
    out->mdt = (g->last_strategy == LB_NS || g->last_strategy == LB_NS_PHYS || g->last_strategy == LB_HP) ? g->mdt : 0;
    out->strategy = g->last_strategy;
    out->device_ms = ms;
    out->status = status_from_error(h.error);
    return LB_OK;
}

lb_status lb_last_trace(lb_graph *g, lb_step_record *out, int64_t cap, int64_t *len) {
    if (!g || !len || (cap > 0 && !out)) return fail(LB_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    if (!g->has_last) return fail(LB_ERR_ARG, "no query has run on this graph");
    Ctl h;
    LB_TRY(read_ctl(g, &h));
    const int64_t k = h.trace_len < (uint32_t)kTraceMax ? h.trace_len : kTraceMax;
    *len = k;
    const int64_t c = k < cap ? k : cap;
    if (c > 0) {
        static_assert(sizeof(TraceRec) == sizeof(lb_step_record), "trace record layout");
        LB_CU(cudaMemcpy(out, g->ctl->trace, sizeof(TraceRec) * (size_t)c, cudaMemcpyDeviceToHost));
    }
    return LB_OK;
}

lb_status lb_mem_report(lb_graph *g, lb_strategy s, lb_mem_stats *out) {
    if (!g || !out) return fail(LB_ERR_ARG, "NULL argument");
    if (s == LB_AUTO) s = LB_WD;
    if ((int)s < 0 || (int)s >= kStrategies) return fail(LB_ERR_ARG, "unknown strategy %d", (int)s);
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    memset(out, 0, sizeof(*out));
    const int64_t n = g->n, m = g->m;
    out->csr_offsets = 8 * (n + 1);
    out->csr_cols = 4 * (m > 0 ? m : 1);
    out->csr_weights = g->weighted ? 4 * (m > 0 ? m : 1) : 0;
    out->base_total = out->csr_offsets + out->csr_cols + out->csr_weights;
    out->status = 4 * n;
    out->visited = 4 * bitmap_alloc_words(n);
    const int64_t tcap = round_tiles(m);
    if (s == LB_NS || s == LB_NS_PHYS || s == LB_HP) {
        LB_TRY(ensure_mdt(g));
        out->mdt = g->mdt;
        out->ns_children = g->ns_children;
    }
    if (s == LB_NS_PHYS) out->ns_split = 4 * n + 8 * (out->ns_children > 0 ? out->ns_children : 1);
    if (is_ep(s)) {
        out->coo_src = 4 * (m > 0 ? m : 1);
        out->edge_lists = 2 * 4 * (m > 0 ? m : 1);
    } else {
        const int64_t cap = node_list_cap(g, s);
        out->node_lists = 2 * (4 * cap + 4 * cap + 4 * (cap + 1));
        if (s == LB_WD || s == LB_HP) out->tile_starts = 2 * 4 * tcap;
        if (s == LB_HP) out->sub_lists = 2 * (4 * n + 4 * n + 4 * (n + 1) + 4 * tcap);
    }
    out->control = (int64_t)sizeof(Ctl) + (s == LB_WD ? fast_entries(n) * (int64_t)sizeof(int4) : 0);
    out->extra_total = out->status + out->visited + out->node_lists + out->tile_starts + out->coo_src +
                       out->edge_lists + out->sub_lists + out->control + out->ns_split;
    out->resident = g->resident;
    return LB_OK;
}

lb_status lb_release_workspaces(lb_graph *g) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    if (g->has_last) cudaEventSynchronize(g->ev_done);
    cudaStreamSynchronize(g->stream);
    free_workspace(g);
    g->has_last = false;
    return LB_OK;
}

lb_status lb_autotune(lb_graph *g, int32_t kind, lb_strategy s, const int32_t *srcs, int32_t nsrc, lb_options *best,
                      double *best_ms) {
    if (!g || !srcs || nsrc < 1 || nsrc > 1024) return fail(LB_ERR_ARG, "need a graph and 1..1024 sources");
    if (kind != LB_KIND_BFS && kind != LB_KIND_SSSP && kind != LB_TUNE_BOTH) return fail(LB_ERR_ARG, "bad kind");
    if (s == LB_AUTO) s = LB_WD;
    if ((int)s < 0 || (int)s >= kStrategies) return fail(LB_ERR_ARG, "unknown strategy");
    for (int32_t i = 0; i < nsrc; ++i)
        if (srcs[i] < 0 || (int64_t)srcs[i] >= g->n) return fail(LB_ERR_ARG, "source out of range");
    if (kind != LB_KIND_BFS && !g->weighted) return fail(LB_ERR_UNSUPPORTED, "SSSP needs a weighted graph");
    const lb_options base = g->opt;
    // candidate grid per strategy: block shapes (CTAs per SM the relax grid
    // is sized for, the largest WD tile), the bin thresholds of the binned
    // forms (edges a thread / a warp serves), the granule size of node
    // splitting (MDT: the histogram's, or fixed), and HP's switch threshold
    // and hierarchy depth
    const int32_t ctas[] = {0, 2, 3, 4};
    std::vector<lb_options> cands;
    if (s == LB_WD) {
        for (int32_t t : {2048, 4096, 8192, 16384})
            for (int32_t c : ctas) {
                lb_options o = base;
                o.wd_tile = t;
                o.ctas_per_sm = c;
                cands.push_back(o);
            }
    } else if (s == LB_HP) {
        for (int32_t h : {256, 1024, 4096})
            for (int32_t d : {1, 2, 3}) {
                lb_options o = base;
                o.hp_mode = 0;
                o.hp_threshold = h;
                o.hp_depth = d;
                cands.push_back(o);
            }
        for (int32_t h : {256, 1024})
            for (int32_t tm : {8, 32, 128})
                for (int32_t wm : {512, 4096}) {
                    lb_options o = base;
                    o.hp_mode = 1;
                    o.hp_threshold = h;
                    o.thread_max = tm;
                    o.hp_warp_max = wm;
                    cands.push_back(o);
                }
    } else if (s == LB_NS || s == LB_NS_PHYS) {
        for (int32_t md : {0, 32, 256, 2048}) {
            lb_options o = base;
            o.ns_mode = 0;
            o.mdt_override = md;
            cands.push_back(o);
        }
        if (s == LB_NS)
            for (int32_t md : {0, 256, 2048})
                for (int32_t tm : {8, 32, 128}) {
                    lb_options o = base;
                    o.ns_mode = 1;
                    o.mdt_override = md;
                    o.thread_max = tm;
                    cands.push_back(o);
                }
    } else {
        for (int32_t c : ctas) {
            lb_options o = base;
            o.ctas_per_sm = c;
            cands.push_back(o);
        }
    }
    double best_t = 1e300;
    lb_options best_o = base;
    uint32_t *out = nullptr;
    {
        std::lock_guard<std::mutex> lk(g->mu);
        DeviceGuard dg(g->device);
        if (!g->out_internal) LB_TRY(g->alloc(&g->out_internal, g->n));
        out = g->out_internal;
    }
    // any failure part way through puts the caller's options back
    auto restore = [&](lb_status st) {
        const std::string msg = t_err;
        lb_set_options(g, &base);
        t_err = msg;
        return st;
    };
    // times o on every source: LB_OK with *usable false when a query of o
    // ended with an error status (o is then not a candidate)
    auto time_opts = [&](const lb_options &o, bool *usable, double *t) -> lb_status {
        lb_status so = lb_set_options(g, &o);
        if (so != LB_OK) return so;
        double tot = 0.0;
        bool ok = true;
        for (int32_t i = 0; i < nsrc * (kind == LB_TUNE_BOTH ? 2 : 1) && ok; ++i) {
            const int32_t k = kind == LB_TUNE_BOTH ? (i & 1) : kind;
            const int32_t src = srcs[kind == LB_TUNE_BOTH ? i / 2 : i];
            for (int rep = 0; rep < 2 && ok; ++rep) {  // first run builds the loop; the second is timed
                lb_status st;
                {
                    std::lock_guard<std::mutex> lk(g->mu);
                    DeviceGuard dg(g->device);
                    st = run_query(g, k, s, src, out, nullptr, g->stream);
                }
                if (st != LB_OK) return st;
                lb_query_stats qs;
                st = lb_last_stats(g, &qs);
                if (st != LB_OK) return st;
                if (qs.status != LB_OK && qs.status != LB_ERR_OVERFLOW) ok = false;
                if (rep == 1) tot += qs.device_ms;
            }
        }
        *usable = ok;
        *t = tot;
        return LB_OK;
    };
    // Every candidate timed once, fastest first (usable ones only).
    auto time_all = [&](const std::vector<lb_options> &cs, lb_status *err) {
        std::vector<std::pair<double, int>> t;
        for (size_t i = 0; i < cs.size() && *err == LB_OK; ++i) {
            bool ok = false;
            double tot = 0.0;
            *err = time_opts(cs[i], &ok, &tot);
            if (*err == LB_OK && ok) t.push_back({tot, (int)i});
        }
        std::sort(t.begin(), t.end());
        return t;
    };
    // One timing per candidate, then the three fastest are timed twice more
    // (interleaved) and ranked by the sum of their three timings, so one
    // noisy timing does not pick the options.  Returns the index in cs.
    auto pick = [&](const std::vector<lb_options> &cs, lb_status *err) -> int {
        std::vector<std::pair<double, int>> t = time_all(cs, err);
        if (*err != LB_OK || t.empty()) return -1;
        if (t.size() > 3) t.resize(3);
        for (int rep = 0; rep < 2 && t.size() > 1; ++rep)
            for (auto &c : t) {
                bool ok = false;
                double tot = 0.0;
                *err = time_opts(cs[(size_t)c.second], &ok, &tot);
                if (*err != LB_OK) return -1;
                c.first += ok ? tot : 1e300;
            }
        std::sort(t.begin(), t.end());
        best_t = t[0].first / (t.size() > 1 ? 3.0 : 1.0);
        return t[0].second;
    };
    // The grid at the caller's bitmap placement; the three fastest options
    // go on to the placement pass.
    std::vector<lb_options> top;
    {
        lb_status err = LB_OK;
        const std::vector<std::pair<double, int>> t = time_all(cands, &err);
        if (err != LB_OK) return restore(err);
        for (size_t k = 0; k < t.size() && k < 3; ++k) top.push_back(cands[(size_t)t[k].second]);
        if (!t.empty()) {
            best_t = t[0].first;
            best_o = top[0];
        }
    }
    // For WD, whether levels with small lists are better left to the whole
    // grid than to the small-list team, decided on the fastest grid option and applied to all three.
    if (!top.empty() && s == LB_WD && top[0].small_edges != 0) {
        std::vector<lb_options> two{top[0], top[0]};
        two[1].small_edges = 0;
        lb_status err = LB_OK;
        const int i = pick(two, &err);
        if (err != LB_OK) return restore(err);
        if (i == 1)
            for (lb_options &o : top) o.small_edges = 0;
        if (i >= 0) best_o = top[0];
    }
    // Then every bitmap placement of each of the three (the placement and
    // the grid shape interact: a placement that is slow for one CTA count
    // can make another win the grid pass).
    if (!top.empty()) {
        std::vector<lb_options> places;
        for (const lb_options &t : top)
            for (int32_t pl = 0; pl < kBitmapPlaces; ++pl) {
                lb_options o = t;
                o.bitmap_place = pl;
                places.push_back(o);
            }
        lb_status err = LB_OK;
        const int i = pick(places, &err);
        if (err != LB_OK) return restore(err);
        if (i >= 0) best_o = places[(size_t)i];
    }
    LB_TRY(lb_set_options(g, &best_o));
    if (best) *best = best_o;
    if (best_ms) *best_ms = best_t / nsrc;
    return LB_OK;
}

lb_status lb_mdt(lb_graph *g, int32_t bins, int64_t *mdt, int64_t *max_degree, int32_t *bin_index) {
    if (!g) return fail(LB_ERR_ARG, "graph is NULL");
    if (bins < 1 || bins > 4096) return fail(LB_ERR_ARG, "bins must be in [1, 4096]");
    std::lock_guard<std::mutex> lk(g->mu);
    DeviceGuard dg(g->device);
    if (g->has_last) LB_CU(cudaStreamWaitEvent(g->stream, g->ev_done, 0));
    GraphDev gd{g->off, g->col, g->w, g->n, g->m};
    LB_CU(launch_mdt(gd, bins, g->scratch, g->dres, g->stream));
    LB_CU(cudaMemcpyAsync(g->hres, g->dres, 3 * sizeof(int64_t), cudaMemcpyDeviceToHost, g->stream));
    LB_CU(cudaStreamSynchronize(g->stream));
    if (mdt) *mdt = g->hres[0];
    if (max_degree) *max_degree = g->hres[1];
    if (bin_index) *bin_index = (int32_t)g->hres[2];
    return LB_OK;
}

lb_status lb_wd_offsets(const int64_t *deg, int64_t F, int64_t T, int64_t *node_off, int64_t *edge_off,
                        int64_t *ept) {
    if (F < 0 || F > ((int64_t)1 << 24) || T < 1 || T > ((int64_t)1 << 24)) return fail(LB_ERR_ARG, "F or T out of range");
    if ((F > 0 && !deg) || !node_off || !edge_off || !ept) return fail(LB_ERR_ARG, "NULL argument");
    int64_t E = 0;
    for (int64_t i = 0; i < F; ++i) {
        if (deg[i] < 0 || deg[i] >= ((int64_t)1 << 31)) return fail(LB_ERR_ARG, "deg[%lld] out of range", (long long)i);
        E += deg[i];
    }
    if (E >= ((int64_t)1 << 31)) return fail(LB_ERR_ARG, "sum of degrees must be < 2^31");
    Allocator al;
    {
        std::lock_guard<std::mutex> lk(g_alloc_mu);
        al.alloc_fn = g_alloc_fn;
        al.free_fn = g_free_fn;
        al.ctx = g_alloc_ctx;
    }
    cudaStream_t st = nullptr;
    LB_CU(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    void *bufs[7] = {nullptr};
    const size_t sizes[7] = {sizeof(int64_t) * (size_t)(F > 0 ? F : 1), sizeof(int32_t) * (size_t)(F > 0 ? F : 1),
                             sizeof(int32_t) * (size_t)(F > 0 ? F : 1), sizeof(int32_t) * (size_t)(F + 1),
                             sizeof(int32_t) * (size_t)(T + 1), sizeof(Ctl), sizeof(int64_t)};
    lb_status status = LB_OK;
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 7 && e == cudaSuccess; ++i) e = al.alloc(&bufs[i], sizes[i]);
    std::string msg;
    if (e == cudaSuccess && F > 0) e = cudaMemcpyAsync(bufs[0], deg, sizes[0], cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(bufs[5], 0, sizeof(Ctl), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(bufs[4], 0, sizes[4], st);
    NodeList L{(int32_t *)bufs[1], (int32_t *)bufs[2], (int32_t *)bufs[3], (int32_t *)bufs[4]};
    if (e == cudaSuccess) e = launch_wd_offsets((const int64_t *)bufs[0], F, T, L, (Ctl *)bufs[5], (int64_t *)bufs[6], st);
    int64_t h_ept = 0;
    int32_t *h_ts = new (std::nothrow) int32_t[(size_t)T + 1];
    int32_t *h_scan = new (std::nothrow) int32_t[(size_t)F + 1];
    if (!h_ts || !h_scan) e = cudaErrorMemoryAllocation;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h_ept, bufs[6], sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_ts, bufs[4], sizes[4], cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_scan, bufs[3], sizes[3], cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        status = fail(e == cudaErrorMemoryAllocation ? LB_ERR_OOM : LB_ERR_CUDA, "lb_wd_offsets: %s", cudaGetErrorString(e));
    } else {
        *ept = h_ept;
        for (int64_t t = 0; t < T; ++t) {
            const int64_t s0 = t * h_ept;
            if (h_ept == 0 || s0 >= E) {
                node_off[t] = F;
                edge_off[t] = 0;
            } else {
                node_off[t] = h_ts[t];
                edge_off[t] = s0 - h_scan[h_ts[t]];
            }
        }
    }
    delete[] h_ts;
    delete[] h_scan;
    for (int i = 0; i < 7; ++i)
        if (bufs[i]) al.release(bufs[i]);
    cudaStreamDestroy(st);
    return status;
}

}  // extern "C"
