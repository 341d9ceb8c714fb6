// Host side of the C ABI declared in include/kbisim.h: contexts, workspace
// planning, the per-round driver loop (paper Alg. 1: rounds 1..k with the
// block-count stop test), host-buffer refinement and timing.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "kb_internal.cuh"

struct kb_context {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::string last_error;
    // scratch: caller-provided or library-owned (grow-only)
    void* user_ws = nullptr;
    size_t user_ws_bytes = 0;
    void* own_ws = nullptr;
    size_t own_ws_bytes = 0;
    // small persistent device state
    kb::Counters* d_ctr = nullptr;
    kb::Counters* h_ctr = nullptr;  // pinned: the last counters read, and a slot per round in flight (queue_counters)
    cudaEvent_t slot_ev[4] = {};
    int fused_ctas = 0;  // largest grid of the fused kernel (launch_fused_rounds),
    int fused_most = 0;  //   as the device has it,
    uint32_t fused_polls = kb::kFusedPolls;  // and its limit of waiting (kb_set_round_kernel)
    int64_t fused_launches = 0, fused_refused = 0, fused_gave_up = 0;  // kb_get_round_kernel
    uint32_t* d_dense = nullptr;  // label minima and (minimum, id) pairs of a small-label level 0
    bool dense_empty = false;     // the minima are all ones (launch_dense_level0 leaves them so)
    char* h_hubs = nullptr;       // pinned: the first kEagerHubs hubs of a plan and their degrees
    void* class_tmp = nullptr;    // degree-class bitmaps of the last plan; its tile counts and hub list
    size_t class_tmp_bytes = 0;
    void* plan_tmp = nullptr;    // in-degree scratch used by kb_workspace_size
    size_t plan_tmp_bytes = 0;
    // host-buffer refinement staging (library-owned)
    void* stage = nullptr;
    size_t stage_bytes = 0;
    // autotuned values per size class (kb_autotune); plan_graphs is the graph
    // count of the batched call being planned
    std::map<int32_t, kb_tuning> tuned;
    int64_t plan_graphs = 1;
    // block table and empty-signature minima, kept between calls (grow-only)
    // unless the caller gives the workspace: entries of earlier rounds lose by
    // their epoch or round word, so a call clears neither
    void* tab = nullptr;
    size_t tab_bytes = 0;
    uint32_t tab_epoch = 0;
    void* emin = nullptr;
    size_t emin_bytes = 0;
    uint32_t emin_round = 0;
    // batched refinement
    void* batch_ws = nullptr;
    size_t batch_ws_bytes = 0;
    void* tune_buf = nullptr;
    size_t tune_buf_bytes = 0;
    // fixpoint refinement: the last two levels
    void* fix_buf = nullptr;
    size_t fix_buf_bytes = 0;
    // summary graph: triple table, first edges, edge bitmap and its ranks
    void* sum_buf = nullptr;
    size_t sum_buf_bytes = 0;
    // incremental refinement: bitmaps, old blocks' smallest members
    void* upd_buf = nullptr;
    size_t upd_buf_bytes = 0;
    cudaStream_t copy_stream = nullptr;  // level rows back to the host (kb_refine_host)
    cudaEvent_t row_ev = nullptr;
    // timing: CUDA events per kernel family; with work, also the vertices and
    // edges every round re-keys (one extra pass over the row offsets a round)
    bool timing = false;
    bool work = false;
    std::vector<float> round_ms;
    // per round of the last kb_refine / kb_refine_from / kb_refine_fixpoint
    // call: vertices and processed edges re-keyed by the small, medium and hub
    // kernels
    std::vector<std::array<int64_t, 6>> round_keyed;
    float kernel_ms[KB_KERNEL_COUNT] = {};
    int64_t kernel_launches[KB_KERNEL_COUNT] = {};
    cudaEvent_t ev[2 * 10 + 2] = {};  // pairs for the round timer; the last two time whole calls
};

namespace {

using kb::Counters;

kb_status fail(kb_context* ctx, kb_status st, const char* fmt, ...) {
    if (ctx) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        ctx->last_error = buf;
    }
    return st;
}

#define KB_CUDA(ctx, call)                                                                        \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess)                                                                    \
            return fail((ctx), KB_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_));     \
    } while (0)

#define KB_TRY(expr)                       \
    do {                                   \
        kb_status s_ = (expr);             \
        if (s_ != KB_OK) return s_;        \
    } while (0)

// Hubs whose list comes back in the same copy as the counts of the plan.
constexpr int64_t kEagerHubs = 4096;

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

uint64_t next_pow2(uint64_t x) {
    uint64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Block-table slots for n vertices at load factor lf: a power of two of at
// least 1024 and at most 2^31, since a vertex's slot index is kept in the 31
// low bits of its slot_of entry (bit 31 marks an empty signature).  Above
// 2^30 vertices the table can thus be fuller than lf asks (it still holds
// every block: n <= 2^31 - 2).
uint64_t table_capacity(int64_t n, float lf) {
    uint64_t cap = next_pow2((uint64_t)((double)std::max<int64_t>(n, 1) / (double)lf) + 1);
    if (cap < 1024) cap = 1024;
    if (cap > ((uint64_t)1 << 31)) cap = (uint64_t)1 << 31;
    return cap;
}

// Device buffers of one refine call, carved from one workspace allocation.
struct Plan {
    int64_t n = 0, m = 0, m_proc = 0;
    int dir = 0;
    bool labels = false;
    int thr = kb::kDefaultHubThreshold;
    int hub_chunk = kb::kDefaultHubChunk;
    int med_split = kb::kDefaultMedSplit;
    int small_max = kb::kMidDegree;  // small_max_degree: small and mid vertices
    int warp_verts = 0;  // 0: by the graph's size (launch_small_round)
    int32_t size_class = 0;  // key of the tuning cache
    uint64_t cap = 0;
    bool reorder = false;  // locality order of the gather (RoundParams::perm)
    int subject = 0;       // kb_options::subject (generic CSE rounds when > 0)
    bool freeze = false;   // frozen blocks skip the rounds (RoundParams::frozen)
    bool dense0 = false;   // one graph: level 0 may take the small-label path (launch_dense_level0)
    bool sketch = false;     // hub sketches ahead of the exact sets (launch_hub_sketch)
    bool ext_table = false;  // block table and empty-signature minima live outside the workspace
    bool ext_freeze = false;  // frozen-block state lives outside the workspace
    // the per-graph part (processed CSR, degree classes, hub plan, locality
    // order, edgeless bits) lives in a prepared graph's own buffers: layout
    // offsets of that part are relative to them (kb_graph_prepare)
    bool graph_ext = false;
    size_t graph_bytes = 0;
    // hubs (host copies, ascending vertex id)
    std::vector<int32_t> hub_v;
    std::vector<int64_t> chunk_off, set_off;
    // their sizes (the lists themselves are dropped once on the device)
    size_t n_hubs = 0;
    int64_t n_chunks = 0, set_slots = 0;
    int64_t n_mid = 0, n_med = 0;  // mid and medium vertices
    // layout
    size_t o_rowp = 0, o_colp = 0, o_labp = 0, o_cursor = 0, o_inpref = 0, o_i64tmp = 0;
    size_t csr_bytes = 0;
    size_t o_emin = 0, o_mid = 0, o_med = 0, o_slot = 0, o_table = 0, o_bitmap = 0, o_prefix = 0, o_scan = 0, o_hubv = 0, o_chunk = 0, o_setoff = 0,
           o_chunkhub = 0, o_chunkext = 0, o_perm = 0, o_gat = 0, o_colr = 0, o_hist = 0, o_ownkey = 0, o_acc = 0, o_cnt = 0, o_sets = 0, o_exact = 0, o_exactlist = 0, o_twin = 0,
           o_frozen = 0, o_classes = 0, o_shared = 0, o_minof = 0, o_joined = 0, o_moved = 0, o_mark = 0;
    size_t clear_bytes = 0;  // from o_bitmap on
    size_t total = 0;
    // bytes of one degree-class bitmap; four follow one another (kb::DegreeClass)
    size_t class_bytes() const { return align_up(sizeof(uint32_t) * (size_t)((n >> 5) + 1)); }
    static constexpr int kClassBitmaps = 1 + kb::kClassLists;
};

bool needs_in_csr(int dir) { return dir == KB_DIR_IN || dir == KB_DIR_BOTH; }

}  // namespace

// A prepared graph (kb_graph_prepare): the per-graph part of a plan built
// once, in device buffers of its own.
struct kb_prepared {
    int device = 0;
    kb_graph g{};       // the caller's arrays
    int32_t dir = 0;
    int32_t edge_labels = 0;
    Plan P;             // graph_ext layout; host hub lists dropped after upload
    char* csr = nullptr;   // processed CSR (IN / BOTH)
    char* gbuf = nullptr;  // per-graph part
    float build_ms = 0.f;
    ~kb_prepared() {
        if (!csr && !gbuf) return;
        int cur = 0;
        cudaGetDevice(&cur);
        cudaSetDevice(device);
        cudaFree(csr);
        cudaFree(gbuf);
        cudaSetDevice(cur);
    }
};

namespace {

void layout_csr(Plan& P) {
    size_t off = 0;
    P.csr_bytes = 0;
    if (!needs_in_csr(P.dir)) return;
    auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
    P.o_rowp = take(sizeof(int64_t) * (size_t)(P.n + 1));
    P.o_colp = take(sizeof(int32_t) * (size_t)P.m_proc);
    P.o_labp = take(P.labels ? sizeof(int32_t) * (size_t)P.m_proc : 0);
    P.o_cursor = take(sizeof(int64_t) * (size_t)(P.n + 1));
    P.o_inpref = take(sizeof(int64_t) * (size_t)(P.n + 1));
    P.o_i64tmp = take(sizeof(int64_t) * kb::scan_i64_tmp(P.n + 1));
    P.csr_bytes = off;
}

// Round buffers.  The per-graph part comes first, at offsets after the CSR
// (or, with graph_ext, from 0 in a buffer of its own: graph_bytes); the
// per-call part follows in the workspace (total).
void layout_round(Plan& P) {
    size_t goff = P.graph_ext ? 0 : P.csr_bytes;
    auto takeg = [&](size_t bytes) { size_t o = goff; goff += align_up(bytes); return o; };
    const int64_t nw = (P.n >> 5) + 1;
    const size_t H = P.n_hubs;
    // The mid and medium vertices, one list behind the other.  A prepared graph's are
    // as long as they are; a call's have room for as many as n and the edges allow, so
    // that a workspace of the queried size serves every graph of that size without
    // hubs, also one that was changed in place since the query.
    const int64_t most = P.m_proc / (std::min(P.small_max, kb::kSmallDegree) + 1);
    P.o_mid = takeg(sizeof(int32_t) * (size_t)(P.graph_ext ? P.n_mid + P.n_med : std::min(P.n, most)));
    P.o_med = P.o_mid + sizeof(int32_t) * (size_t)P.n_mid;
    P.o_hubv = takeg(sizeof(int32_t) * H);
    P.o_chunk = takeg(sizeof(int64_t) * (H + 1));
    P.o_setoff = takeg(sizeof(int64_t) * (H + 1));
    P.o_chunkhub = takeg(sizeof(int32_t) * (size_t)P.n_chunks);
    P.o_chunkext = takeg(sizeof(uint64_t) * (size_t)P.n_chunks);
    P.o_perm = takeg(P.reorder ? sizeof(int32_t) * (size_t)P.n : 0);
    // a reordered copy of the caller's neighbour ids; the library's own in-edge
    // CSR is reordered in place
    P.o_colr = takeg(P.reorder && !needs_in_csr(P.dir) ? sizeof(int32_t) * (size_t)P.m_proc : 0);
    P.o_hist = takeg(P.reorder ? sizeof(unsigned long long) * 512 : 0);
    P.o_classes = takeg(P.graph_ext ? Plan::kClassBitmaps * P.class_bytes() : 0);  // (else ctx->class_tmp serves)
    P.graph_bytes = P.graph_ext ? goff : 0;
    size_t off = P.graph_ext ? 0 : goff;
    auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
    P.o_emin = take(P.ext_table ? 0 : sizeof(uint64_t) * (size_t)std::max<int64_t>(P.n, 1));
    P.o_slot = take(sizeof(int32_t) * (size_t)std::max<int64_t>(P.n, 1));
    P.o_table = take(P.ext_table ? 0 : sizeof(uint64_t) * (size_t)P.cap);
    // what starts a call clear, together
    const bool own_freeze = P.freeze && !P.ext_freeze;
    P.o_bitmap = take(sizeof(uint32_t) * (size_t)nw);
    P.o_frozen = take(own_freeze ? sizeof(uint32_t) * (size_t)nw : 0);
    P.o_shared = take(own_freeze ? sizeof(uint32_t) * (size_t)nw : 0);
    P.o_moved = take(own_freeze ? sizeof(uint32_t) * (size_t)nw : 0);
    P.o_joined = take(P.freeze ? sizeof(uint32_t) * (size_t)nw : 0);
    P.clear_bytes = off - P.o_bitmap;
    P.o_prefix = take(sizeof(uint2) * (size_t)(nw + 1));
    P.o_scan = take(sizeof(uint32_t) * kb::scan_tmp_words(nw));
    P.o_acc = take(sizeof(uint64_t) * H);
    P.o_cnt = take(sizeof(uint32_t) * H);
    P.o_sets = take(sizeof(uint64_t) * (size_t)P.set_slots);
    P.sketch = P.n_chunks >= kb::kSketchMinChunks && P.thr >= kb::kSketchMinThreshold;
    P.o_exact = take(P.sketch ? sizeof(uint32_t) * H : 0);
    P.o_exactlist = take(P.sketch ? sizeof(int32_t) * (size_t)P.n_chunks : 0);
    P.o_twin = take(P.sketch ? sizeof(uint32_t) * (size_t)next_pow2(2 * H) : 0);
    P.o_gat = take(P.reorder ? sizeof(int32_t) * (size_t)P.n : 0);
    P.o_ownkey = take(P.subject ? sizeof(int32_t) * (size_t)P.n : 0);
    P.o_minof = take(own_freeze ? sizeof(uint32_t) * (size_t)P.n : 0);
    P.o_mark = take(own_freeze ? sizeof(uint32_t) * (size_t)nw : 0);
    P.total = off;
}

kb_status check_graph(kb_context* ctx, const kb_graph* g, const kb_options* opt, int k) {
    if (!g || !opt) return fail(ctx, KB_ERR_INVALID_ARG, "graph and options must not be NULL");
    if (g->n < 0 || g->m < 0) return fail(ctx, KB_ERR_INVALID_ARG, "negative n or m");
    if (g->n > 2147483646LL) return fail(ctx, KB_ERR_INVALID_ARG, "n exceeds 2^31-2");
    if (g->m > (1LL << 45)) return fail(ctx, KB_ERR_INVALID_ARG, "m exceeds 2^45");
    if (k < 0) return fail(ctx, KB_ERR_INVALID_ARG, "k must be >= 0");
    if (opt->direction < 0 || opt->direction > 2) return fail(ctx, KB_ERR_INVALID_ARG, "bad direction");
    if (g->n > 0 && !g->row_offsets) return fail(ctx, KB_ERR_INVALID_ARG, "row_offsets is NULL");
    if (g->m > 0 && !g->col_indices) return fail(ctx, KB_ERR_INVALID_ARG, "col_indices is NULL");
    if (g->n == 0 && g->m != 0) return fail(ctx, KB_ERR_INVALID_ARG, "edges without vertices");
    if (opt->load_factor < 0.f || opt->load_factor > 0.9f)
        return fail(ctx, KB_ERR_INVALID_ARG, "load_factor must be in (0, 0.9]");
    if (opt->hub_threshold < 0 || opt->hub_threshold > kb::kMaxHubThreshold)
        return fail(ctx, KB_ERR_INVALID_ARG, "hub_threshold must be in [0, %d]", kb::kMaxHubThreshold);
    if (opt->hash_mode < 0 || opt->hash_mode > 1) return fail(ctx, KB_ERR_INVALID_ARG, "bad hash_mode");
    if (opt->reorder < 0 || opt->reorder > 2) return fail(ctx, KB_ERR_INVALID_ARG, "reorder must be 0, 1 or 2");
    if (opt->subject < 0 || opt->subject > 3) return fail(ctx, KB_ERR_INVALID_ARG, "subject must be 0..3");
    if (opt->small_task_vertices != 0 && (opt->small_task_vertices < 32 || opt->small_task_vertices > 65536))
        return fail(ctx, KB_ERR_INVALID_ARG, "small_task_vertices must be 0 or in [32, 65536]");
    if (opt->hub_chunk_edges != 0 && opt->hub_chunk_edges != 256 && opt->hub_chunk_edges != 512 &&
        opt->hub_chunk_edges != 1024)
        return fail(ctx, KB_ERR_INVALID_ARG, "hub_chunk_edges must be 0, 256, 512 or 1024");
    if (opt->medium_split < 0 || opt->medium_split > kb::kMaxMedSplit)
        return fail(ctx, KB_ERR_INVALID_ARG, "medium_split must be in [0, %d]", kb::kMaxMedSplit);
    if (opt->small_max_degree < 0 || opt->small_max_degree > kb::kMidDegree)
        return fail(ctx, KB_ERR_INVALID_ARG, "small_max_degree must be in [0, %d]", kb::kMidDegree);
    if (opt->direction == KB_DIR_BOTH && g->m > (int64_t)1 << 62)
        return fail(ctx, KB_ERR_INVALID_ARG, "too many edges");
    return KB_OK;
}

kb_status ensure_buffer(kb_context* ctx, void** buf, size_t* have, size_t need) {
    if (need <= *have) return KB_OK;
    if (*buf) cudaFree(*buf);
    *buf = nullptr;
    *have = 0;
    if (cudaMalloc(buf, need) != cudaSuccess) {
        cudaGetLastError();
        *buf = nullptr;
        return fail(ctx, KB_ERR_OOM, "cannot allocate %zu bytes of device memory", need);
    }
    *have = need;
    return KB_OK;
}

kb_status read_counters(kb_context* ctx) {
    KB_CUDA(ctx, cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(Counters), cudaMemcpyDeviceToHost, ctx->stream));
    KB_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return KB_OK;
}

// The counters as they are after what is queued now (`round`), and waiting for
// them (into ctx->h_ctr) while later rounds are queued already.
constexpr int kCounterSlots = 4;

kb_status queue_counters(kb_context* ctx, int round) {
    const int slot = round % kCounterSlots;
    KB_CUDA(ctx, cudaMemcpyAsync(ctx->h_ctr + 1 + slot, ctx->d_ctr, sizeof(Counters), cudaMemcpyDeviceToHost, ctx->stream));
    KB_CUDA(ctx, cudaEventRecord(ctx->slot_ev[slot], ctx->stream));
    return KB_OK;
}

kb_status wait_counters(kb_context* ctx, int round) {
    const int slot = round % kCounterSlots;
    KB_CUDA(ctx, cudaEventSynchronize(ctx->slot_ev[slot]));
    *ctx->h_ctr = ctx->h_ctr[1 + slot];
    return KB_OK;
}

kb_status device_error(kb_context* ctx) {
    const int32_t e = ctx->h_ctr->err;
    if (e & kb::kErrInvalid)
        return fail(ctx, KB_ERR_INVALID_ARG, "row_offsets not monotone from 0 to m, or a neighbour id out of [0, n)");
    if (e & kb::kErrTableFull) return fail(ctx, KB_ERR_TABLE_FULL, "block table probe limit reached");
    if (e & kb::kErrWait) return fail(ctx, KB_ERR_TIMEOUT, "a wait for the whole grid gave up");
    if (e & (kb::kErrStage | kb::kErrHubSet)) return fail(ctx, KB_ERR_DEVICE_CHECK, "device consistency check failed (%d)", e);
    return KB_OK;
}

// Build the processed CSR (IN / BOTH) into `base` (layout_csr offsets).
kb_status build_processed_csr(kb_context* ctx, const kb_graph* g, Plan& P, char* base) {
    if (!needs_in_csr(P.dir)) return KB_OK;
    int64_t* inpref = reinterpret_cast<int64_t*>(base + P.o_inpref);
    KB_CUDA(ctx, cudaMemsetAsync(inpref, 0, sizeof(int64_t) * (size_t)(P.n + 1), ctx->stream));
    kb::launch_in_degree(P.m, g->col_indices, inpref, ctx->stream);
    kb::launch_scan_i64(inpref, P.n, inpref, reinterpret_cast<int64_t*>(base + P.o_i64tmp), ctx->stream);
    kb::launch_build_csr(P.n, P.m, g->row_offsets, g->col_indices, P.labels ? g->edge_labels : nullptr, inpref,
                         P.dir == KB_DIR_BOTH ? 1 : 0, reinterpret_cast<int64_t*>(base + P.o_rowp),
                         reinterpret_cast<int32_t*>(base + P.o_colp),
                         P.labels ? reinterpret_cast<int32_t*>(base + P.o_labp) : nullptr,
                         reinterpret_cast<int64_t*>(base + P.o_cursor), ctx->stream);
    KB_CUDA(ctx, cudaGetLastError());
    return KB_OK;
}

// Where launch_classes put its results (ctx->class_tmp), for a plan's n.
struct ClassScratch {
    size_t bits = 0, counts = 0, hub_v = 0, hub_deg = 0, total = 0;
    int64_t hub_cap = 0;
    explicit ClassScratch(const Plan& P) {
        counts = Plan::kClassBitmaps * P.class_bytes();
        hub_v = counts + align_up(kb::kClassLists * sizeof(uint32_t) * kb::class_tiles(P.n));
        hub_cap = std::min<int64_t>(P.n, P.m_proc / (P.thr + 1) + 1);
        hub_deg = hub_v + align_up(sizeof(int32_t) * (size_t)hub_cap);
        total = hub_deg + align_up(sizeof(int64_t) * (size_t)hub_cap);
    }
};

// The tile counts lie in the counters, which are cleared in any case, or in the
// scratch.
uint32_t* tile_counts(kb_context* ctx, const Plan& P, const ClassScratch& C) {
    if (kb::kClassLists * kb::class_tiles(P.n) <= sizeof(Counters::tiles) / sizeof(uint32_t)) return ctx->d_ctr->tiles;
    return reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(ctx->class_tmp) + C.counts);
}

// Degree classes of the processed CSR and the host side of the plan: hubs,
// their chunks and sets, the number of medium vertices.  One round trip, which
// also brings back ctx->h_ctr (errors of the validation, the level-0 key
// check).
kb_status plan_classes(kb_context* ctx, Plan& P, const int64_t* row_p, kb::CheckRows check, const kb::CheckIds& ids) {
    cudaStream_t s = ctx->stream;
    P.hub_v.clear();
    P.chunk_off.assign(1, 0);
    P.set_off.assign(1, 0);
    P.n_hubs = 0;
    P.n_chunks = P.set_slots = P.n_mid = P.n_med = 0;
    if (P.n == 0) return read_counters(ctx);
    const ClassScratch C(P);
    KB_TRY(ensure_buffer(ctx, &ctx->class_tmp, &ctx->class_tmp_bytes, C.total));
    char* b = reinterpret_cast<char*>(ctx->class_tmp);
    uint32_t* counts = tile_counts(ctx, P, C);
    if (counts != ctx->d_ctr->tiles)
        KB_CUDA(ctx, cudaMemsetAsync(counts, 0, kb::kClassLists * sizeof(uint32_t) * kb::class_tiles(P.n), s));
    uint32_t* bits = reinterpret_cast<uint32_t*>(b);
    const int64_t pitch = (int64_t)(P.class_bytes() / sizeof(uint32_t));
    const kb::ClassBounds bounds{std::min(P.small_max, kb::kSmallDegree), P.small_max, P.thr};
    // A graph with few possible hubs has them written to pinned memory as they are
    // found; otherwise they are listed, and the first ones copied.
    const int64_t eager = std::min(C.hub_cap, kEagerHubs);
    int32_t* h_v = reinterpret_cast<int32_t*>(ctx->h_hubs);
    int64_t* h_deg = reinterpret_cast<int64_t*>(ctx->h_hubs + sizeof(int32_t) * kEagerHubs);
    kb::HubSink sink;
    if (C.hub_cap <= kEagerHubs) sink = {h_v, h_deg, (uint32_t)C.hub_cap};
    kb::launch_classes(P.n, P.m_proc, row_p, bounds, bits, pitch, counts, check, ids, sink, ctx->d_ctr, s);
    if (!sink.cap) {
        kb::launch_class_lists(P.n, row_p, bits, pitch, counts,
                               {kb::kHub, C.hub_cap, reinterpret_cast<int32_t*>(b + C.hub_v),
                                reinterpret_cast<int64_t*>(b + C.hub_deg)},
                               kb::ClassList{}, s);
        KB_CUDA(ctx, cudaMemcpyAsync(h_v, b + C.hub_v, sizeof(int32_t) * (size_t)eager, cudaMemcpyDeviceToHost, s));
        KB_CUDA(ctx, cudaMemcpyAsync(h_deg, b + C.hub_deg, sizeof(int64_t) * (size_t)eager, cudaMemcpyDeviceToHost, s));
    }
    KB_CUDA(ctx, cudaGetLastError());
    KB_TRY(read_counters(ctx));
    KB_TRY(device_error(ctx));
    P.n_mid = ctx->h_ctr->n_class[0];
    P.n_med = ctx->h_ctr->n_class[1];
    const int64_t H = ctx->h_ctr->n_class[2];
    if (H > C.hub_cap || P.n_mid + P.n_med > std::min(P.n, P.m_proc / (bounds.small + 1))) return fail(ctx, KB_ERR_DEVICE_CHECK, "degree class larger than the graph allows");
    if (H <= 0) return KB_OK;
    P.hub_v.resize((size_t)H);
    std::vector<int64_t> deg((size_t)H);
    if (sink.cap) {
        std::vector<std::pair<int32_t, int64_t>> found((size_t)H);
        for (size_t i = 0; i < (size_t)H; ++i) found[i] = {h_v[i], h_deg[i]};
        std::sort(found.begin(), found.end());
        for (size_t i = 0; i < (size_t)H; ++i) {
            P.hub_v[i] = found[i].first;
            deg[i] = found[i].second;
        }
    } else if (H <= eager) {
        std::memcpy(P.hub_v.data(), h_v, sizeof(int32_t) * (size_t)H);
        std::memcpy(deg.data(), h_deg, sizeof(int64_t) * (size_t)H);
    } else {
        KB_CUDA(ctx, cudaMemcpyAsync(P.hub_v.data(), b + C.hub_v, sizeof(int32_t) * (size_t)H, cudaMemcpyDeviceToHost, s));
        KB_CUDA(ctx, cudaMemcpyAsync(deg.data(), b + C.hub_deg, sizeof(int64_t) * (size_t)H, cudaMemcpyDeviceToHost, s));
        KB_CUDA(ctx, cudaStreamSynchronize(s));
    }
    P.chunk_off.resize((size_t)H + 1);
    P.set_off.resize((size_t)H + 1);
    for (size_t i = 0; i < (size_t)H; ++i) {
        P.chunk_off[i + 1] = P.chunk_off[i] + (deg[i] + P.hub_chunk - 1) / P.hub_chunk;
        P.set_off[i + 1] = P.set_off[i] + kb::hub_set_capacity(deg[i]);
    }
    P.n_hubs = (size_t)H;
    P.n_chunks = P.chunk_off[(size_t)H];
    P.set_slots = P.set_off[(size_t)H];
    return KB_OK;
}

// Size class of a call, the key of the tuning cache: single graphs by
// floor(log2) of their processed edges, batches (64 + ...) by floor(log2) of
// the processed edges per graph.
int32_t size_class(int64_t m_proc, int64_t graphs, bool batch) {
    const int64_t per = std::max<int64_t>(1, m_proc / std::max<int64_t>(graphs, 1));
    int32_t c = 0;
    while ((per >> (c + 1)) > 0) ++c;
    return batch ? 64 + c : c;
}

// The cached tuning of class c, else of the nearest class of the same kind
// at most 3 classes (a factor of 8 in edges) away, else nullptr.
const kb_tuning* tuned_for(const kb_context* ctx, int32_t c) {
    const kb_tuning* best = nullptr;
    int32_t dist = 4;
    for (const auto& kv : ctx->tuned) {
        if ((kv.first >= 64) != (c >= 64)) continue;
        const int32_t d = std::abs(kv.first - c);
        if (d < dist) {
            dist = d;
            best = &kv.second;
        }
    }
    return best;
}

int32_t pick_field(int32_t given, int32_t cached, int32_t dflt) { return given ? given : (cached ? cached : dflt); }

// The plan fields a call may choose on a prepared graph: key subject, frozen
// blocks, table size, medium split and warp task size.
void resolve_call_fields(Plan& P, const kb_options* opt, int rounds, bool multi, const kb_tuning* T) {
    P.subject = opt->subject;
    // stratified rounds of one graph, and always of batched and served graphs
    // (multi); incremental refinement plans without, and generic CSE keys need
    // not hold the own previous block
    P.freeze = multi || (rounds >= 0 && P.subject == KB_SUBJECT_PREVIOUS && opt->rekey_all == 0);
    P.dense0 = !multi;
    P.med_split = pick_field(opt->medium_split, T ? T->medium_split : 0, kb::kDefaultMedSplit);
    P.warp_verts = pick_field(opt->small_task_vertices, T ? T->small_task_vertices : 0, 0);
    float lf = opt->load_factor > 0.f ? opt->load_factor : (T ? T->load_factor : 0.f);
    if (!(lf > 0.f)) lf = 0.5f;
    P.cap = table_capacity(P.n, lf);
}

// `rounds`: refinement rounds the call runs (decides the automatic locality
// order); negative for batched and served refinement, which never reorder.
// With P.graph_ext set (building a prepared graph) the automatic locality
// order is on for at least 2^22 processed edges: its cost is paid once.
kb_status make_plan(kb_context* ctx, const kb_graph* g, const kb_options* opt, Plan& P, char** csr_base_out,
                    bool for_query, int rounds, bool multi = false) {
    P.n = g->n;
    P.m = g->m;
    P.dir = opt->direction;
    P.m_proc = P.dir == KB_DIR_BOTH ? 2 * g->m : g->m;
    const bool auto_order = P.graph_ext || rounds >= 24;
    P.reorder = rounds >= 0 && P.n > 0 && P.m_proc > 0 &&
                (opt->reorder == 2 || (opt->reorder == 0 && auto_order && P.m_proc >= ((int64_t)1 << 22)));
    P.labels = opt->use_edge_labels && g->edge_labels != nullptr;
    // tuning fields: the options' value, else the cached tuning of the call's
    // size class, else the library default
    P.size_class = size_class(P.m_proc, multi ? ctx->plan_graphs : 1, multi);
    const kb_tuning* T = tuned_for(ctx, P.size_class);
    P.thr = pick_field(opt->hub_threshold, T ? T->hub_threshold : 0, kb::kDefaultHubThreshold);
    P.hub_chunk = pick_field(opt->hub_chunk_edges, T ? T->hub_chunk_edges : 0, kb::kDefaultHubChunk);
    P.small_max = std::min(pick_field(opt->small_max_degree, T ? T->small_max_degree : 0, kb::kMidDegree), P.thr);
    resolve_call_fields(P, opt, rounds, multi, T);
    layout_csr(P);
    const int64_t* row_p = g->row_offsets;
    char* csr_base = nullptr;
    if (needs_in_csr(P.dir)) {
        // The processed CSR is needed to find hubs; during a size query it is
        // built in library scratch, otherwise at the head of the workspace.
        if (for_query) {
            KB_TRY(ensure_buffer(ctx, &ctx->plan_tmp, &ctx->plan_tmp_bytes, P.csr_bytes));
            csr_base = reinterpret_cast<char*>(ctx->plan_tmp);
        } else {
            csr_base = *csr_base_out;
        }
        KB_TRY(build_processed_csr(ctx, g, P, csr_base));
        row_p = reinterpret_cast<const int64_t*>(csr_base + P.o_rowp);
    }
    const bool check = opt->validate && !for_query;
    kb::CheckIds ids;
    if (check && !needs_in_csr(P.dir)) {
        ids.a[0] = g->col_indices;
        ids.count[0] = g->m;
    }
    KB_TRY(plan_classes(ctx, P, row_p, check ? kb::CheckRows::kAll : kb::CheckRows::kNone, ids));
    layout_round(P);
    return KB_OK;
}

// Acquire a workspace of `bytes`; returns its base.
kb_status acquire_workspace(kb_context* ctx, size_t bytes, char** base) {
    if (ctx->user_ws) {
        if (bytes > ctx->user_ws_bytes)
            return fail(ctx, KB_ERR_OOM, "caller workspace holds %zu bytes, %zu needed", ctx->user_ws_bytes, bytes);
        *base = reinterpret_cast<char*>(ctx->user_ws);
        return KB_OK;
    }
    KB_TRY(ensure_buffer(ctx, &ctx->own_ws, &ctx->own_ws_bytes, std::max<size_t>(bytes, 256)));
    *base = reinterpret_cast<char*>(ctx->own_ws);
    return KB_OK;
}

struct Timer {
    kb_context* ctx;
    int used = 0;
    int fam[10];
    explicit Timer(kb_context* c) : ctx(c) {}
    void begin(int family) {
        if (!ctx->timing || used >= 10) return;
        fam[used] = family;
        cudaEventRecord(ctx->ev[2 * used], ctx->stream);
    }
    void end() {
        if (!ctx->timing || used >= 10) return;
        cudaEventRecord(ctx->ev[2 * used + 1], ctx->stream);
        ++used;
    }
    // after a stream sync
    float collect() {
        float round = 0.f;
        if (!ctx->timing) return 0.f;
        for (int i = 0; i < used; ++i) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, ctx->ev[2 * i], ctx->ev[2 * i + 1]);
            ctx->kernel_ms[fam[i]] += ms;
            ctx->kernel_launches[fam[i]] += 1;
            round += ms;
        }
        if (used > 0) {
            float span = 0.f;
            cudaEventElapsedTime(&span, ctx->ev[0], ctx->ev[2 * used - 1]);
            round = span;
        }
        used = 0;
        return round;
    }
};

// Everything one refine call needs on the device: the plan, the bound round
// parameters and the table epoch.
struct Prepared {
    Plan P;
    char* ws = nullptr;  // workspace base (round buffers)
    kb::RoundParams p{};
    uint2* prefix = nullptr;  // rank words of the renumbering (launch_renumber)
    uint32_t* scan_tmp = nullptr;
    uint8_t* gactive = nullptr;  // several graphs: those that refine
    int64_t total_chunks = 0;
    size_t set_bytes = 0;
    uint32_t epoch_own = 0, round_own = 0;
    uint32_t* epoch = nullptr;  // last table epoch used, and rounds since the minima were cleared: the two
    uint32_t* round = nullptr;  //   above, or the context's with its table
    size_t table_bytes = 0, emin_bytes = 0;
    // frozen blocks for the next round and their minima, edgeless vertices
    // (Plan::freeze; RoundParams::frozen)
    uint32_t* frozen = nullptr;
    uint32_t* frozen_min = nullptr;
    uint32_t* edgeless = nullptr;
    // clean blocks (frozen blocks on): moved vertices and marked (dirty)
    // blocks; RoundParams::minof
    bool bitmap_fresh = false, counters_fresh = false;  // both clear since prepare
    bool bitmap_ready = false;  // the round's bitmap holds the minima of its frozen blocks already
    bool counters_clear = false;  // the round need not clear the counters (no errors so far; see launch_renumber)
    uint32_t* moved = nullptr;
    uint32_t* mark = nullptr;
    const int32_t* key_checked = nullptr;  // level-0 keys whose label minima are in ctx->d_dense,
    bool key_dense = false;                //   and whether they are all small (launch_dense_labels)
    const uint32_t* class_bits[3] = {};  // mid, medium and hub vertices; nullptr: an empty class
    bool compact = false;  // small-kernel windows skip frozen vertices (many frozen)
    bool sparse = false;   // fewer than 1/64 of the vertices refine: long warp tasks
    // A caller-held block table (ext_cap slots) and empty-signature minima
    // (at least n entries) that outlive one prepare: they are neither carved
    // from the workspace nor cleared, and the table epoch carries on (the
    // server re-plans its arena at every admission).
    uint64_t* ext_table = nullptr;
    uint64_t ext_cap = 0;
    uint64_t* ext_emin = nullptr;
    // Likewise the frozen-block state (frozen, frozen_min, shared, minof,
    // moved, mark; bitmaps of at least n bits, minof of n entries): kept as it
    // is by prepare, so that blocks stay frozen across a re-plan that moves
    // no vertex (the server's admissions, which append at the arena's tail).
    uint32_t* ext_frozen = nullptr;
    uint32_t* ext_frozen_min = nullptr;
    uint32_t* ext_shared = nullptr;
    uint32_t* ext_minof = nullptr;
    uint32_t* ext_moved = nullptr;
    uint32_t* ext_mark = nullptr;
    bool class_on[3] = {true, true, true};  // some mid vertex, medium vertex, hub refines this round
};

// Bind the per-graph part of a plan into p: the processed CSR (csr: IN /
// BOTH), the hub lists, the locality order and the medium list (gws: graph
// part base).  build: also fill them (hub lists uploaded, chunk extents, the
// locality order, using `count_tmp` (n words) as scratch, the medium list and
// the degree-class bitmaps); else they hold a prepared graph's contents.
kb_status bind_graph_part(kb_context* ctx, const kb_graph* g, const Plan& P, char* csr, char* gws, bool build,
                          uint32_t* count_tmp, kb::RoundParams& p, cudaStream_t s) {
    const int64_t n = g->n;
    if (needs_in_csr(P.dir)) {
        p.row = reinterpret_cast<const int64_t*>(csr + P.o_rowp);
        p.col = reinterpret_cast<const int32_t*>(csr + P.o_colp);
        p.lab = P.labels ? reinterpret_cast<const int32_t*>(csr + P.o_labp) : nullptr;
    } else {
        p.row = g->row_offsets;
        p.col = g->col_indices;
        p.lab = P.labels ? g->edge_labels : nullptr;
    }
    const size_t H = P.n_hubs;
    p.n_hubs = (int32_t)H;
    p.hub_v = reinterpret_cast<const int32_t*>(gws + P.o_hubv);
    p.hub_chunk_off = reinterpret_cast<const int64_t*>(gws + P.o_chunk);
    p.hub_set_off = reinterpret_cast<const int64_t*>(gws + P.o_setoff);
    p.chunk_hub = reinterpret_cast<const int32_t*>(gws + P.o_chunkhub);
    p.chunk_ext = reinterpret_cast<const uint64_t*>(gws + P.o_chunkext);
    if (build && H) {
        // the three lists lie one after another: one copy
        std::vector<char> up(P.o_setoff + sizeof(int64_t) * (H + 1) - P.o_hubv);
        std::memcpy(up.data(), P.hub_v.data(), sizeof(int32_t) * H);
        std::memcpy(up.data() + (P.o_chunk - P.o_hubv), P.chunk_off.data(), sizeof(int64_t) * (H + 1));
        std::memcpy(up.data() + (P.o_setoff - P.o_hubv), P.set_off.data(), sizeof(int64_t) * (H + 1));
        // pageable memory: staged before the call returns
        KB_CUDA(ctx, cudaMemcpyAsync(gws + P.o_hubv, up.data(), up.size(), cudaMemcpyHostToDevice, s));
        kb::launch_chunk_ext(P.n_chunks, (int32_t)H, p.hub_v, p.hub_chunk_off, p.row, P.hub_chunk,
                             reinterpret_cast<int32_t*>(gws + P.o_chunkhub),
                             reinterpret_cast<uint64_t*>(gws + P.o_chunkext), s);
        KB_CUDA(ctx, cudaGetLastError());
    }
    if (P.reorder) {
        int32_t* perm = reinterpret_cast<int32_t*>(gws + P.o_perm);
        int32_t* colr = needs_in_csr(P.dir) ? const_cast<int32_t*>(p.col) : reinterpret_cast<int32_t*>(gws + P.o_colr);
        if (build) {
            // rank vertices by how often they are gathered and move the
            // neighbour ids to those ranks
            kb::launch_locality_order(n, P.m_proc, p.col, count_tmp,
                                      reinterpret_cast<unsigned long long*>(gws + P.o_hist), perm, s);
            kb::launch_remap_cols(P.m_proc, p.col, perm, colr, s);
            KB_CUDA(ctx, cudaGetLastError());
        }
        p.col = colr;
        p.perm = perm;
    }
    p.mid_v = reinterpret_cast<int32_t*>(gws + P.o_mid);
    p.n_mid = P.n_mid;
    p.med_v = reinterpret_cast<int32_t*>(gws + P.o_med);
    p.n_med = P.n_med;
    if (build) {
        // the plan's scratch still holds the classes (plan_classes)
        const ClassScratch C(P);
        const char* b = reinterpret_cast<const char*>(ctx->class_tmp);
        const uint32_t* bits = reinterpret_cast<const uint32_t*>(b);
        const int64_t pitch = (int64_t)(P.class_bytes() / sizeof(uint32_t));
        kb::launch_class_lists(n, p.row, bits, pitch, tile_counts(ctx, P, C),
                               {kb::kMid, P.n_mid, const_cast<int32_t*>(p.mid_v), nullptr},
                               {kb::kMedium, P.n_med, const_cast<int32_t*>(p.med_v), nullptr}, s);
        if (P.graph_ext)  // laid out only then
            KB_CUDA(ctx, cudaMemcpyAsync(gws + P.o_classes, b, Plan::kClassBitmaps * P.class_bytes(),
                                         cudaMemcpyDeviceToDevice, s));
        KB_CUDA(ctx, cudaGetLastError());
    }
    return KB_OK;
}

// Bind the block table and the empty-signature minima: the caller's (the
// server's arena), the context's, or with a caller-owned workspace a part of it.
kb_status bind_table(kb_context* ctx, const Plan& P, Prepared& R, cudaStream_t s) {
    kb::RoundParams& p = R.p;
    R.epoch = &R.epoch_own;
    R.round = &R.round_own;
    const size_t table_need = sizeof(uint64_t) * (size_t)P.cap, emin_need = sizeof(uint64_t) * (size_t)P.n;
    if (R.ext_table) {
        p.table = R.ext_table;
        p.mask = R.ext_cap - 1;
        p.emin = R.ext_emin;
        R.table_bytes = sizeof(uint64_t) * (size_t)R.ext_cap;
        return KB_OK;
    }
    p.mask = P.cap - 1;
    if (ctx->user_ws) {
        p.table = reinterpret_cast<uint64_t*>(R.ws + P.o_table);
        p.emin = reinterpret_cast<uint64_t*>(R.ws + P.o_emin);
        R.table_bytes = table_need;
        R.emin_bytes = emin_need;
        R.epoch_own = R.round_own = 0;
        KB_CUDA(ctx, cudaMemsetAsync(p.table, 0, table_need, s));
        KB_CUDA(ctx, cudaMemsetAsync(p.emin, 0xff, emin_need, s));
        return KB_OK;
    }
    if (ctx->tab_bytes < table_need) {
        KB_TRY(ensure_buffer(ctx, &ctx->tab, &ctx->tab_bytes, table_need));
        KB_CUDA(ctx, cudaMemsetAsync(ctx->tab, 0, ctx->tab_bytes, s));
        ctx->tab_epoch = 0;
    }
    if (ctx->emin_bytes < emin_need) {
        KB_TRY(ensure_buffer(ctx, &ctx->emin, &ctx->emin_bytes, emin_need));
        KB_CUDA(ctx, cudaMemsetAsync(ctx->emin, 0xff, ctx->emin_bytes, s));
        ctx->emin_round = 0;
    }
    p.table = reinterpret_cast<uint64_t*>(ctx->tab);
    p.emin = reinterpret_cast<uint64_t*>(ctx->emin);
    R.table_bytes = ctx->tab_bytes;
    R.emin_bytes = ctx->emin_bytes;
    R.epoch = &ctx->tab_epoch;
    R.round = &ctx->emin_round;
    return KB_OK;
}

// Validate the caller's CSR before its in-edges are counted.  An out-edge CSR is
// checked along with the degree classes (plan_classes), which only read its offsets.
kb_status check_input(kb_context* ctx, const kb_graph* g, const kb_options* opt) {
    if (!opt->validate || !needs_in_csr(opt->direction)) return KB_OK;
    kb::launch_validate(g->n, g->m, g->row_offsets, g->col_indices, ctx->d_ctr, ctx->stream);
    KB_CUDA(ctx, cudaGetLastError());
    KB_TRY(read_counters(ctx));
    return device_error(ctx);
}

// Queue the small-label minima of a level 0 (launch_dense_labels).
kb_status check_small_labels(kb_context* ctx, int64_t n, const int32_t* key) {
    if (!ctx->dense_empty)
        KB_CUDA(ctx, cudaMemsetAsync(ctx->d_dense, 0xff, sizeof(uint32_t) * kb::kDenseLabels, ctx->stream));
    ctx->dense_empty = false;
    kb::launch_dense_labels(n, key, ctx->d_dense, ctx->d_ctr, ctx->stream);
    KB_CUDA(ctx, cudaGetLastError());
    return KB_OK;
}

// Validate, plan, acquire the workspace, bind the round parameters, list the
// medium vertices and reset the per-call state (block table, empty-signature
// minima).  With a prepared graph (pg) only the per-call part is planned and
// reset.  key0: level 0's keys, or nullptr; without pg they are checked for the
// small-label path in the plan's round trip.  Synchronises.
kb_status prepare(kb_context* ctx, const kb_graph* g, const kb_options* opt, Prepared& R, int rounds,
                  bool multi = false, const kb_prepared* pg = nullptr, const int32_t* key0 = nullptr) {
    cudaStream_t s = ctx->stream;
    const int64_t n = g->n;
    KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
    R.counters_fresh = true;
    Plan& P = R.P;
    char* csr = nullptr;
    char* gws = nullptr;
    char* ws = nullptr;
    kb::RoundParams& p = R.p;
    p = kb::RoundParams{};
    p.n = n;
    p.ctr = ctx->d_ctr;
    if (pg) {
        P = pg->P;
        P.ext_table = R.ext_table || !ctx->user_ws;
        P.ext_freeze = R.ext_frozen != nullptr;
        resolve_call_fields(P, opt, rounds, multi, tuned_for(ctx, P.size_class));
        layout_round(P);
        KB_TRY(acquire_workspace(ctx, P.total, &ws));
        csr = pg->csr;
        gws = pg->gbuf;
        KB_TRY(bind_graph_part(ctx, g, P, csr, gws, false, nullptr, p, s));
    } else {
        KB_TRY(check_input(ctx, g, opt));
        if (key0) {
            R.key_checked = key0;
            KB_TRY(check_small_labels(ctx, n, key0));
        }
        // The processed CSR sits at the head of the workspace, so its size is known
        // before the hub layout.
        Plan probe;
        probe.n = n;
        probe.m = g->m;
        probe.dir = opt->direction;
        probe.m_proc = probe.dir == KB_DIR_BOTH ? 2 * g->m : g->m;
        probe.labels = opt->use_edge_labels && g->edge_labels != nullptr;
        layout_csr(probe);
        char* base = nullptr;
        if (probe.csr_bytes) {
            // The hub layout is not known yet: reserve the CSR part first.  A
            // library-owned workspace keeps its contents when it does not grow.
            if (ctx->user_ws) {
                KB_TRY(acquire_workspace(ctx, probe.csr_bytes, &base));
            } else {
                KB_TRY(ensure_buffer(ctx, &ctx->plan_tmp, &ctx->plan_tmp_bytes, probe.csr_bytes));
                base = reinterpret_cast<char*>(ctx->plan_tmp);
            }
        }
        P.ext_table = R.ext_table || !ctx->user_ws;
        P.ext_freeze = R.ext_frozen != nullptr;
        KB_TRY(make_plan(ctx, g, opt, P, &base, false, rounds, multi));
        if (ctx->user_ws) {
            KB_TRY(acquire_workspace(ctx, P.total, &ws));
        } else {
            // round buffers live in the owned workspace; the CSR stays in plan_tmp
            const size_t csr_bytes = P.csr_bytes;
            P.csr_bytes = 0;
            layout_round(P);
            P.csr_bytes = csr_bytes;
            KB_TRY(ensure_buffer(ctx, &ctx->own_ws, &ctx->own_ws_bytes, std::max<size_t>(P.total, 256)));
            ws = reinterpret_cast<char*>(ctx->own_ws);
        }
        csr = base;
        gws = ws;
        R.key_dense = R.key_checked && ctx->h_ctr->dense_bad == 0;
        // the slot array serves as the count buffer of the locality order:
        // every round rewrites it
        KB_TRY(bind_graph_part(ctx, g, P, csr, gws, true, reinterpret_cast<uint32_t*>(ws + P.o_slot), p, s));
    }
    R.ws = ws;
    p.hub_threshold = P.thr;
    p.small_max = std::min(P.small_max, kb::kSmallDegree);
    p.mid_max = P.small_max;
    p.warp_verts = P.warp_verts;
    p.hub_chunk = P.hub_chunk;
    p.med_split = P.med_split;
    p.hash_mode = opt->hash_mode;
    p.slot_of = reinterpret_cast<int32_t*>(ws + P.o_slot);
    KB_TRY(bind_table(ctx, P, R, s));
    p.bitmap = reinterpret_cast<uint32_t*>(ws + P.o_bitmap);
    p.ctr = ctx->d_ctr;
    p.hub_sets = reinterpret_cast<uint64_t*>(ws + P.o_sets);
    p.hub_acc = reinterpret_cast<uint64_t*>(ws + P.o_acc);
    p.hub_cnt = reinterpret_cast<uint32_t*>(ws + P.o_cnt);
    if (P.sketch) {
        p.hub_exact = reinterpret_cast<uint32_t*>(ws + P.o_exact);
        p.exact_list = reinterpret_cast<int32_t*>(ws + P.o_exactlist);
        p.hub_twin = reinterpret_cast<uint32_t*>(ws + P.o_twin);
        p.hub_twin_mask = (uint32_t)(next_pow2(2 * P.n_hubs) - 1);
    }
    if (P.reorder) p.gat = reinterpret_cast<int32_t*>(ws + P.o_gat);
    R.prefix = reinterpret_cast<uint2*>(ws + P.o_prefix);
    R.scan_tmp = reinterpret_cast<uint32_t*>(ws + P.o_scan);
    R.total_chunks = P.n_chunks;
    R.set_bytes = sizeof(uint64_t) * (size_t)P.set_slots;
    if (P.freeze) {
        char* classes = P.graph_ext ? gws + P.o_classes : reinterpret_cast<char*>(ctx->class_tmp);
        R.edgeless = reinterpret_cast<uint32_t*>(classes);
        const int64_t members[3] = {P.n_mid, P.n_med, (int64_t)P.n_hubs};
        for (int c = 0; c < 3; ++c)
            R.class_bits[c] = members[c] ? reinterpret_cast<uint32_t*>(classes + (size_t)(c + 1) * P.class_bytes())
                                         : nullptr;
        p.joined = reinterpret_cast<uint32_t*>(ws + P.o_joined);  // all clear between rounds
        if (R.ext_frozen) {
            // the caller's state, kept as it is
            KB_CUDA(ctx, cudaMemsetAsync(p.joined, 0, sizeof(uint32_t) * (size_t)((n >> 5) + 1), s));
            R.frozen = R.ext_frozen;
            R.frozen_min = R.ext_frozen_min;
            p.shared = R.ext_shared;
            p.minof = R.ext_minof;
            R.moved = R.ext_moved;
            R.mark = R.ext_mark;
        } else {
            // nothing frozen before the starting level; shared starts empty, and
            // the locality order's moved bits are set one by one
            R.frozen = reinterpret_cast<uint32_t*>(ws + P.o_frozen);
            p.shared = reinterpret_cast<uint32_t*>(ws + P.o_shared);
            p.minof = reinterpret_cast<uint32_t*>(ws + P.o_minof);
            R.moved = reinterpret_cast<uint32_t*>(ws + P.o_moved);
            R.mark = reinterpret_cast<uint32_t*>(ws + P.o_mark);
            KB_CUDA(ctx, cudaMemsetAsync(p.bitmap, 0, P.clear_bytes, s));
            R.bitmap_fresh = true;
        }
        KB_CUDA(ctx, cudaGetLastError());
    }
    return KB_OK;
}

// Advance the table epoch (entries of other epochs read as empty); the table
// is cleared once every 255 rounds.
kb_status next_epoch(kb_context* ctx, Prepared& R, cudaStream_t s) {
    if (*R.epoch == 255) {
        KB_CUDA(ctx, cudaMemsetAsync(R.p.table, 0, R.table_bytes, s));
        *R.epoch = 0;
    }
    R.p.epoch = ++*R.epoch;
    return KB_OK;
}

// The round word of the next round's empty-signature minima: smaller than any
// before.
kb_status next_empty_round(kb_context* ctx, Prepared& R, cudaStream_t s) {
    if (*R.round >= 0xffffff00u) {
        KB_CUDA(ctx, cudaMemsetAsync(R.p.emin, 0xff, R.emin_bytes, s));
        *R.round = 0;
    }
    R.p.ehigh = 0xffffffffu - ++*R.round;
    return KB_OK;
}

// The freeze pass after a signature round of one graph or a batch.
kb::FreezePass freeze_pass(kb_context* ctx, const Prepared& R) {
    kb::FreezePass f;
    f.n = R.p.n;
    f.bitmap = R.p.bitmap;
    f.shared = R.p.shared;
    f.edgeless = R.edgeless;
    f.names = R.p.minof;
    f.mark = R.mark;
    f.frozen = R.frozen;
    // straight into the bitmap, which the next round builds on (the server, which
    // can admit and move graphs in between, keeps the minima apart)
    f.frozen_min = R.ext_frozen ? R.frozen_min : R.p.bitmap;
    f.vgraph = R.p.lgraph;
    f.gactive = R.gactive;
    f.moved_clear = R.p.perm ? R.moved : nullptr;
    for (int c = 0; c < 3; ++c) f.classes[c] = R.class_bits[c];
    f.ctr = ctx->d_ctr;
    return f;
}

// Starting level: canonical renumbering of `key` (labels or a given
// partition; all-zero partition when key is NULL in a batched run).
// dense_path: set when the small-label path was taken.
kb_status launch_level0(kb_context* ctx, Prepared& R, const int32_t* key, int32_t* out, cudaStream_t s,
                        bool* dense_path = nullptr) {
    KB_TRY(next_epoch(ctx, R, s));
    if (!R.counters_fresh) KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
    if (!R.bitmap_fresh)
        KB_CUDA(ctx, cudaMemsetAsync(R.p.bitmap, 0, sizeof(uint32_t) * (size_t)((R.p.n >> 5) + 1), s));
    R.counters_fresh = R.bitmap_fresh = false;
    R.p.prev = key;
    R.p.frozen = nullptr;
    R.p.frozen_min = nullptr;
    // small non-negative keys (one graph): each label's smallest vertex
    // directly; the check for the range costs one host round trip, unless it
    // came with the plan's
    bool dense = false;
    if (key && R.P.dense0 && R.p.n > 0) {
        if (key == R.key_checked) {
            dense = R.key_dense;
            R.key_checked = nullptr;
        } else {
            KB_TRY(check_small_labels(ctx, R.p.n, key));
            KB_TRY(read_counters(ctx));
            dense = ctx->h_ctr->dense_bad == 0;
        }
    }
    if (dense_path) *dense_path = dense;
    if (dense) {
        kb::launch_dense_level0(R.p, key, ctx->d_dense, reinterpret_cast<uint2*>(ctx->d_dense + kb::kDenseLabels),
                                R.prefix, R.scan_tmp, out, s);
        ctx->dense_empty = true;
    } else {
        kb::launch_small_round(R.p, true, kb::SmallWindows::kConsecutive, s);
        kb::launch_renumber(R.p, R.prefix, R.scan_tmp, out, nullptr, false, s);
    }
    // a starting level may mix edgeless vertices with others in one block:
    // only its singletons are frozen in the first round
    if (R.p.shared) {
        kb::FreezePass f = freeze_pass(ctx, R);
        f.edgeless = nullptr;
        f.mark = nullptr;
        f.moved_clear = nullptr;
        kb::launch_freeze_clean(f, s);
        R.bitmap_ready = !R.ext_frozen;
    }
    KB_CUDA(ctx, cudaGetLastError());
    return KB_OK;
}

// Up to this many vertices the small, mid and medium vertices of a round that
// keys most of them go in one launch (kb::launch_keys).  It holds four CTAs of the
// small body per SM instead of five, which costs large graphs more than the
// draining between the classes.  Prepared power-law graphs, n = m/6, whole calls
// in us apart / together:
//   edges               3.2e6      6.4e6      1.3e7      2.6e7      5.1e7
//   labelled, out     526/485    692/659    999/949  1618/1584  2742/2735
//   kaushik, in       659/634    888/874  1321/1301  2082/2082  3767/3818
//   schaetzle, out    633/605    938/914  1356/1330  2190/2175  3720/3739
//   labelled, both    551/500    705/669  1054/1002  1664/1621  3023/2998
// and 10^8 edges of 10^7 vertices 4970 / 5080.
constexpr int64_t kKeysVertices = 6 << 20;

// One refinement round up to (not including) the renumbering.
kb_status launch_round_body(kb_context* ctx, Prepared& R, cudaStream_t s, Timer* T) {
    kb::RoundParams& p = R.p;
    // with frozen blocks, the mid, medium and hub kernels run only while some
    // of their vertices refine (after the first rounds, hubs are mostly alone
    // in their blocks)
    const bool mid = p.n_mid && (!p.frozen || R.class_on[0]);
    const bool med = p.n_med && (!p.frozen || R.class_on[1]);
    const bool hub = p.n_hubs && (!p.frozen || R.class_on[2]);
    if (T) T->begin(KB_KERNEL_OTHER);
    if (!R.counters_clear) KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
    if (!R.bitmap_ready) kb::launch_clear_round(p, s);
    R.bitmap_ready = false;
    if (T) T->end();
    if ((mid || med) && !R.compact && !R.sparse && !ctx->timing && p.n <= kKeysVertices) {
        kb::RoundParams q = p;
        if (!mid) q.n_mid = 0;
        if (!med) q.n_med = 0;
        kb::launch_keys(q, s);
    } else {
        if (T) T->begin(KB_KERNEL_SMALL);
        kb::launch_small_round(p, false,
                               R.sparse ? kb::SmallWindows::kSparse
                                        : (R.compact ? kb::SmallWindows::kCompact : kb::SmallWindows::kConsecutive),
                               s);
        if (mid) kb::launch_mid_round(p, s);
        if (T) T->end();
        if (med) {
            if (T) T->begin(KB_KERNEL_MEDIUM);
            kb::launch_medium_round(p, s);
            if (T) T->end();
        }
    }
    if (hub) {
        if (T) T->begin(KB_KERNEL_HUB_CHUNK);
        if (R.P.sketch) kb::launch_hub_sketch(p, R.total_chunks, s);
        kb::launch_clear_hubs(p, (int64_t)(R.set_bytes / sizeof(uint64_t)), s);
        kb::launch_hub_chunk(p, R.total_chunks, s);
        if (T) T->end();
        if (T) T->begin(KB_KERNEL_HUB_FINAL);
        kb::launch_hub_final(p, s);
        if (T) T->end();
    }
    KB_CUDA(ctx, cudaGetLastError());
    return KB_OK;
}

void reset_timing(kb_context* ctx) {
    ctx->round_ms.clear();
    for (int f = 0; f < KB_KERNEL_COUNT; ++f) {
        ctx->kernel_ms[f] = 0.f;
        ctx->kernel_launches[f] = 0;
    }
}

// Where the levels go: the caller's (k+1) x n array, or (fixpoint mode, levels
// == nullptr) two library buffers used in turn.
struct LevelRows {
    int32_t* levels = nullptr;
    int32_t* ping[2] = {nullptr, nullptr};
    int64_t n = 0;
    // optional host copy of `levels` (kb_refine_host): every row is copied on
    // a second stream as soon as it is final, overlapping the later rounds
    int32_t* host = nullptr;
    int32_t* row(int i) const { return levels ? levels + (size_t)i * (size_t)n : ping[i & 1]; }
};

// Queue the device-to-host copy of rows first..last, final on ctx->stream since
// ctx->row_ev was recorded.
kb_status emit_rows(kb_context* ctx, const LevelRows& rows, int first, int last) {
    if (!rows.host || rows.n == 0 || last < first) return KB_OK;
    KB_CUDA(ctx, cudaStreamWaitEvent(ctx->copy_stream, ctx->row_ev, 0));
    KB_CUDA(ctx, cudaMemcpyAsync(rows.host + (size_t)first * (size_t)rows.n, rows.row(first),
                                 sizeof(int32_t) * (size_t)rows.n * (size_t)(last - first + 1), cudaMemcpyDeviceToHost,
                                 ctx->copy_stream));
    return KB_OK;
}

// Waits for the row copies when leaving refine_core by any path, so no copy
// into the caller's host buffer outlives the call.
struct RowCopyGuard {
    cudaStream_t cs;
    ~RowCopyGuard() {
        if (cs) cudaStreamSynchronize(cs);
    }
};

// Graphs up to this size (vertices and processed edges) take the fused kernel.
// Its passes have fewer CTAs in flight (80 registers and the largest of all
// passes' shared memory), so larger graphs lose by it what the launches cost.
// Prepared power-law graphs, whole calls in us without it / with it:
//   vertices + edges     2.3e5      9.3e5      1.9e6      3.7e6      7.5e6
//   labelled, out      374/261    412/329    464/400    542/565    715/717
//   kaushik, in        386/267    462/393    578/498    673/738    909/910
//   schaetzle, out     350/232    459/382    627/555    674/741    946/950
constexpr int64_t kFusedSize = (int64_t)1 << 21;

// Rounds i_start + 1 .. k after the starting level is queued, kb::kFusedRounds at
// a time.  all_on: no freeze pass ran yet.
// key0: the starting level's keys, when it is not queued yet and they are small.
// broken_off: -1, or when the launch was refused or a wait of the kernel ran out
// (then nothing else is reported) the last level that it got to; the level before
// it is whole.
kb_status fused_rounds(kb_context* ctx, Prepared& R, const LevelRows& rows, int i_start, int k, bool stop, bool all_on,
                       const int32_t* key0, int64_t* counts, int* levels_computed, int64_t* last_count,
                       bool* stopped_stable, int* broken_off) {
    cudaStream_t s = ctx->stream;
    *broken_off = -1;
    int reached = i_start;
    kb::FusedRounds a;
    a.p = R.p;
    a.p.prev = reinterpret_cast<const int32_t*>(R.p.minof);  // blocks by name
    a.p.frozen = R.frozen;
    a.p.moved = R.moved;
    a.f = freeze_pass(ctx, R);
    a.rank = R.prefix;
    a.sums = ctx->d_dense + kb::kDenseLabels;  // the pairs, with which the starting level is through
    a.levels = rows.levels;
    a.ping[0] = rows.ping[0];
    a.ping[1] = rows.ping[1];
    a.total_chunks = R.total_chunks;
    a.k = k;
    a.stop_stable = stop;
    a.max_polls = ctx->fused_polls;
    a.edges = R.P.m_proc;
    if (R.p.n_hubs) {
        KB_CUDA(ctx, cudaMemsetAsync(R.p.hub_sets, 0xff, R.set_bytes, s));
        KB_CUDA(ctx, cudaMemsetAsync(R.p.hub_acc, 0, sizeof(uint64_t) * (size_t)R.p.n_hubs, s));
        KB_CUDA(ctx, cudaMemsetAsync(R.p.hub_cnt, 0, sizeof(uint32_t) * (size_t)R.p.n_hubs, s));
    }
    if (all_on && !R.bitmap_fresh)
        KB_CUDA(ctx, cudaMemsetAsync(R.p.bitmap, 0, sizeof(uint32_t) * (size_t)((R.p.n >> 5) + 1), s));
    bool stable = false;
    for (int first = i_start + 1; first <= k && !stable;) {
        // every round takes an epoch of the table and a round word of the minima
        KB_TRY(next_epoch(ctx, R, s));
        KB_TRY(next_empty_round(ctx, R, s));
        a.first = first;
        a.last = std::min({k, first + kb::kFusedRounds - 1, first + (int)(255u - *R.epoch)});
        a.p.epoch = R.p.epoch;
        a.p.ehigh = R.p.ehigh;
        a.all_on = all_on && first == i_start + 1;
        *R.epoch += (uint32_t)(a.last - first);
        *R.round += (uint32_t)(a.last - first);
        a.key0 = first == i_start + 1 ? key0 : nullptr;
        a.lmin = ctx->d_dense;
        if (kb::launch_fused_rounds(a, ctx->fused_ctas, first > i_start + 1, s) != cudaSuccess) {
            cudaGetLastError();  // (an error of the device itself comes back with the next call)
            ++ctx->fused_refused;
            *broken_off = reached;
            return KB_OK;
        }
        ++ctx->fused_launches;
        KB_TRY(read_counters(ctx));
        reached = std::max(reached, (int)ctx->h_ctr->last_round);
        const kb_status st = device_error(ctx);
        if (st == KB_ERR_TIMEOUT) {
            ++ctx->fused_gave_up;
            *broken_off = reached;
            return KB_OK;
        }
        KB_TRY(st);
        if (a.key0) ctx->dense_empty = true;  // (a kernel that gave up may have left minima)
        const Counters& hc = *ctx->h_ctr;
        if (hc.last_round < first || hc.last_round > a.last)
            return fail(ctx, KB_ERR_DEVICE_CHECK, "the fused rounds ended at %d of %d..%d", hc.last_round, first, a.last);
        if (counts && first == i_start + 1) counts[i_start] = hc.start_count;
        for (int i = first; i <= hc.last_round; ++i) {
            ctx->round_ms.push_back(0.f);
            if (counts) counts[i] = hc.round_count[i - first];
        }
        if (last_count) *last_count = hc.count;
        if (levels_computed) *levels_computed = hc.last_round;
        stable = stop && hc.count == hc.prev_count;
        if (stable && counts)
            for (int i = hc.last_round + 1; i <= k; ++i) counts[i] = hc.count;
        first = hc.last_round + 1;
    }
    if (stable && stopped_stable) *stopped_stable = true;
    if (rows.host) {
        KB_CUDA(ctx, cudaEventRecord(ctx->row_ev, s));
        KB_TRY(emit_rows(ctx, rows, key0 ? i_start : i_start + 1, k));
    }
    return KB_OK;
}

// The refinement driver shared by kb_refine, kb_refine_from and
// kb_refine_fixpoint.  counts (k+1 entries) may be NULL in fixpoint mode;
// *last_count receives the block count of the last level computed and
// *stopped_stable whether a round reproduced its input partition.  may_fuse:
// small graphs may run all rounds in one kernel.
kb_status refine_core(kb_context* ctx, const kb_graph* g, const kb_options* opt, const int32_t* start, int i_start,
                      int k, const LevelRows& rows, int64_t* counts, int* levels_computed, int64_t* last_count,
                      bool* stopped_stable = nullptr, const kb_prepared* pg = nullptr, bool may_fuse = true) {
    const int64_t n = g->n;
    const bool fixpoint = rows.levels == nullptr;
    if (levels_computed) *levels_computed = i_start;
    if (stopped_stable) *stopped_stable = false;
    if (n == 0) {
        if (counts)
            for (int i = i_start; i <= k; ++i) counts[i] = 0;
        if (last_count) *last_count = 0;
        return KB_OK;
    }
    cudaStream_t s = ctx->stream;
    ctx->round_keyed.clear();
    RowCopyGuard copies{rows.host ? ctx->copy_stream : nullptr};
    Prepared R;
    const int32_t* init_key = start ? start : (opt->use_vertex_labels ? g->vertex_labels : nullptr);
    KB_TRY(prepare(ctx, g, opt, R, k - i_start, false, pg, opt->subject == KB_SUBJECT_LABEL ? nullptr : init_key));
    kb::RoundParams& p = R.p;

    // ---- the subject part of every key (generic CSE rounds)
    if (R.P.subject) {
        int32_t* own = reinterpret_cast<int32_t*>(R.ws + R.P.o_ownkey);
        if (R.P.subject == KB_SUBJECT_ALL || (R.P.subject == KB_SUBJECT_LABEL && !g->vertex_labels)) {
            kb::launch_fill_i32(own, n, 0, s);
        } else if (R.P.subject == KB_SUBJECT_ID) {
            kb::launch_iota_i32(own, n, s);
        } else {
            // label classes with canonical ids < n (the level-0 pass on the labels)
            KB_TRY(launch_level0(ctx, R, g->vertex_labels, own, s));
            KB_TRY(read_counters(ctx));
            KB_TRY(device_error(ctx));
        }
        KB_CUDA(ctx, cudaGetLastError());
    }

    // Small graphs run all their rounds in one kernel.
    const bool fused = may_fuse && p.minof && ctx->fused_ctas > 0 && !ctx->timing && !ctx->work && !R.P.sketch && k > i_start &&
                       R.P.m_proc + n <= kFusedSize;

    // ---- the starting level
    int32_t* row0 = rows.row(i_start);
    int64_t prev_count = 1;
    bool count_known = true;  // the starting level's block count is on the host
    if (fused && init_key && !R.key_checked && R.P.dense0) {  // (a prepared graph's plan checked no keys)
        KB_TRY(check_small_labels(ctx, n, init_key));
        KB_TRY(read_counters(ctx));
        R.key_checked = init_key;
        R.key_dense = ctx->h_ctr->dense_bad == 0;
    }
    // with the rounds of a small graph when the keys are known to be small
    // (not in place: a kernel that is broken off while it writes the level would leave neither the keys nor the level)
    const bool in_place = init_key < row0 + n && row0 < init_key + n;
    const bool fused0 = fused && init_key && init_key == R.key_checked && R.key_dense && R.counters_fresh &&
                        R.bitmap_fresh && !in_place;
    if (fused0) {
        R.key_checked = nullptr;
    } else if (init_key) {
        bool dense = false;
        KB_TRY(launch_level0(ctx, R, init_key, row0, s, &dense));
        // At most kDenseLabels blocks after the small-label path: how many are
        // frozen decides nothing about the first round, and the count comes
        // back with that round's.
        count_known = !((dense || fused) && R.P.freeze && !ctx->work && k > i_start);
        if (count_known) {
            KB_TRY(read_counters(ctx));
            KB_TRY(device_error(ctx));
            prev_count = ctx->h_ctr->count;
            R.compact = R.P.freeze && ctx->h_ctr->frozen * 4 > n;
            R.sparse = R.P.freeze && (n - ctx->h_ctr->frozen) * 64 < n;
            for (int c = 0; c < 3; ++c) R.class_on[c] = ctx->h_ctr->class_on[c] > 0;
        }
    } else {
        // the count's low byte, for the rounds that compare with the previous one
        KB_CUDA(ctx, cudaMemsetAsync(&ctx->d_ctr->count, 1, 1, s));
        kb::launch_fill_i32(row0, n, 0, s);
        if (p.perm) kb::launch_fill_i32(p.gat, n, 0, s);
        // P_0 = {V}: one block, named by vertex 0 (no freeze pass reads its bitmap)
        if (p.minof) kb::launch_fill_i32(reinterpret_cast<int32_t*>(p.minof), n, 0, s);
    }
    if (counts) counts[i_start] = prev_count;
    if (last_count) *last_count = prev_count;
    if (!fused0) {
        if (rows.host) KB_CUDA(ctx, cudaEventRecord(ctx->row_ev, s));
        KB_TRY(emit_rows(ctx, rows, i_start, i_start));
    }

    if (fused) {
        int broken_off = -1;
        KB_TRY(fused_rounds(ctx, R, rows, i_start, k, opt->early_stop || fixpoint, !init_key, fused0 ? init_key : nullptr,
                            counts, levels_computed, last_count, stopped_stable, &broken_off));
        if (broken_off < 0) return KB_OK;
        // Again, one kernel per pass.  Once the starting level is written, it is
        // started from: the caller's start may be a later row of the levels, which the
        // rounds have overwritten (the two levels of a fixpoint are the library's own).
        const bool level_written = rows.levels && init_key && (!fused0 || broken_off > i_start);
        ctx->round_ms.clear();
        return refine_core(ctx, g, opt, level_written ? row0 : start, i_start, k, rows, counts, levels_computed, last_count,
                           stopped_stable, pg, false);
    }

    // ---- refinement rounds
    R.counters_clear = !R.P.subject;
    for (int i = i_start + 1; i <= k; ++i) {
        Timer T(ctx);
        KB_TRY(next_epoch(ctx, R, s));
        KB_TRY(next_empty_round(ctx, R, s));
        p.prev = rows.row(i - 1);
        p.own_key = R.P.subject ? reinterpret_cast<const int32_t*>(R.ws + R.P.o_ownkey) : nullptr;
        p.frozen = R.frozen;
        p.frozen_min = R.frozen_min;
        if (p.minof) {
            p.prev = reinterpret_cast<const int32_t*>(p.minof);  // blocks by name
            p.moved = R.moved;
        }
        int32_t* out = rows.row(i);
        KB_TRY(launch_round_body(ctx, R, s, &T));
        if (ctx->work) {
            KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr->keyed_v, 0, 6 * sizeof(int64_t), s));
            kb::launch_round_work(p, s);
        }
        T.begin(KB_KERNEL_RENUMBER);
        // under early stop a round that keeps the count is the last one
        const bool stop_stable = (opt->early_stop || fixpoint) && p.minof;
        kb::launch_renumber(p, R.prefix, R.scan_tmp, out, R.mark, stop_stable, s);
        if (rows.host) KB_CUDA(ctx, cudaEventRecord(ctx->row_ev, s));
        // the next round's frozen blocks: singletons; a block formed by this
        // round that holds an edgeless vertex holds only edgeless vertices with
        // one previous block; and clean blocks, none of whose members has an
        // edge to a vertex whose smallest block member this round changed
        if (p.shared && i < k) {
            kb::launch_dirty_blocks(p, R.edgeless, R.moved, kb::kMaxHubThreshold, R.mark, nullptr, stop_stable, s);
            kb::FreezePass f = freeze_pass(ctx, R);
            f.stop_stable = stop_stable;
            kb::launch_freeze_clean(f, s);
            R.bitmap_ready = true;
        }
        T.end();
        // CSE levels need not refine each other: compare whole levels
        if (R.P.subject) kb::launch_levels_differ(out, p.prev, n, ctx->d_ctr, s);
        KB_CUDA(ctx, cudaGetLastError());
        KB_TRY(read_counters(ctx));
        if (ctx->work) {
            const Counters& hc = *ctx->h_ctr;
            ctx->round_keyed.push_back(
                {hc.keyed_v[0], hc.keyed_v[1], hc.keyed_v[2], hc.keyed_e[0], hc.keyed_e[1], hc.keyed_e[2]});
        }
        // compacted small-kernel windows pay once a quarter of the vertices are frozen
        R.compact = R.P.freeze && ctx->h_ctr->frozen * 4 > n;
        R.sparse = R.P.freeze && (n - ctx->h_ctr->frozen) * 64 < n;
        for (int c = 0; c < 3; ++c) R.class_on[c] = ctx->h_ctr->class_on[c] > 0;
        ctx->round_ms.push_back(T.collect());
        KB_TRY(device_error(ctx));
        const int64_t c = ctx->h_ctr->count;
        if (!count_known) {
            prev_count = ctx->h_ctr->prev_count;
            if (counts) counts[i_start] = prev_count;
            count_known = true;
        }
        if (counts) counts[i] = c;
        if (last_count) *last_count = c;
        if (levels_computed) *levels_computed = i;
        const bool unchanged = R.P.subject ? ctx->h_ctr->diff == 0 : c == prev_count;
        if ((opt->early_stop || fixpoint) && unchanged) {
            // stratified levels only split blocks, so an unchanged count means an
            // unchanged partition; generic CSE levels were compared entry by entry
            if (stopped_stable) *stopped_stable = true;
            // with frozen blocks the renumbering left this row to be copied too
            const int src = p.minof ? i - 1 : i;
            if (!fixpoint) {
                kb::launch_copy_rows(rows.levels, n, src, src + 1, k, s);
                if (rows.host) KB_CUDA(ctx, cudaEventRecord(ctx->row_ev, s));
                KB_TRY(emit_rows(ctx, rows, i, k));
            } else if (p.minof) {
                KB_CUDA(ctx, cudaMemcpyAsync(out, rows.row(i - 1), sizeof(int32_t) * (size_t)n,
                                             cudaMemcpyDeviceToDevice, s));
            }
            if (counts)
                for (int j = i + 1; j <= k; ++j) counts[j] = c;
            KB_CUDA(ctx, cudaGetLastError());
            break;
        }
        KB_TRY(emit_rows(ctx, rows, i, i));
        prev_count = c;
    }
    KB_CUDA(ctx, cudaStreamSynchronize(s));
    return KB_OK;
}

kb_status refine_impl(kb_context* ctx, const kb_graph* g, const kb_options* opt, const int32_t* start, int i_start,
                      int k, int32_t* levels, int64_t* counts, int* levels_computed,
                      const kb_prepared* pg = nullptr, int32_t* host_levels = nullptr);

// Incremental refinement (kb_refine_update): levels holds the levels of the
// graph before the change (same options); each round re-keys only the work set
// and keeps the old grouping elsewhere (see kb_update.cu), then renumbers.
kb_status update_impl(kb_context* ctx, const kb_graph* g, const kb_options* opt, int k, const int32_t* changed,
                      int64_t n_changed, int32_t* levels, int64_t* counts, int* levels_computed, int64_t* work) {
    KB_TRY(check_graph(ctx, g, opt, k));
    if (opt->subject != KB_SUBJECT_PREVIOUS)
        return fail(ctx, KB_ERR_INVALID_ARG, "incremental refinement takes subject = KB_SUBJECT_PREVIOUS only");
    if (!counts) return fail(ctx, KB_ERR_INVALID_ARG, "counts is NULL");
    if (n_changed < 0 || (n_changed > 0 && !changed)) return fail(ctx, KB_ERR_INVALID_ARG, "bad changed list");
    const int64_t n = g->n;
    if (n > 0 && !levels) return fail(ctx, KB_ERR_INVALID_ARG, "levels is NULL");
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    reset_timing(ctx);
    if (levels_computed) *levels_computed = 0;
    if (n == 0) {
        for (int i = 0; i <= k; ++i) counts[i] = 0;
        if (work)
            for (int i = 0; i <= k; ++i) work[i] = 0;
        return KB_OK;
    }
    cudaStream_t s = ctx->stream;
    auto row = [&](int i) { return levels + (size_t)i * (size_t)n; };

    // scratch: six bitmaps, the smallest vertex of every old block and, per
    // vertex, of its old block
    const size_t szb = align_up(sizeof(uint32_t) * (size_t)((n >> 5) + 1)), sz4 = align_up(sizeof(int32_t) * (size_t)n);
    KB_TRY(ensure_buffer(ctx, &ctx->upd_buf, &ctx->upd_buf_bytes, 6 * szb + 2 * sz4));
    char* b = reinterpret_cast<char*>(ctx->upd_buf);
    auto bits = [&](int j) { return reinterpret_cast<uint32_t*>(b + (size_t)j * szb); };
    uint32_t *changed_bits = bits(0), *flag = bits(1), *taint = bits(2), *dirty = bits(3), *moved = bits(4), *wmask = bits(5);
    uint32_t* old_min = reinterpret_cast<uint32_t*>(b + 6 * szb);
    uint32_t* old_name = reinterpret_cast<uint32_t*>(b + 6 * szb + sz4);

    // The old levels must be partitions with ids in [0, n); the changed ids too.
    // The first round re-keys at least every vertex of an old level-0 block that
    // holds a changed vertex.  When that is over a quarter of the vertices
    // (level-0 blocks are label classes, often huge), recomputing with the frozen
    // blocks of a full refinement costs less than re-keying whole blocks round
    // after round.
    KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
    KB_CUDA(ctx, cudaMemsetAsync(changed_bits, 0, 3 * szb, s));
    kb::launch_check_ids(n * (int64_t)(k + 1), n, levels, ctx->d_ctr, s);
    kb::launch_changed(n, n_changed, changed, row(0), changed_bits, flag, ctx->d_ctr, s);
    KB_CUDA(ctx, cudaGetLastError());
    KB_TRY(read_counters(ctx));
    if (ctx->h_ctr->err & kb::kErrInvalid)
        return fail(ctx, KB_ERR_INVALID_ARG, "old levels or changed vertices hold ids outside [0, n)");
    if (ctx->h_ctr->work_set * 4 > n) {
        KB_TRY(refine_impl(ctx, g, opt, nullptr, 0, k, levels, counts, levels_computed));
        if (work) {
            const int lc = levels_computed ? *levels_computed : k;
            for (int i = 0; i <= k; ++i) work[i] = i <= lc ? n : 0;
        }
        return KB_OK;
    }

    Prepared R;
    // no locality order: the dirty pass reads neighbour ids, not ranks
    const int32_t* init_key = opt->use_vertex_labels ? g->vertex_labels : nullptr;
    KB_TRY(prepare(ctx, g, opt, R, -1, false, nullptr, init_key));
    kb::RoundParams& p = R.p;

    // level 0 from scratch, in place of the old one; its moved vertices start
    // the dirty set
    p.old_min = old_min;
    p.old_name = old_name;
    p.taint = taint;
    p.keep_old = row(0);
    kb::launch_old_min(n, row(0), old_min, s);
    if (init_key)
        KB_TRY(launch_level0(ctx, R, init_key, row(0), s));
    else
        kb::launch_one_block(p, row(0), s);
    kb::launch_moved(n, nullptr, old_name, taint, moved, ctx->d_ctr, s);
    KB_CUDA(ctx, cudaGetLastError());
    KB_TRY(read_counters(ctx));
    KB_TRY(device_error(ctx));
    counts[0] = init_key ? ctx->h_ctr->count : 1;
    if (work) work[0] = n;

    R.counters_clear = true;
    R.compact = true;  // windows packed from the work set
    for (int i = 1; i <= k; ++i) {
        Timer T(ctx);
        // dirty = changed | moved | predecessors of moved; W = their previous-level blocks
        // (the pass over every edge only when some vertex moved)
        const bool any_moved = ctx->h_ctr->moved > 0;
        if (any_moved) kb::launch_dirty_from_moved(n, R.P.m_proc, p.row, p.col, moved, dirty, s);
        kb::launch_work_set(n, row(i - 1), changed_bits, moved, any_moved ? dirty : nullptr, flag, wmask, ctx->d_ctr, s);
        kb::launch_old_min(n, row(i), old_min, s);
        KB_CUDA(ctx, cudaMemsetAsync(taint, 0, szb, s));
        KB_TRY(next_epoch(ctx, R, s));
        KB_TRY(next_empty_round(ctx, R, s));
        p.prev = row(i - 1);
        p.vmask = wmask;
        p.keep_old = row(i);
        KB_TRY(launch_round_body(ctx, R, s, &T));
        kb::launch_keep_bits(n, wmask, row(i), old_min, p.bitmap, s);
        T.begin(KB_KERNEL_RENUMBER);
        kb::launch_renumber(p, R.prefix, R.scan_tmp, row(i), nullptr, false, s);
        T.end();
        kb::launch_moved(n, wmask, old_name, taint, moved, ctx->d_ctr, s);
        KB_CUDA(ctx, cudaGetLastError());
        KB_TRY(read_counters(ctx));
        ctx->round_ms.push_back(T.collect());
        KB_TRY(device_error(ctx));
        counts[i] = ctx->h_ctr->count;
        if (work) work[i] = ctx->h_ctr->work_set;
        if (levels_computed) *levels_computed = i;
        if (opt->early_stop && counts[i] == counts[i - 1]) {
            if (i < k) kb::launch_copy_rows(levels, n, i, i + 1, k, s);
            for (int j = i + 1; j <= k; ++j) {
                counts[j] = counts[i];
                if (work) work[j] = 0;
            }
            KB_CUDA(ctx, cudaGetLastError());
            break;
        }
    }
    KB_CUDA(ctx, cudaStreamSynchronize(s));
    return KB_OK;
}

kb_status refine_impl(kb_context* ctx, const kb_graph* g, const kb_options* opt, const int32_t* start, int i_start,
                      int k, int32_t* levels, int64_t* counts, int* levels_computed, const kb_prepared* pg,
                      int32_t* host_levels) {
    KB_TRY(check_graph(ctx, g, opt, k));
    if (i_start < 0 || i_start > k) return fail(ctx, KB_ERR_INVALID_ARG, "i_start must be in [0, k]");
    if (!counts) return fail(ctx, KB_ERR_INVALID_ARG, "counts is NULL");
    if (g->n > 0 && !levels) return fail(ctx, KB_ERR_INVALID_ARG, "levels is NULL");
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    reset_timing(ctx);
    LevelRows rows;
    rows.levels = levels;
    rows.n = g->n;
    rows.host = host_levels;
    if (host_levels && !ctx->copy_stream) {
        KB_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
        KB_CUDA(ctx, cudaEventCreateWithFlags(&ctx->row_ev, cudaEventDisableTiming));
    }
    return refine_core(ctx, g, opt, start, i_start, k, rows, counts, levels_computed, nullptr, nullptr, pg);
}

// Summary graph of (src_level, dst_level): distinct triples in order of first
// occurrence (see kb_summary in kbisim.h).  Scratch is library-owned and
// grow-only (released by kb_destroy), like the refinement workspace.
kb_status summary_impl(kb_context* ctx, const kb_graph* g, int direction, int use_edge_labels,
                       const int32_t* src_level, const int32_t* dst_level, int32_t* out_src, int32_t* out_label,
                       int32_t* out_dst, int64_t capacity, int64_t* count) {
    if (!g || !count) return fail(ctx, KB_ERR_INVALID_ARG, "graph and count must not be NULL");
    if (g->n < 0 || g->m < 0 || g->n > 2147483646LL) return fail(ctx, KB_ERR_INVALID_ARG, "bad n or m");
    if (g->m >= ((int64_t)1 << 32)) return fail(ctx, KB_ERR_INVALID_ARG, "the summary graph takes m < 2^32");
    if (direction != KB_DIR_OUT && direction != KB_DIR_IN)
        return fail(ctx, KB_ERR_INVALID_ARG, "direction must be out or in (call once per direction)");
    if (capacity < 0) return fail(ctx, KB_ERR_INVALID_ARG, "negative capacity");
    if (g->n > 0 && (!g->row_offsets || !src_level || !dst_level))
        return fail(ctx, KB_ERR_INVALID_ARG, "row_offsets and levels must not be NULL");
    if (g->m > 0 && !g->col_indices) return fail(ctx, KB_ERR_INVALID_ARG, "col_indices is NULL");
    if (capacity > 0 && (!out_src || !out_label || !out_dst))
        return fail(ctx, KB_ERR_INVALID_ARG, "output arrays must not be NULL when capacity > 0");
    *count = 0;
    if (g->m == 0) return KB_OK;
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->stream;
    const int64_t m = g->m;
    const uint64_t cap = std::max<uint64_t>(1024, next_pow2((uint64_t)(m + m / 4 + 64)));
    const int64_t nw = (m >> 5) + 1;
    const size_t sz_table = 16 * (size_t)cap, sz_bitmap = 4 * (size_t)nw,
                 sz_prefix = 4 * (size_t)(nw + 1), sz_scan = 4 * kb::scan_tmp_words(nw);
    const size_t total = align_up(sz_table) + align_up(sz_bitmap) + align_up(sz_prefix) + align_up(sz_scan);
    KB_TRY(ensure_buffer(ctx, &ctx->sum_buf, &ctx->sum_buf_bytes, total));
    char* base = reinterpret_cast<char*>(ctx->sum_buf);
    kb::SummaryParams q{};
    q.n = g->n;
    q.m = m;
    q.row = g->row_offsets;
    q.col = g->col_indices;
    q.lab = use_edge_labels ? g->edge_labels : nullptr;
    q.dir = direction;
    q.lsrc = src_level;
    q.ldst = dst_level;
    size_t off = 0;
    q.table = reinterpret_cast<unsigned long long*>(base + off);
    off += align_up(sz_table);
    q.bitmap = reinterpret_cast<uint32_t*>(base + off);
    off += align_up(sz_bitmap);
    uint32_t* prefix = reinterpret_cast<uint32_t*>(base + off);
    off += align_up(sz_prefix);
    uint32_t* scan_tmp = reinterpret_cast<uint32_t*>(base + off);
    q.mask = cap - 1;
    q.ctr = ctx->d_ctr;
    kb_status st = KB_OK;
    auto run = [&]() -> kb_status {
        KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
        KB_CUDA(ctx, cudaMemsetAsync(q.table, 0, sz_table, s));
        KB_CUDA(ctx, cudaMemsetAsync(q.bitmap, 0, sz_bitmap, s));
        kb::launch_validate(g->n, m, g->row_offsets, g->col_indices, ctx->d_ctr, s);
        // (the insert does nothing when that found something)
        kb::launch_summary_insert(q, s);
        kb::launch_bitmap_rank(q.bitmap, nw, scan_tmp, prefix, ctx->d_ctr, s);
        KB_CUDA(ctx, cudaGetLastError());
        KB_TRY(read_counters(ctx));
        if (ctx->h_ctr->err & kb::kErrTableFull) return fail(ctx, KB_ERR_TABLE_FULL, "summary table probe limit reached");
        KB_TRY(device_error(ctx));
        *count = ctx->h_ctr->count;
        if (*count > capacity)
            return fail(ctx, KB_ERR_INVALID_ARG, "capacity %lld is below the %lld summary edges", (long long)capacity,
                        (long long)*count);
        kb::launch_summary_emit(q, prefix, out_src, out_label, out_dst, s);
        KB_CUDA(ctx, cudaGetLastError());
        return KB_OK;
    };
    st = run();
    if (cudaStreamSynchronize(s) != cudaSuccess && st == KB_OK) st = fail(ctx, KB_ERR_CUDA, "summary graph failed");
    return st;
}

// Rounds until the partition is stable (or max_rounds), keeping only the
// last two levels.
kb_status fixpoint_impl(kb_context* ctx, const kb_graph* g, const kb_options* opt, const int32_t* initial,
                        int max_rounds, int32_t* final_level, int64_t* count, int* rounds, int* stable) {
    KB_TRY(check_graph(ctx, g, opt, max_rounds));
    if (!count || !rounds) return fail(ctx, KB_ERR_INVALID_ARG, "count and rounds must not be NULL");
    if (g->n > 0 && !final_level) return fail(ctx, KB_ERR_INVALID_ARG, "final_level is NULL");
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    reset_timing(ctx);
    const int64_t n = g->n;
    LevelRows rows;
    rows.n = n;
    if (n > 0) {
        const size_t half = (sizeof(int32_t) * (size_t)n + 255) & ~(size_t)255;
        KB_TRY(ensure_buffer(ctx, &ctx->fix_buf, &ctx->fix_buf_bytes, 2 * half));
        rows.ping[0] = reinterpret_cast<int32_t*>(ctx->fix_buf);
        rows.ping[1] = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ctx->fix_buf) + half);
    }
    int last = 0;
    int64_t c = 0;
    bool st = false;
    KB_TRY(refine_core(ctx, g, opt, initial, 0, max_rounds, rows, nullptr, &last, &c, &st));
    *rounds = last;
    *count = c;
    if (stable) *stable = (st || n == 0) ? 1 : 0;
    if (n == 0) return KB_OK;
    KB_CUDA(ctx, cudaMemcpyAsync(final_level, rows.row(last), sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice,
                                 ctx->stream));
    KB_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return KB_OK;
}

// Batched refinement of G graphs held as one disjoint union (see
// kb_refine_batch in kbisim.h).  Blocks go by their smallest member while the
// rounds run: the own previous block is part of every key, so vertices of
// different graphs never share a block, and level 0 hashes the graph id into the
// key.  Stopping is decided per graph on the device, which freezes all blocks of
// a stopped graph.  The host queues every round before it looks at the one
// before, and stops once no graph refines.
constexpr size_t kBatchStage = 512 << 10;  // some 30,000 graphs
kb_status batch_impl(kb_context* ctx, const kb_graph* g, const int64_t* voff_h, int64_t G, const int32_t* k_h,
                     const kb_options* opt, int32_t* levels, int64_t* counts, int32_t* lc_out) {
    if (!g || !opt) return fail(ctx, KB_ERR_INVALID_ARG, "graph and options must not be NULL");
    if (G < 0 || G > (int64_t)1 << 30) return fail(ctx, KB_ERR_INVALID_ARG, "bad graph count");
    if (G > 0 && (!voff_h || !k_h || !counts)) return fail(ctx, KB_ERR_INVALID_ARG, "NULL batch arrays");
    int kmax = 0;
    for (int64_t j = 0; j < G; ++j) {
        if (k_h[j] < 0) return fail(ctx, KB_ERR_INVALID_ARG, "k of graph %lld is negative", (long long)j);
        kmax = std::max(kmax, (int)k_h[j]);
        if (voff_h[j + 1] < voff_h[j]) return fail(ctx, KB_ERR_INVALID_ARG, "graph_vertex_offsets not monotone");
    }
    if (G > 0 && (voff_h[0] != 0 || voff_h[G] != g->n))
        return fail(ctx, KB_ERR_INVALID_ARG, "graph_vertex_offsets must run from 0 to n");
    KB_TRY(check_graph(ctx, g, opt, kmax));
    if (opt->subject != KB_SUBJECT_PREVIOUS)
        return fail(ctx, KB_ERR_INVALID_ARG, "batched refinement takes subject = KB_SUBJECT_PREVIOUS only");
    const int64_t n = g->n;
    if (G == 0) return KB_OK;
    for (int64_t j = 0; j < G * (kmax + 1); ++j) counts[j] = 0;
    if (lc_out)
        for (int64_t j = 0; j < G; ++j) lc_out[j] = 0;
    if (n == 0) return KB_OK;
    if (!levels) return fail(ctx, KB_ERR_INVALID_ARG, "levels is NULL");
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    reset_timing(ctx);
    cudaStream_t s = ctx->stream;
    Prepared R;
    ctx->plan_graphs = G;
    const kb_status pst = prepare(ctx, g, opt, R, -1, true);
    ctx->plan_graphs = 1;
    KB_TRY(pst);
    kb::RoundParams& p = R.p;

    // batch scratch
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += align_up(b); return o; };
    const size_t o_vgraph = take(sizeof(int32_t) * (size_t)n);
    const size_t o_voff = take(sizeof(int64_t) * (size_t)(G + 1));
    const size_t o_k = take(sizeof(int32_t) * (size_t)G);
    const size_t o_act = take((size_t)G);
    const size_t o_last = take(sizeof(int32_t) * (size_t)G);
    const size_t up_bytes = off - o_voff;  // voff .. glast
    const size_t o_bases = take(sizeof(uint32_t) * (size_t)(G + 1) * (size_t)(kmax + 1));
    KB_TRY(ensure_buffer(ctx, &ctx->batch_ws, &ctx->batch_ws_bytes, off));
    char* b = reinterpret_cast<char*>(ctx->batch_ws);
    int32_t* vgraph = reinterpret_cast<int32_t*>(b + o_vgraph);
    int64_t* voff = reinterpret_cast<int64_t*>(b + o_voff);
    int32_t* kd = reinterpret_cast<int32_t*>(b + o_k);
    uint8_t* gact = reinterpret_cast<uint8_t*>(b + o_act);
    int32_t* glast = reinterpret_cast<int32_t*>(b + o_last);
    uint32_t* bases = reinterpret_cast<uint32_t*>(b + o_bases);
    // From the host in one copy (staged before it returns), but with many graphs what
    // is here already from where it lies: filling a buffer with it took longer than the
    // copies (5 x 10^6 graphs of two vertices: 38.4 -> 44.7 ms).
    const bool together = up_bytes <= kBatchStage;
    const size_t up_from = together ? o_voff : o_act, up_to = together ? o_voff + up_bytes : o_last;
    std::vector<char> up(up_to - up_from, 0);
    if (together) {
        std::memcpy(up.data(), voff_h, sizeof(int64_t) * (size_t)(G + 1));
        std::memcpy(up.data() + (o_k - o_voff), k_h, sizeof(int32_t) * (size_t)G);
    } else {
        KB_CUDA(ctx, cudaMemcpyAsync(voff, voff_h, sizeof(int64_t) * (size_t)(G + 1), cudaMemcpyHostToDevice, s));
        KB_CUDA(ctx, cudaMemcpyAsync(kd, k_h, sizeof(int32_t) * (size_t)G, cudaMemcpyHostToDevice, s));
        KB_CUDA(ctx, cudaMemsetAsync(glast, 0, sizeof(int32_t) * (size_t)G, s));
    }
    for (int64_t j = 0; j < G; ++j) up[o_act - up_from + (size_t)j] = k_h[j] > 0 ? 1 : 0;
    KB_CUDA(ctx, cudaMemcpyAsync(b + up_from, up.data(), up.size(), cudaMemcpyHostToDevice, s));
    kb::launch_vertex_graph(voff, (int32_t)G, n, vgraph, s);
    p.voff = voff;
    p.n_graphs = (int32_t)G;
    p.lgraph = vgraph;
    R.gactive = gact;

    // level 0 for every graph: key (graph, label) or (graph) without labels
    p.vgraph = vgraph;
    p.gbase_cur = bases;
    KB_TRY(launch_level0(ctx, R, opt->use_vertex_labels ? g->vertex_labels : nullptr, levels, s));

    // rounds 1..kmax
    p.vgraph = nullptr;  // block names tell the graphs apart
    R.counters_clear = true;
    cudaEvent_t e0 = ctx->ev[20], e1 = ctx->ev[21];
    KB_CUDA(ctx, cudaEventRecord(e0, s));
    int last = 0;  // last round queued
    for (int i = 1; i <= kmax; ++i) {
        KB_TRY(next_epoch(ctx, R, s));
        KB_TRY(next_empty_round(ctx, R, s));
        p.prev = reinterpret_cast<const int32_t*>(p.minof);
        p.gbase_prev = bases + (size_t)(i - 1) * (size_t)(G + 1);
        p.gbase_cur = bases + (size_t)i * (size_t)(G + 1);
        // frozen blocks as in a single-graph call (blocks never span graphs); the
        // mid, medium and hub kernels always launch (nothing is known of the
        // round before yet)
        p.frozen = R.frozen;
        p.frozen_min = R.frozen_min;
        p.moved = R.moved;
        // from round 2 on, windows packed from the vertices that refine
        // (frozen blocks and stopped graphs take no lane)
        R.compact = i >= 2;
        KB_TRY(launch_round_body(ctx, R, s, nullptr));
        kb::GraphStop stop;
        stop.active = gact;
        stop.round = i;
        stop.k = kd;
        stop.early = opt->early_stop != 0;
        stop.last = glast;
        kb::launch_renumber(p, R.prefix, R.scan_tmp, levels + (size_t)i * (size_t)n, R.mark, false, s, stop);
        if (i < kmax) {
            kb::launch_dirty_blocks(p, R.edgeless, R.moved, kb::kMaxHubThreshold, R.mark, gact, false, s);
            kb::launch_freeze_clean(freeze_pass(ctx, R), s);
            R.bitmap_ready = true;
        }
        KB_CUDA(ctx, cudaGetLastError());
        KB_TRY(queue_counters(ctx, i));
        last = i;
        if (i >= 2) {
            KB_TRY(wait_counters(ctx, i - 1));
            if (ctx->h_ctr->graphs_on == 0) break;  // this round repeated the last levels
        }
    }
    KB_CUDA(ctx, cudaEventRecord(e1, s));
    // the remaining rows repeat the last one
    kb::launch_copy_rows(levels, n, last, last + 1, kmax, s);

    // results: per-graph counts, last refined level
    std::vector<uint32_t> bases_h((size_t)(G + 1) * (size_t)(last + 1));
    KB_CUDA(ctx, cudaMemcpyAsync(bases_h.data(), bases, sizeof(uint32_t) * bases_h.size(), cudaMemcpyDeviceToHost, s));
    if (lc_out) KB_CUDA(ctx, cudaMemcpyAsync(lc_out, glast, sizeof(int32_t) * (size_t)G, cudaMemcpyDeviceToHost, s));
    KB_TRY(read_counters(ctx));
    KB_TRY(device_error(ctx));
    if (kmax > 0) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ctx->round_ms.push_back(ms);
    }
    for (int64_t j = 0; j < G; ++j)
        for (int i = 0; i <= kmax; ++i) {
            const uint32_t* bi = bases_h.data() + (size_t)std::min(i, last) * (size_t)(G + 1);
            counts[j * (kmax + 1) + i] = (int64_t)(bi[j + 1] - bi[j]);
        }
    return KB_OK;
}


// ============================================================================
// Serving: continuous batching over a device arena (see kb_server_* in
// kbisim.h).  Every admitted request owns one graph slot of the arena, in
// arena order; retired slots stay as dead ranges until a compaction packs the
// live ones into the other arena buffer.
// ============================================================================
struct Arena {
    int64_t* row = nullptr;   // [Ncap+1]
    int32_t* col = nullptr;   // [Mcap]
    int32_t* lab = nullptr;   // [Mcap]
    int32_t* vlab = nullptr;  // [Ncap]
    uint32_t* name = nullptr;  // [Ncap] smallest member of every vertex's block (RoundParams::minof)
};

struct ServeRequest {
    int64_t ticket = 0;
    int state = 0;  // 0 waiting, 1 running, 2 done, 3 failed (rejected at admission)
    int64_t n = 0, m = 0, m_proc = 0;
    // the caller's host arrays, read at admission (lab / vlab null when unused)
    const int64_t* row = nullptr;
    const int32_t* col = nullptr;
    const int32_t* lab = nullptr;
    const int32_t* vlab = nullptr;
    kb_options opt;
    int k = 0;
    int slot = -1;
    int round = 0;  // next level to compute (0 = level 0)
    int32_t* d_levels = nullptr;
    size_t level_bytes = 0;
    int32_t* out = nullptr;               // caller's host levels, or null: kept in `levels`
    bool early_rows = false;              // rows go to `out` as soon as they are final (kEarlyRowBytes)
    int rows_queued = 0;                  // rows whose copies to `out` are queued
    bool draining = false;                // finished but for the copies of its levels (state 1)
    std::unique_ptr<int32_t[]> levels;    // host copy after completion (when out is null)
    std::vector<int64_t> counts;
    int32_t levels_computed = 0;
    double t_submit = 0, t_done = 0;
    std::string error;
};

// Device copy of a waiting request's host arrays (and room for its processed
// CSR).  Two of them, so that the next request's copies run while one is
// checked and placed.
struct Stage {
    void* buf = nullptr;
    size_t bytes = 0;
    size_t o_row = 0, o_col = 0, o_lab = 0, o_vlab = 0, o_csr = 0;
    int64_t ticket = 0;           // whose arrays it holds (0: nobody's)
    cudaEvent_t full = nullptr;   // copied
    cudaEvent_t free = nullptr;   // placed: may be overwritten
};

// A finished request's level store, returned once the copies out of it are done.
struct Draining {
    int64_t ticket;
    int32_t* d_levels;
    size_t level_bytes;
};

struct Slot {
    int64_t ticket = -1;  // -1: dead
    int64_t vbase = 0, n = 0, ebase = 0, m = 0;
};

// Rows of at least this size go to a pinned host buffer one by one, as soon as
// they are final, while the next rounds run (a copy costs the host about what
// the link takes for 400 KB); smaller ones together when the request finishes.
constexpr size_t kEarlyRowBytes = 512 << 10;

double now_s() {
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

}  // namespace

struct kb_server {
    kb_context* ctx = nullptr;
    kb_server_config cfg{};
    std::string last_error;
    std::mutex mu;  // guards queue, requests, stats (submit vs step)
    Arena arena[2];
    int cur = 0;  // active arena buffer
    int64_t n_used = 0, m_used = 0;
    std::vector<Slot> slots;
    std::deque<int64_t> waiting;
    std::map<int64_t, ServeRequest> reqs;
    int64_t next_ticket = 1;
    size_t level_bytes_in_use = 0;
    // level stores are reused: freed ones wait in a list per power-of-two size
    std::map<size_t, std::vector<int32_t*>> level_pool;
    // block table and empty-signature minima of the arena, kept across re-plans
    uint64_t* table = nullptr;
    uint64_t table_cap = 0;
    uint64_t* emin = nullptr;
    // Frozen-block state of the arena, sized for a full arena and kept across
    // re-plans: frozen vertices, minima of frozen blocks, shared marks, moved
    // vertices, dirty blocks (and Arena::name).
    uint32_t* frz[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    int64_t planned_n = 0;        // arena vertices at the last re-plan
    bool vertices_moved = false;  // a compaction since the last re-plan
    // Block names are those of the last step, against which this step's moved
    // vertices are told (false after a compaction, which renames blocks and
    // clears the frozen ones)
    bool history = false;
    int64_t frozen = 0;  // frozen vertices after the last step
    // per-slot device arrays (capacity max_requests + dead slots: sized by max_slots)
    int32_t max_slots = 0;
    int32_t* vgraph = nullptr;
    int64_t* voff = nullptr;
    uint32_t* bases = nullptr;
    // what the host says about every slot at a step, in one copy: where its level
    // goes, its count before, then a byte each for active, level 0 and the stop
    // mode (kb::GraphStop)
    char* slot_up = nullptr;
    std::vector<char> slot_up_h;
    std::vector<uint32_t> gbase_host;
    // staging for admission (raw graph, processed CSR for IN / BOTH), and the
    // streams of the copies in and out: they overlap the rounds
    Stage stage[2];
    cudaStream_t up = nullptr, down = nullptr;
    // Requests placed straight from pinned host arrays in this step and not yet
    // known to be well formed: tickets in the order of their slots, which are the
    // last ones, and a device word each (kb::launch_place_checked)
    std::vector<int64_t> unchecked;
    int32_t* verdict = nullptr;           // [max_requests]
    int32_t* verdict_h = nullptr;         // pinned
    bool host_access = false;             // kernels can read all host memory
    std::vector<Draining> draining;
    cudaEvent_t drained = nullptr;  // after the last copy out of a store in `draining`
    // round state
    Prepared R;
    bool dirty = true;

    // stats
    double t_first = -1;
    int64_t submitted = 0, completed = 0, failed = 0, steps = 0, compactions = 0;
    double edge_rounds = 0;
    std::vector<double> latencies_ms;
};

namespace {

kb_status sfail(kb_server* sv, kb_status st, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    sv->last_error = buf;
    return st;
}

#define SV_CUDA(sv, call)                                                                            \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ != cudaSuccess) return sfail((sv), KB_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

#define SV_TRY(sv, expr)                                                     \
    do {                                                                     \
        kb_status s_ = (expr);                                               \
        if (s_ != KB_OK) {                                                   \
            if ((sv)->last_error.empty()) (sv)->last_error = (sv)->ctx->last_error; \
            return s_;                                                       \
        }                                                                    \
    } while (0)

// Whether the device reads `count` elements at x in place: aligned (a kernel's
// loads are, a copy takes any address), pinned at both ends, on a device that can
// read what may lie between them in any case.
template <class T>
bool device_reads(const T* x, int64_t count) {
    if (!x || !count) return true;
    if (reinterpret_cast<uintptr_t>(x) % sizeof(T)) return false;
    const size_t bytes = sizeof(T) * (size_t)count;
    for (const void* q : {(const void*)x, (const void*)((const char*)x + bytes - 1)}) {
        cudaPointerAttributes a{};
        if (cudaPointerGetAttributes(&a, q) != cudaSuccess || a.type != cudaMemoryTypeHost || a.devicePointer != q) {
            cudaGetLastError();
            return false;
        }
    }
    return true;
}

// Out-edge requests in pinned memory are read in place (launch_place_checked):
// their verdicts come back for all of them at once.
bool read_in_place(const kb_server* sv, const ServeRequest& r) {
    return sv->host_access && r.n > 0 && !needs_in_csr(r.opt.direction) &&
           device_reads(r.row, r.n + 1) && device_reads(r.col, r.m) && device_reads(r.lab, r.m) && device_reads(r.vlab, r.n);
}

// A request by its ticket, for the stepping thread, which does not hold sv->mu:
// other threads submit and fetch meanwhile.  (A request stays where it is while
// others come and go, and is only fetched once the step is through with it.)
ServeRequest& request(kb_server* sv, int64_t ticket) {
    std::lock_guard<std::mutex> lk(sv->mu);
    return sv->reqs.find(ticket)->second;
}

// Append a slot for r's graph, which is placed at the arena's tail.
void push_slot(kb_server* sv, ServeRequest& r) {
    Slot sl;
    sl.ticket = r.ticket;
    sl.vbase = sv->n_used;
    sl.n = r.n;
    sl.ebase = sv->m_used;
    sl.m = r.m_proc;
    r.slot = (int)sv->slots.size();
    sv->slots.push_back(sl);
    sv->n_used += r.n;
    sv->m_used += r.m_proc;
}

// Request r is in the arena and runs from the next round on (sv->mu held).
void start_request(ServeRequest& r) {
    r.state = 1;
    r.round = 0;
    r.rows_queued = 0;
    cudaPointerAttributes attr{};
    r.early_rows = sizeof(int32_t) * (size_t)r.n >= kEarlyRowBytes && r.out &&
                   cudaPointerGetAttributes(&attr, r.out) == cudaSuccess && attr.type == cudaMemoryTypeHost;
    cudaGetLastError();
    r.counts.assign((size_t)r.k + 1, 0);
    r.row = nullptr;  // the caller's graph arrays are no longer read
    r.col = r.lab = r.vlab = nullptr;
}

// Request r is malformed (sv->mu held).
void reject_request(kb_server* sv, ServeRequest& r) {
    sv->level_pool[r.level_bytes].push_back(r.d_levels);
    sv->level_bytes_in_use -= r.level_bytes;
    r.d_levels = nullptr;
    r.state = 3;
    r.error = "row_offsets not monotone from 0 to m, or a neighbour id out of [0, n)";
    r.row = nullptr;
    ++sv->failed;
}

// Settle the unchecked requests.  A malformed one leaves the arena, and with it
// those behind it, which wait again.
kb_status check_placed(kb_server* sv, bool* changed) {
    const size_t count = sv->unchecked.size();
    if (!count) return KB_OK;
    cudaStream_t s = sv->ctx->stream;
    SV_CUDA(sv, cudaMemcpyAsync(sv->verdict_h, sv->verdict, sizeof(int32_t) * count, cudaMemcpyDeviceToHost, s));
    SV_CUDA(sv, cudaStreamSynchronize(s));
    std::lock_guard<std::mutex> lk(sv->mu);
    size_t good = 0;
    while (good < count && !sv->verdict_h[good]) ++good;
    for (size_t i = 0; i < good; ++i) start_request(sv->reqs[sv->unchecked[i]]);
    if (good) *changed = true;
    if (good < count) {
        const size_t slot = sv->slots.size() - (count - good);
        sv->n_used = sv->slots[slot].vbase;
        sv->m_used = sv->slots[slot].ebase;
        sv->slots.resize(slot);
    }
    for (size_t i = count; i-- > good;) {
        ServeRequest& r = sv->reqs[sv->unchecked[i]];
        r.slot = -1;
        if (sv->verdict_h[i]) {
            reject_request(sv, r);
        } else {
            sv->level_pool[r.level_bytes].push_back(r.d_levels);
            sv->level_bytes_in_use -= r.level_bytes;
            r.d_levels = nullptr;
            sv->waiting.push_front(r.ticket);
        }
    }
    sv->unchecked.clear();
    return KB_OK;
}

// Queue the copies of a waiting request's arrays into S.
kb_status stage_request(kb_server* sv, const ServeRequest& r, Stage& S) {
    const int64_t n = r.n, m = r.m;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += align_up(b); return o; };
    S.ticket = 0;
    S.o_row = take(sizeof(int64_t) * (size_t)(n + 1));
    S.o_col = take(sizeof(int32_t) * (size_t)m);
    S.o_lab = take(sizeof(int32_t) * (size_t)m);
    S.o_vlab = take(sizeof(int32_t) * (size_t)n);
    Plan P;
    P.n = n;
    P.m = m;
    P.dir = r.opt.direction;
    P.m_proc = r.m_proc;
    P.labels = r.lab != nullptr;
    layout_csr(P);
    S.o_csr = take(P.csr_bytes);
    if (off > S.bytes) {
        if (S.buf) cudaFree(S.buf);
        S.buf = nullptr;
        S.bytes = 0;
        if (cudaMalloc(&S.buf, off) != cudaSuccess) {
            cudaGetLastError();
            return sfail(sv, KB_ERR_OOM, "cannot allocate %zu bytes of staging", off);
        }
        S.bytes = off;
    }
    char* b = reinterpret_cast<char*>(S.buf);
    SV_CUDA(sv, cudaStreamWaitEvent(sv->up, S.free, 0));
    SV_CUDA(sv, cudaMemcpyAsync(b + S.o_row, r.row, sizeof(int64_t) * (size_t)(n + 1), cudaMemcpyHostToDevice, sv->up));
    if (m)
        SV_CUDA(sv, cudaMemcpyAsync(b + S.o_col, r.col, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, sv->up));
    if (m && P.labels)
        SV_CUDA(sv, cudaMemcpyAsync(b + S.o_lab, r.lab, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, sv->up));
    if (r.vlab)
        SV_CUDA(sv, cudaMemcpyAsync(b + S.o_vlab, r.vlab, sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, sv->up));
    SV_CUDA(sv, cudaEventRecord(S.full, sv->up));
    S.ticket = r.ticket;
    return KB_OK;
}

// Copy request r's graph into the arena at the tail, as a new slot.  next: the
// request that is likely to follow (or null), whose arrays are copied meanwhile.
kb_status place_request(kb_server* sv, ServeRequest& r, const ServeRequest* next, bool* rejected) {
    *rejected = false;
    kb_context* ctx = sv->ctx;
    cudaStream_t s = ctx->stream;
    Arena& A = sv->arena[sv->cur];
    const int64_t n = r.n, m = r.m, mp = r.m_proc;
    const int at = sv->stage[1].ticket == r.ticket ? 1 : 0;
    Stage& S = sv->stage[at];
    if (S.ticket != r.ticket) SV_TRY(sv, stage_request(sv, r, S));
    S.ticket = 0;
    Plan P;
    P.n = n;
    P.m = m;
    P.dir = r.opt.direction;
    P.m_proc = mp;
    P.labels = r.lab != nullptr;
    layout_csr(P);
    const size_t o_row = S.o_row, o_col = S.o_col, o_lab = S.o_lab, o_vlab = S.o_vlab, o_csr = S.o_csr;
    char* b = reinterpret_cast<char*>(S.buf);
    SV_CUDA(sv, cudaStreamWaitEvent(s, S.full, 0));
    // the arena is shared: a malformed CSR is checked on the device before it
    // is placed, and the request fails alone
    SV_CUDA(sv, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
    kb::launch_validate(n, m, reinterpret_cast<const int64_t*>(b + o_row), reinterpret_cast<const int32_t*>(b + o_col),
                        ctx->d_ctr, s);
    SV_CUDA(sv, cudaGetLastError());
    SV_CUDA(sv, cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
    if (next && stage_request(sv, *next, sv->stage[1 - at]) != KB_OK) {
        sv->last_error.clear();  // staged when its turn comes
        cudaGetLastError();
    }
    SV_CUDA(sv, cudaStreamSynchronize(s));
    if (ctx->h_ctr->err & kb::kErrInvalid) {
        *rejected = true;
        return KB_OK;
    }
    kb::PlaceArgs a{};
    a.srow = reinterpret_cast<const int64_t*>(b + o_row);
    a.scol = reinterpret_cast<const int32_t*>(b + o_col);
    a.slab = P.labels ? reinterpret_cast<const int32_t*>(b + o_lab) : nullptr;
    if (needs_in_csr(P.dir)) {
        kb_graph g{n, m, a.srow, a.scol, a.slab, nullptr};
        char* csr = b + o_csr;
        SV_TRY(sv, build_processed_csr(ctx, &g, P, csr));
        a.srow = reinterpret_cast<const int64_t*>(csr + P.o_rowp);
        a.scol = reinterpret_cast<const int32_t*>(csr + P.o_colp);
        a.slab = P.labels ? reinterpret_cast<const int32_t*>(csr + P.o_labp) : nullptr;
    }
    a.svlab = r.vlab ? reinterpret_cast<const int32_t*>(b + o_vlab) : nullptr;
    a.drow = A.row;
    a.dcol = A.col;
    a.dlab = A.lab;
    a.dvlab = A.vlab;
    a.n = n;
    a.m = mp;
    a.src_vbase = 0;
    a.src_ebase = 0;
    a.dst_vbase = sv->n_used;
    a.dst_ebase = sv->m_used;
    kb::launch_place(a, s);
    SV_CUDA(sv, cudaGetLastError());
    SV_CUDA(sv, cudaEventRecord(S.free, s));
    push_slot(sv, r);
    return KB_OK;
}

// Pack the live slots into the other arena buffer.
kb_status compact(kb_server* sv) {
    kb_context* ctx = sv->ctx;
    cudaStream_t s = ctx->stream;
    Arena& S = sv->arena[sv->cur];
    Arena& D = sv->arena[1 - sv->cur];
    std::vector<Slot> live;
    int64_t nv = 0, ne = 0;
    SV_CUDA(sv, cudaMemsetAsync(D.row, 0, sizeof(int64_t), s));
    for (size_t j = 0; j < sv->slots.size(); ++j) {
        const Slot& o = sv->slots[j];
        if (o.ticket < 0) continue;
        kb::PlaceArgs a{};
        a.srow = S.row;
        a.scol = S.col;
        a.slab = S.lab;
        a.svlab = S.vlab;
        a.sname = S.name;
        a.drow = D.row;
        a.dcol = D.col;
        a.dlab = D.lab;
        a.dvlab = D.vlab;
        a.dname = D.name;
        a.n = o.n;
        a.m = o.m;
        a.src_vbase = o.vbase;
        a.src_ebase = o.ebase;
        a.dst_vbase = nv;
        a.dst_ebase = ne;
        kb::launch_place(a, s);
        Slot ns = o;
        ns.vbase = nv;
        ns.ebase = ne;
        request(sv, o.ticket).slot = (int)live.size();
        live.push_back(ns);
        nv += o.n;
        ne += o.m;
    }
    SV_CUDA(sv, cudaGetLastError());
    sv->slots = live;
    sv->n_used = nv;
    sv->m_used = ne;
    sv->cur = 1 - sv->cur;
    sv->dirty = true;
    sv->vertices_moved = true;
    ++sv->compactions;
    return KB_OK;
}

size_t free_device_bytes() {
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return fr;
}

// Size class of a level store: the next power of two of at least 256 bytes.
size_t level_store_bytes(size_t bytes) {
    size_t b = 256;
    while (b < bytes) b <<= 1;
    return b;
}

// A finished request whose levels have reached the host (sv->mu held).
void publish(kb_server* sv, ServeRequest& r) {
    r.draining = false;
    r.t_done = now_s();
    r.state = 2;
    ++sv->completed;
    sv->latencies_ms.push_back(1000.0 * (r.t_done - r.t_submit));
    sv->edge_rounds += (double)r.m_proc * (double)r.levels_computed;
}

// Return the level stores whose copies are done; wait: all of them.
kb_status release_drained(kb_server* sv, bool wait) {
    if (sv->draining.empty()) return KB_OK;
    if (wait) {
        SV_CUDA(sv, cudaEventSynchronize(sv->drained));
    } else {
        const cudaError_t e = cudaEventQuery(sv->drained);
        if (e == cudaErrorNotReady) return KB_OK;
        SV_CUDA(sv, e);
    }
    std::lock_guard<std::mutex> lk(sv->mu);
    for (const Draining& d : sv->draining) {
        sv->level_pool[d.level_bytes].push_back(d.d_levels);
        sv->level_bytes_in_use -= d.level_bytes;
        auto it = sv->reqs.find(d.ticket);
        if (it != sv->reqs.end() && it->second.draining) publish(sv, it->second);
    }
    sv->draining.clear();
    return KB_OK;
}

// Admit waiting requests in arrival order while they fit.
kb_status admit(kb_server* sv, bool* changed) {
    while (true) {
        int64_t t = 0;
        const ServeRequest* next = nullptr;
        {
            std::lock_guard<std::mutex> lk(sv->mu);
            if (!sv->waiting.empty()) t = sv->waiting.front();
            if (sv->waiting.size() > 1) next = &sv->reqs[sv->waiting[1]];
        }
        if (!t) {
            if (sv->unchecked.empty()) break;
            SV_TRY(sv, check_placed(sv, changed));  // may leave requests waiting again
            continue;
        }
        SV_TRY(sv, release_drained(sv, true));  // their stores may be needed
        ServeRequest& r = request(sv, t);
        int live = 0;
        for (const Slot& sl : sv->slots) live += sl.ticket >= 0;
        const size_t lb = level_store_bytes(sizeof(int32_t) * (size_t)r.n * (size_t)(r.k + 1));
        std::vector<int32_t*>& pooled = sv->level_pool[lb];
        const size_t budget = sv->cfg.memory_budget;
        bool fits = live < sv->cfg.max_requests;
        if (fits && budget) {
            fits = sv->level_bytes_in_use + lb <= budget;
        } else if (fits && pooled.empty()) {
            fits = free_device_bytes() >= lb + ((size_t)1 << 30);
        }
        bool pack = false;
        if (fits && !(sv->n_used + r.n <= sv->cfg.max_vertices && sv->m_used + r.m_proc <= sv->cfg.max_edges &&
                      (int)sv->slots.size() < sv->max_slots)) {
            int64_t ln = 0, lm = 0;
            for (const Slot& sl : sv->slots)
                if (sl.ticket >= 0) {
                    ln += sl.n;
                    lm += sl.m;
                }
            fits = ln + r.n <= sv->cfg.max_vertices && lm + r.m_proc <= sv->cfg.max_edges;
            pack = fits;
        }
        const bool direct = fits && !pack && read_in_place(sv, r);
        if (!direct && !sv->unchecked.empty()) {
            // (a malformed one among them may make room)
            SV_TRY(sv, check_placed(sv, changed));
            continue;
        }
        if (!fits) break;
        if (pack) SV_TRY(sv, compact(sv));
        if (!pooled.empty()) {
            r.d_levels = pooled.back();
            pooled.pop_back();
        } else if (cudaMalloc(&r.d_levels, lb) != cudaSuccess) {
            cudaGetLastError();
            r.d_levels = nullptr;
            if (sv->unchecked.empty()) break;
            SV_TRY(sv, check_placed(sv, changed));
            continue;
        }
        r.level_bytes = lb;
        sv->level_bytes_in_use += lb;
        if (direct) {
            cudaStream_t s = sv->ctx->stream;
            if (sv->unchecked.empty())
                SV_CUDA(sv, cudaMemsetAsync(sv->verdict, 0, sizeof(int32_t) * (size_t)sv->cfg.max_requests, s));
            Arena& A = sv->arena[sv->cur];
            kb::PlaceArgs a{};
            a.srow = r.row;
            a.scol = r.col;
            a.slab = r.lab;
            a.svlab = r.vlab;
            a.drow = A.row;
            a.dcol = A.col;
            a.dlab = A.lab;
            a.dvlab = A.vlab;
            a.n = r.n;
            a.m = r.m;
            a.dst_vbase = sv->n_used;
            a.dst_ebase = sv->m_used;
            kb::launch_place_checked(a, sv->verdict + sv->unchecked.size(), s);
            SV_CUDA(sv, cudaGetLastError());
            push_slot(sv, r);
            sv->unchecked.push_back(t);
            std::lock_guard<std::mutex> lk(sv->mu);
            sv->waiting.pop_front();
            continue;
        }
        // the next one's copies start already if it fits behind this one
        if (next && (live + 2 > sv->cfg.max_requests || (int)sv->slots.size() + 2 > sv->max_slots ||
                     sv->n_used + r.n + next->n > sv->cfg.max_vertices ||
                     sv->m_used + r.m_proc + next->m_proc > sv->cfg.max_edges || read_in_place(sv, *next)))
            next = nullptr;
        bool rejected = false;
        SV_TRY(sv, place_request(sv, r, next, &rejected));
        std::lock_guard<std::mutex> lk(sv->mu);
        sv->waiting.pop_front();
        if (rejected) {
            reject_request(sv, r);
        } else {
            start_request(r);
            *changed = true;
        }
    }
    // one that did not follow after all is copied again when it is admitted
    for (Stage& S : sv->stage)
        if (S.ticket) {
            SV_CUDA(sv, cudaEventSynchronize(S.full));
            S.ticket = 0;
        }
    return KB_OK;
}

// Queue the copies of request r's rows up to `last`, which is final, to its host
// levels (the caller's buffer given at submission, else a buffer of its own).
kb_status copy_rows_out(kb_server* sv, ServeRequest& r, int last) {
    const size_t n = (size_t)r.n, q = (size_t)r.rows_queued;
    if (!r.out && !r.levels) {
        r.levels.reset(new (std::nothrow) int32_t[std::max<size_t>(n * (size_t)(r.k + 1), 1)]);
        if (!r.levels) return sfail(sv, KB_ERR_OOM, "cannot allocate host memory for the levels");
    }
    int32_t* dst = r.out ? r.out : r.levels.get();
    if (n && r.rows_queued <= last)
        SV_CUDA(sv, cudaMemcpyAsync(dst + q * n, r.d_levels + q * n, sizeof(int32_t) * n * ((size_t)last + 1 - q),
                                    cudaMemcpyDeviceToHost, sv->down));
    r.rows_queued = last + 1;
    return KB_OK;
}

// Finish request r after its last round: its slot is free, and its levels and
// level store follow when the copies are done (publish, release_drained).  Rows
// after the last refined level repeat it.
kb_status retire(kb_server* sv, ServeRequest& r, int last) {
    const size_t n = (size_t)r.n;
    SV_TRY(sv, copy_rows_out(sv, r, last));
    int32_t* dst = r.out ? r.out : r.levels.get();
    for (int j = last + 1; n && j <= r.k; ++j)
        SV_CUDA(sv, cudaMemcpyAsync(dst + (size_t)j * n, r.d_levels + (size_t)last * n, sizeof(int32_t) * n,
                                    cudaMemcpyDeviceToHost, sv->down));
    SV_CUDA(sv, cudaEventRecord(sv->drained, sv->down));
    std::lock_guard<std::mutex> lk(sv->mu);
    for (int j = last + 1; j <= r.k; ++j) r.counts[(size_t)j] = r.counts[(size_t)last];
    r.levels_computed = last;
    r.draining = true;
    sv->draining.push_back({r.ticket, r.d_levels, r.level_bytes});
    r.d_levels = nullptr;
    sv->slots[(size_t)r.slot].ticket = -1;
    r.slot = -1;
    return KB_OK;
}

// The caller asks for a request: one that has finished waits for the copies of
// its levels (sv->mu held).
kb_status settle(kb_server* sv, ServeRequest& r) {
    if (!r.draining) return KB_OK;
    SV_CUDA(sv, cudaEventSynchronize(sv->drained));
    publish(sv, r);
    return KB_OK;
}

kb_status server_step(kb_server* sv, int32_t* running, int32_t* waiting_out) {
    kb_context* ctx = sv->ctx;
    cudaStream_t s = ctx->stream;
    SV_CUDA(sv, cudaSetDevice(ctx->device));
    bool changed = false;
    SV_TRY(sv, admit(sv, &changed));
    if (changed) sv->dirty = true;
    int live = 0;
    int64_t live_n = 0;
    for (const Slot& sl : sv->slots)
        if (sl.ticket >= 0) {
            ++live;
            live_n += sl.n;
        }
    // every round's kernels span the whole arena, retired ranges included:
    // pack the live requests once the dead ones dominate (cheap under light
    // load, when little is live)
    if (live > 0 && sv->n_used - live_n > 4 * live_n + ((int64_t)1 << 22)) SV_TRY(sv, compact(sv));
    if (live > 0) {
        const int G = (int)sv->slots.size();
        Arena& A = sv->arena[sv->cur];
        kb::RoundParams& p = sv->R.p;
        if (sv->dirty) {
            // re-plan the arena: medium / hub lists, block table, minima
            kb_graph view{sv->n_used, sv->m_used, A.row, A.col, A.lab, nullptr};
            kb_options o = kb_options_default();
            o.validate = 0;
            o.load_factor = sv->cfg.load_factor;
            o.hub_threshold = sv->cfg.hub_threshold;
            o.hash_mode = sv->cfg.hash_mode;
            sv->R.ext_table = sv->table;
            sv->R.ext_cap = sv->table_cap;
            sv->R.emin_bytes = sizeof(uint64_t) * (size_t)sv->cfg.max_vertices;
            sv->R.ext_emin = sv->emin;
            sv->R.ext_frozen = sv->frz[0];
            sv->R.ext_frozen_min = sv->frz[1];
            sv->R.ext_shared = sv->frz[2];
            sv->R.ext_moved = sv->frz[3];
            sv->R.ext_mark = sv->frz[4];
            sv->R.ext_minof = A.name;
            const size_t bw = sizeof(uint32_t) * (size_t)((sv->n_used >> 5) + 1);
            if (sv->vertices_moved) {
                // compacted: vertex ids moved, nothing carries over
                for (int f = 0; f < 3; ++f) SV_CUDA(sv, cudaMemsetAsync(sv->frz[f], 0, bw, s));
                sv->history = false;
                sv->vertices_moved = false;
            } else {
                // admitted at the tail: the new vertices start unfrozen, the
                // others keep their blocks' state; the bits past the last
                // vertex are cleared too (rank scans count whole words)
                const int64_t word_end = ((sv->n_used >> 5) + 1) * 32;
                for (int f = 0; f < 3; ++f) kb::launch_clear_bits(sv->frz[f], sv->planned_n, word_end, s);
            }
            SV_TRY(sv, prepare(ctx, &view, &o, sv->R, -1, true));
            for (bool& on : sv->R.class_on) on = true;  // new vertices refine
            sv->planned_n = sv->n_used;
            std::vector<int64_t> voff((size_t)G + 1);
            for (int j = 0; j < G; ++j) voff[(size_t)j] = sv->slots[(size_t)j].vbase;
            voff[(size_t)G] = sv->n_used;
            SV_CUDA(sv, cudaMemcpyAsync(sv->voff, voff.data(), sizeof(int64_t) * (size_t)(G + 1), cudaMemcpyHostToDevice, s));
            kb::launch_vertex_graph(sv->voff, G, sv->n_used, sv->vgraph, s);
            sv->dirty = false;
        }
        // per-slot words for this step
        const size_t o_cnt = sizeof(int32_t*) * (size_t)G, o_act = o_cnt + sizeof(int64_t) * (size_t)G,
                     o_mode = o_act + (size_t)G, o_stop = o_mode + (size_t)G;
        std::vector<char>& up = sv->slot_up_h;
        up.assign(o_stop + (size_t)G, 0);
        int32_t** lev = reinterpret_cast<int32_t**>(up.data());
        int64_t* before = reinterpret_cast<int64_t*>(up.data() + o_cnt);
        for (int j = 0; j < G; ++j) {
            const Slot& sl = sv->slots[(size_t)j];
            if (sl.ticket < 0) continue;
            ServeRequest& r = request(sv, sl.ticket);
            lev[j] = r.d_levels + (size_t)r.round * (size_t)r.n;
            before[j] = r.round > 0 ? r.counts[(size_t)r.round - 1] : 0;
            up[o_act + (size_t)j] = 1;
            up[o_mode + (size_t)j] = r.round == 0 ? 1 : 0;
            up[o_stop + (size_t)j] = r.round >= r.k ? 1 : (r.round > 0 && r.opt.early_stop ? 2 : 0);
        }
        SV_CUDA(sv, cudaMemcpyAsync(sv->slot_up, up.data(), up.size(), cudaMemcpyHostToDevice, s));
        uint8_t* gactive = reinterpret_cast<uint8_t*>(sv->slot_up + o_act);
        const uint8_t* gmode = reinterpret_cast<const uint8_t*>(sv->slot_up + o_mode);
        // one round for everything in flight
        SV_TRY(sv, next_epoch(ctx, sv->R, s));
        SV_TRY(sv, next_empty_round(ctx, sv->R, s));
        p.vgraph = sv->vgraph;
        p.lgraph = sv->vgraph;
        p.voff = sv->voff;
        p.n_graphs = G;
        p.gmode = gmode;
        p.gout = reinterpret_cast<int32_t* const*>(sv->slot_up);
        p.vlab = A.vlab;
        p.prev = reinterpret_cast<const int32_t*>(A.name);
        p.gbase_cur = sv->bases;
        sv->R.gactive = gactive;
        // frozen blocks, as in a single-graph call (blocks never span graphs)
        p.frozen = sv->R.frozen;
        p.frozen_min = sv->R.frozen_min;
        p.moved = sv->history ? sv->R.moved : nullptr;
        sv->R.compact = sv->history && sv->frozen * 4 > sv->n_used;  // (retired graphs' vertices are frozen)
        SV_TRY(sv, launch_round_body(ctx, sv->R, s, nullptr));
        kb::GraphStop stop;
        stop.active = gactive;
        stop.mode = reinterpret_cast<const uint8_t*>(sv->slot_up + o_stop);
        stop.prev_count = reinterpret_cast<const int64_t*>(sv->slot_up + o_cnt);
        kb::launch_renumber(p, sv->R.prefix, sv->R.scan_tmp, nullptr, p.moved ? sv->R.mark : nullptr, false, s, stop);
        if (p.moved)
            kb::launch_dirty_blocks(p, sv->R.edgeless, sv->R.moved, kb::kMaxHubThreshold, sv->R.mark, gactive, false, s);
        kb::FreezePass f = freeze_pass(ctx, sv->R);
        f.mark = p.moved ? sv->R.mark : nullptr;
        f.gmode = gmode;
        kb::launch_freeze_clean(f, s);
        sv->history = true;
        SV_CUDA(sv, cudaGetLastError());
        sv->gbase_host.assign((size_t)G + 1, 0);
        SV_CUDA(sv, cudaMemcpyAsync(sv->gbase_host.data(), p.gbase_cur, sizeof(uint32_t) * (size_t)(G + 1),
                                    cudaMemcpyDeviceToHost, s));
        SV_CUDA(sv, cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
        SV_CUDA(sv, cudaStreamSynchronize(s));
        if (ctx->h_ctr->err) {
            SV_TRY(sv, device_error(ctx));
        }
        for (int c = 0; c < 3; ++c) sv->R.class_on[c] = ctx->h_ctr->class_on[c] > 0;
        sv->frozen = ctx->h_ctr->frozen;
        // bookkeeping and retirement.  The copies out run on a stream of their
        // own while the other requests refine: those of finished requests first,
        // then the new rows of large ones.
        SV_TRY(sv, release_drained(sv, false));
        for (int j = 0; j < G; ++j) {
            const Slot sl = sv->slots[(size_t)j];
            if (sl.ticket < 0) continue;
            ServeRequest& r = request(sv, sl.ticket);
            const int64_t cnt = (int64_t)(sv->gbase_host[(size_t)j + 1] - sv->gbase_host[(size_t)j]);
            r.counts[(size_t)r.round] = cnt;
            const int done_round = r.round;
            bool done = done_round >= r.k;
            if (done_round > 0 && r.opt.early_stop && cnt == r.counts[(size_t)done_round - 1]) done = true;
            ++r.round;
            if (done) SV_TRY(sv, retire(sv, r, done_round));
        }
        for (int j = 0; j < G; ++j) {
            if (sv->slots[(size_t)j].ticket < 0) continue;
            ServeRequest& r = request(sv, sv->slots[(size_t)j].ticket);
            if (r.early_rows) SV_TRY(sv, copy_rows_out(sv, r, r.round - 1));
        }
        ++sv->steps;
    }
    int run = 0;
    for (const Slot& sl : sv->slots) run += sl.ticket >= 0;
    if (run == 0) SV_TRY(sv, release_drained(sv, true));
    std::lock_guard<std::mutex> lk(sv->mu);
    if (running) *running = run;
    if (waiting_out) *waiting_out = (int32_t)sv->waiting.size();
    return KB_OK;
}
}  // namespace

extern "C" {

kb_options kb_options_default(void) {
    kb_options o;
    std::memset(&o, 0, sizeof(o));
    o.direction = KB_DIR_OUT;
    o.use_vertex_labels = 1;
    o.use_edge_labels = 1;
    o.early_stop = 1;
    o.validate = 1;
    return o;
}

kb_options kb_options_schaetzle(void) {
    kb_options o = kb_options_default();
    o.direction = KB_DIR_OUT;
    o.use_vertex_labels = 0;
    o.use_edge_labels = 1;
    return o;
}

kb_options kb_options_kaushik(void) {
    kb_options o = kb_options_default();
    o.direction = KB_DIR_IN;
    o.use_vertex_labels = 1;
    o.use_edge_labels = 0;
    return o;
}

const char* kb_status_string(kb_status st) {
    switch (st) {
        case KB_OK: return "ok";
        case KB_ERR_INVALID_ARG: return "invalid argument";
        case KB_ERR_OOM: return "out of device memory";
        case KB_ERR_TABLE_FULL: return "block table full";
        case KB_ERR_TIMEOUT: return "device wait timed out";
        case KB_ERR_CUDA: return "CUDA error";
        case KB_ERR_DEVICE_CHECK: return "device consistency check failed";
        case KB_ERR_NOT_FOUND: return "not found";
    }
    return "unknown status";
}

kb_status kb_create(kb_context** out, int device, void* stream) {
    if (!out) return KB_ERR_INVALID_ARG;
    *out = nullptr;
    kb_context* ctx = new (std::nothrow) kb_context();
    if (!ctx) return KB_ERR_OOM;
    ctx->device = device;
    ctx->stream = reinterpret_cast<cudaStream_t>(stream);
    if (cudaSetDevice(device) != cudaSuccess || cudaMalloc(&ctx->d_ctr, sizeof(Counters)) != cudaSuccess ||
        cudaMalloc(&ctx->d_dense, (sizeof(uint32_t) + sizeof(uint2)) * kb::kDenseLabels) != cudaSuccess ||
        cudaMallocHost(&ctx->h_hubs, (sizeof(int32_t) + sizeof(int64_t)) * kEagerHubs) != cudaSuccess ||
        cudaMallocHost(&ctx->h_ctr, sizeof(Counters) * (1 + kCounterSlots)) != cudaSuccess) {
        cudaGetLastError();
        kb_destroy(ctx);
        return KB_ERR_CUDA;
    }
    for (auto& e : ctx->ev) cudaEventCreate(&e);
    for (auto& e : ctx->slot_ev) cudaEventCreateWithFlags(&e, cudaEventDisableTiming);
    kb::set_medium_kernel_attributes();
    ctx->fused_ctas = ctx->fused_most = kb::fused_max_ctas();
    cudaGetLastError();
    *out = ctx;
    return KB_OK;
}

kb_status kb_destroy(kb_context* ctx) {
    if (!ctx) return KB_OK;
    cudaSetDevice(ctx->device);
    if (ctx->stream) cudaStreamSynchronize(ctx->stream); else cudaDeviceSynchronize();
    cudaFree(ctx->d_ctr);
    cudaFree(ctx->d_dense);
    cudaFreeHost(ctx->h_hubs);
    cudaFreeHost(ctx->h_ctr);
    cudaFree(ctx->own_ws);
    cudaFree(ctx->class_tmp);
    cudaFree(ctx->plan_tmp);
    cudaFree(ctx->stage);
    cudaFree(ctx->tab);
    cudaFree(ctx->emin);
    cudaFree(ctx->batch_ws);
    cudaFree(ctx->tune_buf);
    cudaFree(ctx->fix_buf);
    cudaFree(ctx->sum_buf);
    cudaFree(ctx->upd_buf);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    if (ctx->row_ev) cudaEventDestroy(ctx->row_ev);

    for (auto& e : ctx->ev)
        if (e) cudaEventDestroy(e);
    for (auto& e : ctx->slot_ev)
        if (e) cudaEventDestroy(e);
    delete ctx;
    return KB_OK;
}

const char* kb_last_error(const kb_context* ctx) { return ctx ? ctx->last_error.c_str() : "no context"; }

kb_status kb_workspace_size(kb_context* ctx, const kb_graph* g, const kb_options* opt, int k, size_t* bytes) {
    if (!ctx || !bytes) return KB_ERR_INVALID_ARG;
    KB_TRY(check_graph(ctx, g, opt, k));
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    if (g->n == 0) {
        *bytes = 0;
        return KB_OK;
    }
    Plan P;
    char* unused = nullptr;
    KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), ctx->stream));
    KB_TRY(make_plan(ctx, g, opt, P, &unused, true, k));
    *bytes = P.total;
    return KB_OK;
}

kb_status kb_set_workspace(kb_context* ctx, void* ptr, size_t bytes) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    ctx->user_ws = ptr;
    ctx->user_ws_bytes = ptr ? bytes : 0;
    return KB_OK;
}

kb_status kb_set_round_kernel(kb_context* ctx, int32_t max_ctas, int32_t max_polls) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (max_ctas < -1 || max_polls < 0) return fail(ctx, KB_ERR_INVALID_ARG, "bad limits of the round kernel");
    ctx->fused_ctas = max_ctas < 0 || ctx->fused_most == 0 ? ctx->fused_most : max_ctas;
    ctx->fused_polls = max_polls > 0 ? (uint32_t)max_polls : (uint32_t)kb::kFusedPolls;
    return KB_OK;
}

kb_status kb_get_round_kernel(const kb_context* ctx, int64_t* launches, int64_t* refused, int64_t* gave_up) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (launches) *launches = ctx->fused_launches;
    if (refused) *refused = ctx->fused_refused;
    if (gave_up) *gave_up = ctx->fused_gave_up;
    return KB_OK;
}

kb_status kb_refine(kb_context* ctx, const kb_graph* g, const kb_options* opt, int k, int32_t* levels,
                    int64_t* counts, int* levels_computed) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    return refine_impl(ctx, g, opt, nullptr, 0, k, levels, counts, levels_computed);
}

kb_status kb_refine_from(kb_context* ctx, const kb_graph* g, const kb_options* opt, const int32_t* start,
                         int i_start, int k, int32_t* levels, int64_t* counts, int* levels_computed) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (!start && g && g->n > 0) return fail(ctx, KB_ERR_INVALID_ARG, "start is NULL");
    return refine_impl(ctx, g, opt, start, i_start, k, levels, counts, levels_computed);
}

kb_status kb_graph_prepare(kb_context* ctx, const kb_graph* g, const kb_options* opt, kb_prepared** out) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (!out) return fail(ctx, KB_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    KB_TRY(check_graph(ctx, g, opt, 0));
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    const auto t0 = std::chrono::steady_clock::now();
    cudaStream_t s = ctx->stream;
    std::unique_ptr<kb_prepared> pg(new kb_prepared);
    pg->device = ctx->device;
    pg->g = *g;
    pg->dir = opt->direction;
    pg->edge_labels = opt->use_edge_labels ? 1 : 0;
    const int64_t n = g->n;
    KB_CUDA(ctx, cudaMemsetAsync(ctx->d_ctr, 0, sizeof(Counters), s));
    if (n > 0) KB_TRY(check_input(ctx, g, opt));
    Plan& P = pg->P;
    P.graph_ext = true;
    Plan probe;
    probe.n = n;
    probe.m = g->m;
    probe.dir = opt->direction;
    probe.m_proc = probe.dir == KB_DIR_BOTH ? 2 * g->m : g->m;
    probe.labels = opt->use_edge_labels && g->edge_labels != nullptr;
    layout_csr(probe);
    auto alloc = [&](char** ptr, size_t bytes) -> kb_status {
        if (cudaMalloc(reinterpret_cast<void**>(ptr), std::max<size_t>(bytes, 256)) != cudaSuccess) {
            cudaGetLastError();
            *ptr = nullptr;
            return fail(ctx, KB_ERR_OOM, "cannot allocate %zu bytes of device memory", bytes);
        }
        return KB_OK;
    };
    if (probe.csr_bytes) KB_TRY(alloc(&pg->csr, probe.csr_bytes));
    char* base = pg->csr;
    if (n > 0) KB_TRY(make_plan(ctx, g, opt, P, &base, false, 1, false));
    KB_TRY(alloc(&pg->gbuf, P.graph_bytes));
    if (n > 0) {
        char* count_tmp = nullptr;
        if (P.reorder) KB_TRY(alloc(&count_tmp, sizeof(uint32_t) * (size_t)n));
        kb::RoundParams p{};
        p.n = n;
        const kb_status st = bind_graph_part(ctx, g, P, pg->csr, pg->gbuf, true,
                                             reinterpret_cast<uint32_t*>(count_tmp), p, s);
        const cudaError_t e = cudaStreamSynchronize(s);
        cudaFree(count_tmp);
        KB_TRY(st);
        if (e != cudaSuccess) return fail(ctx, KB_ERR_CUDA, "prepare: %s", cudaGetErrorString(e));
    }
    // the hub lists are on the device now
    std::vector<int32_t>().swap(P.hub_v);
    std::vector<int64_t>().swap(P.chunk_off);
    std::vector<int64_t>().swap(P.set_off);
    pg->build_ms = std::chrono::duration<float, std::milli>(std::chrono::steady_clock::now() - t0).count();
    *out = pg.release();
    return KB_OK;
}

kb_status kb_graph_release(kb_prepared* pg) {
    delete pg;
    return KB_OK;
}

kb_status kb_prepared_get_info(const kb_prepared* pg, kb_prepared_info* info) {
    if (!pg || !info) return KB_ERR_INVALID_ARG;
    std::memset(info, 0, sizeof(*info));
    info->device_bytes = (pg->csr ? pg->P.csr_bytes : 0) + pg->P.graph_bytes;
    info->n_hubs = (int64_t)pg->P.n_hubs;
    info->n_hub_chunks = pg->P.n_chunks;
    info->n_medium = pg->P.n_med;
    info->reorder = pg->P.reorder ? 1 : 0;
    info->hub_threshold = pg->P.thr;
    info->small_max_degree = pg->P.small_max;
    info->hub_chunk_edges = pg->P.hub_chunk;
    info->build_ms = pg->build_ms;
    return KB_OK;
}

kb_status kb_refine_prepared(kb_context* ctx, const kb_prepared* pg, const kb_options* opt, int k, int32_t* levels,
                             int64_t* counts, int* levels_computed) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (!pg || !opt) return fail(ctx, KB_ERR_INVALID_ARG, "prepared graph and options must not be NULL");
    if (pg->device != ctx->device)
        return fail(ctx, KB_ERR_INVALID_ARG, "the graph was prepared on device %d, the context is on %d", pg->device,
                    ctx->device);
    if (opt->direction != pg->dir || (opt->use_edge_labels ? 1 : 0) != pg->edge_labels)
        return fail(ctx, KB_ERR_INVALID_ARG, "direction and use_edge_labels must be those of kb_graph_prepare");
    return refine_impl(ctx, &pg->g, opt, nullptr, 0, k, levels, counts, levels_computed, pg);
}

kb_status kb_refine_update(kb_context* ctx, const kb_graph* g, const kb_options* opt, int k, const int32_t* changed,
                           int64_t n_changed, int32_t* levels, int64_t* counts, int* levels_computed, int64_t* work) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    return update_impl(ctx, g, opt, k, changed, n_changed, levels, counts, levels_computed, work);
}

kb_status kb_summary(kb_context* ctx, const kb_graph* g, int direction, int use_edge_labels,
                     const int32_t* src_level, const int32_t* dst_level, int32_t* out_src, int32_t* out_label,
                     int32_t* out_dst, int64_t capacity, int64_t* count) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    return summary_impl(ctx, g, direction, use_edge_labels, src_level, dst_level, out_src, out_label, out_dst,
                        capacity, count);
}

kb_status kb_refine_fixpoint(kb_context* ctx, const kb_graph* g, const kb_options* opt, const int32_t* initial,
                             int max_rounds, int32_t* final_level, int64_t* count, int* rounds, int* stable) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    return fixpoint_impl(ctx, g, opt, initial, max_rounds, final_level, count, rounds, stable);
}

kb_status kb_refine_host(kb_context* ctx, const kb_graph* g, const kb_options* opt, int k, int32_t* levels,
                         int64_t* counts, int* levels_computed) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    KB_TRY(check_graph(ctx, g, opt, k));
    if (!counts) return fail(ctx, KB_ERR_INVALID_ARG, "counts is NULL");
    if (g->n > 0 && !levels) return fail(ctx, KB_ERR_INVALID_ARG, "levels is NULL");
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    const int64_t n = g->n, m = g->m;
    const bool el = g->edge_labels && opt->use_edge_labels;
    const bool vl = g->vertex_labels && opt->use_vertex_labels;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off += align_up(b); return o; };
    const size_t o_row = take(sizeof(int64_t) * (size_t)(n + 1));
    const size_t o_col = take(sizeof(int32_t) * (size_t)m);
    const size_t o_el = take(el ? sizeof(int32_t) * (size_t)m : 0);
    const size_t o_vl = take(vl ? sizeof(int32_t) * (size_t)n : 0);
    const size_t o_lv = take(sizeof(int32_t) * (size_t)n * (size_t)(k + 1));
    KB_TRY(ensure_buffer(ctx, &ctx->stage, &ctx->stage_bytes, std::max<size_t>(off, 256)));
    char* b = reinterpret_cast<char*>(ctx->stage);
    cudaStream_t s = ctx->stream;
    if (n > 0) {
        KB_CUDA(ctx, cudaMemcpyAsync(b + o_row, g->row_offsets, sizeof(int64_t) * (size_t)(n + 1),
                                     cudaMemcpyHostToDevice, s));
    }
    if (m > 0) KB_CUDA(ctx, cudaMemcpyAsync(b + o_col, g->col_indices, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, s));
    if (el && m > 0) KB_CUDA(ctx, cudaMemcpyAsync(b + o_el, g->edge_labels, sizeof(int32_t) * (size_t)m, cudaMemcpyHostToDevice, s));
    if (vl && n > 0) KB_CUDA(ctx, cudaMemcpyAsync(b + o_vl, g->vertex_labels, sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, s));
    kb_graph dg = *g;
    dg.row_offsets = reinterpret_cast<const int64_t*>(b + o_row);
    dg.col_indices = reinterpret_cast<const int32_t*>(b + o_col);
    dg.edge_labels = el ? reinterpret_cast<const int32_t*>(b + o_el) : nullptr;
    dg.vertex_labels = vl ? reinterpret_cast<const int32_t*>(b + o_vl) : nullptr;
    int32_t* dlev = reinterpret_cast<int32_t*>(b + o_lv);
    // every level row goes back to the host as soon as it is final
    KB_TRY(refine_impl(ctx, &dg, opt, nullptr, 0, k, dlev, counts, levels_computed, nullptr, levels));
    KB_CUDA(ctx, cudaStreamSynchronize(s));
    return KB_OK;
}

kb_status kb_set_timing(kb_context* ctx, int enable) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (enable < 0 || enable > 2) return fail(ctx, KB_ERR_INVALID_ARG, "timing mode must be 0, 1 or 2");
    ctx->timing = enable != 0;
    ctx->work = enable == 2;
    return KB_OK;
}

kb_status kb_get_timing(const kb_context* ctx, float* round_ms, int max_rounds, int* n_rounds, float* kernel_ms,
                        int64_t* kernel_launches) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    const int nr = (int)ctx->round_ms.size();
    if (n_rounds) *n_rounds = nr;
    if (round_ms)
        for (int i = 0; i < nr && i < max_rounds; ++i) round_ms[i] = ctx->round_ms[(size_t)i];
    for (int f = 0; f < KB_KERNEL_COUNT; ++f) {
        if (kernel_ms) kernel_ms[f] = ctx->kernel_ms[f];
        if (kernel_launches) kernel_launches[f] = ctx->kernel_launches[f];
    }
    return KB_OK;
}

kb_status kb_get_round_work(const kb_context* ctx, int64_t* vertices, int64_t* edges, int max_rounds,
                            int* n_rounds) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    const int nr = (int)ctx->round_keyed.size();
    if (n_rounds) *n_rounds = nr;
    for (int i = 0; i < nr && i < max_rounds; ++i)
        for (int f = 0; f < 3; ++f) {
            if (vertices) vertices[3 * i + f] = ctx->round_keyed[(size_t)i][(size_t)f];
            if (edges) edges[3 * i + f] = ctx->round_keyed[(size_t)i][(size_t)f + 3];
        }
    return KB_OK;
}

kb_status kb_refine_batch(kb_context* ctx, const kb_graph* union_graph, const int64_t* graph_vertex_offsets,
                          int64_t G, const int32_t* k_per_graph, const kb_options* opt, int32_t* levels,
                          int64_t* counts, int32_t* levels_computed) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    return batch_impl(ctx, union_graph, graph_vertex_offsets, G, k_per_graph, opt, levels, counts, levels_computed);
}

kb_status kb_autotune(kb_context* ctx, const kb_graph* g, const int64_t* voff, int64_t G, const int32_t* k_per_graph,
                      const kb_options* opt, int rounds, kb_tuning* out) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    if (!g || !opt) return fail(ctx, KB_ERR_INVALID_ARG, "graph and options must not be NULL");
    const bool batch = voff != nullptr;
    if (batch && (G < 1 || G > (int64_t)1 << 30)) return fail(ctx, KB_ERR_INVALID_ARG, "bad graph count");
    std::vector<int32_t> ks;
    int kmax = rounds;
    if (batch) {
        ks.assign((size_t)G, rounds);
        if (k_per_graph) {
            kmax = 0;
            for (int64_t j = 0; j < G; ++j) {
                ks[(size_t)j] = k_per_graph[j];
                kmax = std::max(kmax, (int)k_per_graph[j]);
            }
        }
    }
    if (kmax < 1) return fail(ctx, KB_ERR_INVALID_ARG, "the timed call must run at least one round");
    KB_TRY(check_graph(ctx, g, opt, kmax));
    KB_CUDA(ctx, cudaSetDevice(ctx->device));
    const int64_t n = g->n;
    KB_TRY(ensure_buffer(ctx, &ctx->tune_buf, &ctx->tune_buf_bytes,
                         std::max<size_t>(256, sizeof(int32_t) * (size_t)n * (size_t)(kmax + 1))));
    int32_t* lev = reinterpret_cast<int32_t*>(ctx->tune_buf);
    std::vector<int64_t> counts((size_t)(batch ? G : 1) * (size_t)(kmax + 1));
    const int64_t m_proc = opt->direction == KB_DIR_BOTH ? 2 * g->m : g->m;
    const int32_t cls = size_class(m_proc, batch ? G : 1, batch);

    // every tuning field explicit, so no cached tuning is consulted while timing
    // (the warp task size starts at 0, by the graph's size, so the cache is set
    // aside meanwhile)
    struct CacheAside {
        kb_context* ctx;
        std::map<int32_t, kb_tuning> kept;
        explicit CacheAside(kb_context* c) : ctx(c) { kept.swap(ctx->tuned); }
        ~CacheAside() { ctx->tuned.swap(kept); }
    };
    std::unique_ptr<CacheAside> aside(new CacheAside(ctx));
    kb_options base = *opt;
    base.early_stop = 0;
    base.validate = 0;
    kb_options dflt = base;
    dflt.load_factor = 0.5f;
    dflt.hub_threshold = kb::kDefaultHubThreshold;
    dflt.small_task_vertices = 0;
    dflt.hub_chunk_edges = kb::kDefaultHubChunk;
    dflt.medium_split = kb::kDefaultMedSplit;
    dflt.small_max_degree = kb::kMidDegree;
    kb_options start = dflt;
    if (base.load_factor > 0.f) start.load_factor = base.load_factor;
    if (base.hub_threshold) start.hub_threshold = base.hub_threshold;
    if (base.small_task_vertices) start.small_task_vertices = base.small_task_vertices;
    if (base.hub_chunk_edges) start.hub_chunk_edges = base.hub_chunk_edges;
    if (base.medium_split) start.medium_split = base.medium_split;
    if (base.small_max_degree) start.small_max_degree = base.small_max_degree;

    // one warm-up run, then the best of two timed runs
    auto timed = [&](const kb_options& t, float* best_ms) -> kb_status {
        float best = 1e30f;
        for (int rep = 0; rep < 3; ++rep) {
            cudaEvent_t e0 = ctx->ev[20], e1 = ctx->ev[21];
            KB_CUDA(ctx, cudaEventRecord(e0, ctx->stream));
            if (batch)
                KB_TRY(batch_impl(ctx, g, voff, G, ks.data(), &t, lev, counts.data(), nullptr));
            else
                KB_TRY(refine_impl(ctx, g, &t, nullptr, 0, rounds, lev, counts.data(), nullptr));
            KB_CUDA(ctx, cudaEventRecord(e1, ctx->stream));
            KB_CUDA(ctx, cudaEventSynchronize(e1));
            float ms = 0.f;
            KB_CUDA(ctx, cudaEventElapsedTime(&ms, e0, e1));
            if (rep > 0) best = std::min(best, ms);
        }
        *best_ms = best;
        return KB_OK;
    };
    float default_ms = 0.f;
    KB_TRY(timed(dflt, &default_ms));
    float best = default_ms;
    kb_options win = start;
    if (std::memcmp(&start, &dflt, sizeof(kb_options)) != 0) KB_TRY(timed(start, &best));

    // coordinate search, one field at a time
    const float lfs[] = {0.35f, 0.5f, 0.7f};
    const int32_t thrs[] = {256, 512, 1024};
    const int32_t smaxs[] = {16, 24, 32};
    const int32_t splits[] = {64, 128, 256};
    const int32_t wvs[] = {64, 128, 256, 512};
    const int32_t chunks[] = {256, 512, 1024};
    const int n_values[6] = {3, 3, 3, 3, 4, 3};
    for (int axis = 0; axis < 6; ++axis) {
        kb_options center = win;
        for (int c = 0; c < n_values[axis]; ++c) {
            kb_options t = center;
            switch (axis) {
                case 0: t.load_factor = lfs[c]; break;
                case 1: t.hub_threshold = thrs[c]; break;
                case 2: t.small_max_degree = smaxs[c]; break;
                case 3: t.medium_split = splits[c]; break;
                case 4: t.small_task_vertices = wvs[c]; break;
                default: t.hub_chunk_edges = chunks[c]; break;
            }
            if (std::memcmp(&t, &center, sizeof(kb_options)) == 0) continue;  // timed already
            float ms = 0.f;
            KB_TRY(timed(t, &ms));
            if (ms < 0.98f * best) {
                best = ms;
                win = t;
            }
        }
    }
    kb_tuning T;
    std::memset(&T, 0, sizeof(T));
    T.load_factor = win.load_factor;
    T.hub_threshold = win.hub_threshold;
    T.small_task_vertices = win.small_task_vertices;
    T.hub_chunk_edges = win.hub_chunk_edges;
    T.medium_split = win.medium_split;
    T.small_max_degree = win.small_max_degree;
    T.ms = best;
    T.default_ms = default_ms;
    T.size_class = cls;
    aside.reset();
    ctx->tuned[cls] = T;
    if (T.small_task_vertices == 0) T.small_task_vertices = kb::kDefaultWarpVerts;  // the default, as a value
    if (out) *out = T;
    return KB_OK;
}

kb_status kb_clear_tuning(kb_context* ctx) {
    if (!ctx) return KB_ERR_INVALID_ARG;
    ctx->tuned.clear();
    return KB_OK;
}


kb_server_config kb_server_config_default(void) {
    kb_server_config c;
    std::memset(&c, 0, sizeof(c));
    c.max_vertices = (int64_t)1 << 26;
    c.max_edges = (int64_t)1 << 28;
    c.max_requests = 256;
    return c;
}

kb_status kb_server_create(kb_server** out, int device, void* stream, const kb_server_config* cfg) {
    if (!out || !cfg) return KB_ERR_INVALID_ARG;
    *out = nullptr;
    if (cfg->max_vertices < 1 || cfg->max_vertices > 2147483646LL || cfg->max_edges < 0 || cfg->max_requests < 1)
        return KB_ERR_INVALID_ARG;
    if (cfg->load_factor < 0.f || cfg->load_factor > 0.9f) return KB_ERR_INVALID_ARG;
    if (cfg->hub_threshold < 0 || cfg->hub_threshold > kb::kMaxHubThreshold) return KB_ERR_INVALID_ARG;
    if (cfg->hash_mode < 0 || cfg->hash_mode > 1) return KB_ERR_INVALID_ARG;
    kb_server* sv = new (std::nothrow) kb_server();
    if (!sv) return KB_ERR_OOM;
    sv->cfg = *cfg;
    sv->max_slots = 4 * cfg->max_requests;
    kb_status st = kb_create(&sv->ctx, device, stream);
    if (st != KB_OK) {
        delete sv;
        return st;
    }
    const int64_t N = cfg->max_vertices, M = std::max<int64_t>(cfg->max_edges, 1), S = sv->max_slots;
    bool ok = true;
    auto alloc = [&](void** ptr, size_t bytes) {
        if (ok && cudaMalloc(ptr, std::max<size_t>(bytes, 16)) != cudaSuccess) {
            cudaGetLastError();
            ok = false;
        }
    };
    for (int a = 0; a < 2; ++a) {
        Arena& A = sv->arena[a];
        alloc((void**)&A.row, sizeof(int64_t) * (size_t)(N + 1));
        alloc((void**)&A.col, sizeof(int32_t) * (size_t)M);
        alloc((void**)&A.lab, sizeof(int32_t) * (size_t)M);
        alloc((void**)&A.vlab, sizeof(int32_t) * (size_t)N);
        alloc((void**)&A.name, sizeof(uint32_t) * (size_t)N);
    }
    alloc((void**)&sv->vgraph, sizeof(int32_t) * (size_t)N);
    alloc((void**)&sv->voff, sizeof(int64_t) * (size_t)(S + 1));
    alloc((void**)&sv->bases, sizeof(uint32_t) * (size_t)(S + 1));
    alloc((void**)&sv->slot_up, (sizeof(int32_t*) + sizeof(int64_t) + 3) * (size_t)S);
    // the arena's block table and empty-signature minima, sized for a full arena
    const float lf = cfg->load_factor > 0.f ? cfg->load_factor : 0.5f;
    sv->table_cap = table_capacity(N, lf);
    alloc((void**)&sv->table, sizeof(uint64_t) * (size_t)sv->table_cap);
    alloc((void**)&sv->emin, sizeof(uint64_t) * (size_t)N);
    const size_t bwN = sizeof(uint32_t) * (size_t)((N >> 5) + 1);
    for (int f = 0; f < 5; ++f) alloc((void**)&sv->frz[f], bwN);
    alloc((void**)&sv->verdict, sizeof(int32_t) * (size_t)cfg->max_requests);
    if (ok && cudaMallocHost(&sv->verdict_h, sizeof(int32_t) * (size_t)cfg->max_requests) != cudaSuccess) ok = false;
    int access = 0;
    if (cudaDeviceGetAttribute(&access, cudaDevAttrPageableMemoryAccess, device) == cudaSuccess) sv->host_access = access != 0;
    if (ok) {
        ok = cudaMemset(sv->arena[0].row, 0, sizeof(int64_t)) == cudaSuccess &&
             cudaMemset(sv->arena[1].row, 0, sizeof(int64_t)) == cudaSuccess &&
             cudaMemset(sv->table, 0, sizeof(uint64_t) * (size_t)sv->table_cap) == cudaSuccess &&
             cudaMemset(sv->emin, 0xff, sizeof(uint64_t) * (size_t)N) == cudaSuccess &&
             cudaMemset(sv->frz[0], 0, bwN) == cudaSuccess && cudaMemset(sv->frz[1], 0, bwN) == cudaSuccess &&
             cudaMemset(sv->frz[2], 0, bwN) == cudaSuccess;
    }
    ok = ok && cudaStreamCreateWithFlags(&sv->up, cudaStreamNonBlocking) == cudaSuccess &&
         cudaStreamCreateWithFlags(&sv->down, cudaStreamNonBlocking) == cudaSuccess &&
         cudaEventCreateWithFlags(&sv->drained, cudaEventDisableTiming) == cudaSuccess;
    for (Stage& S : sv->stage)
        ok = ok && cudaEventCreateWithFlags(&S.full, cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&S.free, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        kb_server_destroy(sv);
        return KB_ERR_OOM;
    }
    *out = sv;
    return KB_OK;
}

kb_status kb_server_destroy(kb_server* sv) {
    if (!sv) return KB_OK;
    if (sv->ctx) {
        cudaSetDevice(sv->ctx->device);
        if (sv->ctx->stream) cudaStreamSynchronize(sv->ctx->stream); else cudaDeviceSynchronize();
    }
    // copies to and from the callers' arrays
    for (cudaStream_t c : {sv->up, sv->down})
        if (c) {
            cudaStreamSynchronize(c);
            cudaStreamDestroy(c);
        }
    if (sv->drained) cudaEventDestroy(sv->drained);
    cudaFree(sv->verdict);
    if (sv->verdict_h) cudaFreeHost(sv->verdict_h);
    for (const Draining& d : sv->draining) cudaFree(d.d_levels);
    for (auto& kv : sv->reqs)
        if (kv.second.d_levels) cudaFree(kv.second.d_levels);
    for (auto& kv : sv->level_pool)
        for (int32_t* b : kv.second) cudaFree(b);
    cudaFree(sv->table);
    cudaFree(sv->emin);
    for (int f = 0; f < 5; ++f) cudaFree(sv->frz[f]);
    for (int a = 0; a < 2; ++a) {
        Arena& A = sv->arena[a];
        cudaFree(A.row);
        cudaFree(A.col);
        cudaFree(A.lab);
        cudaFree(A.vlab);
        cudaFree(A.name);
    }
    cudaFree(sv->vgraph);
    cudaFree(sv->voff);
    cudaFree(sv->bases);
    cudaFree(sv->slot_up);
    for (Stage& S : sv->stage) {
        cudaFree(S.buf);
        if (S.full) cudaEventDestroy(S.full);
        if (S.free) cudaEventDestroy(S.free);
    }
    kb_destroy(sv->ctx);
    delete sv;
    return KB_OK;
}

const char* kb_server_last_error(const kb_server* sv) { return sv ? sv->last_error.c_str() : "no server"; }

kb_status kb_server_submit(kb_server* sv, const kb_graph* g, const kb_options* opt, int k, int32_t* levels_out,
                           int64_t* ticket) {
    static const int64_t kEmptyRow[1] = {0};
    if (!sv || !ticket) return KB_ERR_INVALID_ARG;
    if (!g || !opt) return sfail(sv, KB_ERR_INVALID_ARG, "graph and options must not be NULL");
    if (opt->subject != KB_SUBJECT_PREVIOUS)
        return sfail(sv, KB_ERR_INVALID_ARG, "served refinement takes subject = KB_SUBJECT_PREVIOUS only");
    if (g->n < 0 || g->m < 0 || k < 0 || opt->direction < 0 || opt->direction > 2)
        return sfail(sv, KB_ERR_INVALID_ARG, "bad request");
    if (g->n > 0 && !g->row_offsets) return sfail(sv, KB_ERR_INVALID_ARG, "row_offsets is NULL");
    if (g->m > 0 && !g->col_indices) return sfail(sv, KB_ERR_INVALID_ARG, "col_indices is NULL");
    if (g->n == 0 && g->m != 0) return sfail(sv, KB_ERR_INVALID_ARG, "edges without vertices");
    const int64_t mp = opt->direction == KB_DIR_BOTH ? 2 * g->m : g->m;
    if (g->n > sv->cfg.max_vertices || mp > sv->cfg.max_edges)
        return sfail(sv, KB_ERR_INVALID_ARG, "request larger than the arena");
    // the ends of the offsets here; every offset and neighbour id is checked
    // on the device at admission, before the graph reaches the shared arena
    if (g->n > 0 && (g->row_offsets[0] != 0 || g->row_offsets[g->n] != g->m))
        return sfail(sv, KB_ERR_INVALID_ARG, "row_offsets must run from 0 to m");
    ServeRequest r;
    r.n = g->n;
    r.m = g->m;
    r.m_proc = mp;
    r.opt = *opt;
    r.k = k;
    r.row = g->n > 0 ? g->row_offsets : kEmptyRow;
    r.col = g->col_indices;
    r.lab = (g->m && g->edge_labels && opt->use_edge_labels) ? g->edge_labels : nullptr;
    r.vlab = (g->n && g->vertex_labels && opt->use_vertex_labels) ? g->vertex_labels : nullptr;
    r.out = levels_out;
    r.t_submit = now_s();
    std::lock_guard<std::mutex> lk(sv->mu);
    r.ticket = sv->next_ticket++;
    *ticket = r.ticket;
    if (sv->t_first < 0) sv->t_first = r.t_submit;
    ++sv->submitted;
    const int64_t t = r.ticket;
    sv->reqs.emplace(t, std::move(r));
    sv->waiting.push_back(t);
    return KB_OK;
}

kb_status kb_server_step(kb_server* sv, int32_t* running, int32_t* waiting) {
    if (!sv) return KB_ERR_INVALID_ARG;
    sv->last_error.clear();
    return server_step(sv, running, waiting);
}

kb_status kb_server_poll(kb_server* sv, int64_t ticket, int32_t* state) {
    if (!sv || !state) return KB_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(sv->mu);
    auto it = sv->reqs.find(ticket);
    if (it == sv->reqs.end()) return KB_ERR_NOT_FOUND;
    KB_TRY(settle(sv, it->second));
    *state = it->second.state;
    return KB_OK;
}

kb_status kb_server_fetch(kb_server* sv, int64_t ticket, int32_t* levels, int64_t* counts, int32_t* levels_computed) {
    if (!sv) return KB_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(sv->mu);
    auto it = sv->reqs.find(ticket);
    if (it == sv->reqs.end()) return KB_ERR_NOT_FOUND;
    ServeRequest& r = it->second;
    KB_TRY(settle(sv, r));
    if (r.state == 3) {
        const std::string why = r.error;
        sv->reqs.erase(it);
        return sfail(sv, KB_ERR_INVALID_ARG, "request %lld was rejected at admission: %s", (long long)ticket,
                     why.c_str());
    }
    if (r.state != 2) return sfail(sv, KB_ERR_INVALID_ARG, "request %lld has not finished", (long long)ticket);
    if (levels && r.n) {
        const size_t bytes = sizeof(int32_t) * (size_t)r.n * (size_t)(r.k + 1);
        if (r.out) {
            if (levels != r.out) std::memcpy(levels, r.out, bytes);
        } else {
            std::memcpy(levels, r.levels.get(), bytes);
        }
    }
    if (counts) std::memcpy(counts, r.counts.data(), sizeof(int64_t) * r.counts.size());
    if (levels_computed) *levels_computed = r.levels_computed;
    sv->reqs.erase(it);
    return KB_OK;
}

kb_status kb_server_get_stats(kb_server* sv, kb_server_stats* st) {
    if (!sv || !st) return KB_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(sv->mu);
    for (auto& kv : sv->reqs) KB_TRY(settle(sv, kv.second));
    std::memset(st, 0, sizeof(*st));
    st->submitted = sv->submitted;
    st->completed = sv->completed;
    st->failed = sv->failed;
    for (const auto& kv : sv->reqs) st->running += kv.second.state == 1;  // (the slots are the stepping thread's)
    st->waiting = (int64_t)sv->waiting.size();
    st->steps = sv->steps;
    st->compactions = sv->compactions;
    if (!sv->latencies_ms.empty()) {
        std::vector<double> l = sv->latencies_ms;
        std::sort(l.begin(), l.end());
        auto pct = [&](double q) {
            const size_t i = (size_t)std::min<double>((double)(l.size() - 1), std::ceil(q * (double)l.size()) - 1);
            return l[i];
        };
        st->p50_ms = pct(0.50);
        st->p99_ms = pct(0.99);
        double sum = 0;
        for (double x : l) sum += x;
        st->mean_ms = sum / (double)l.size();
    }
    const double span = sv->t_first >= 0 ? now_s() - sv->t_first : 0;
    if (span > 0) {
        st->requests_per_s = (double)sv->completed / span;
        st->edge_rounds_per_s = sv->edge_rounds / span;
    }
    return KB_OK;
}

}  // extern "C"
