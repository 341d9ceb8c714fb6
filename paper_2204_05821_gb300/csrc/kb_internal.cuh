// Internal declarations of the GB300 k-bisimulation library: tile geometry,
// device-side parameter blocks, hashing and pair packing, and the host-side
// launchers implemented in kb_kernels.cu / kb_setup.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kbisim.h"

namespace kb {

// ---------------------------------------------------------------- geometry
// Vertices with more than hub_threshold edges (at most kMaxHubThreshold) are
// hubs, split into chunks of RoundParams::hub_chunk edges (256, 512 or 1024);
// medium vertices keep their pairs in one shared-memory set of 2 x
// kMaxHubThreshold entries.
constexpr int kMaxHubThreshold = 1024;
constexpr int kDefaultHubThreshold = kMaxHubThreshold;
constexpr int kDefaultHubChunk = 512;   // edges per hub-chunk CTA
constexpr int kMaxHubChunk = 1024;
constexpr int kHubThreads = 128;        // threads of a hub-chunk CTA
static_assert(kMaxHubChunk < 65536, "a chunk's edge count is packed in 16 bits");
// Medium vertices up to this degree take a warp each, larger ones a CTA
// (RoundParams::med_split, at most kMaxMedSplit).
constexpr int kMaxMedSplit = 256;
constexpr int kDefaultMedSplit = kMaxMedSplit;
constexpr int kHubFinalThreads = 256;
// Sketches (kb_hub.cu) go ahead of the exact sets from this many hub chunks on
// (a million edges), where they cost less than the launches they add, and for
// thresholds that leave room for one in every hub's set.
constexpr int64_t kSketchMinChunks = 2048;
constexpr int kSketchMinThreshold = 128;
constexpr int kProbeLimit = 1 << 22;  // bound on block-table probes per vertex
constexpr int kSmallDegree = 8;       // vertices with at most this many edges take a lane each (kb_small.cu),
constexpr int kMidDegree = 32;        // with at most this many eight lanes each (kb_medium.cu)
constexpr int kDefaultWarpVerts = 128;

constexpr uint64_t kEmptyPair = ~0ull;  // block field 0x7fffffff never occurs (n <= 2^31-2)

// bits of Counters::err
enum : int32_t { kErrTableFull = 1, kErrInvalid = 2, kErrStage = 4, kErrHubSet = 8, kErrWait = 16 };

// Rounds that one launch of the fused kernel runs at most.
constexpr int kFusedRounds = 64;
// How often one of its CTAs looks for the others before it gives up (each look a
// round trip to the L2, some seconds in all).
constexpr int32_t kFusedPolls = 1 << 24;

struct Counters {
    int32_t err;
    int32_t diff;   // set when two compared levels differ (launch_levels_differ)
    int64_t count;  // blocks at the level just assigned
    int64_t frozen; // vertices frozen for the next round (launch_freeze_clean)
    int64_t class_on[3]; // mid and medium vertices and hubs that refine next round (launch_freeze_clean)
    int64_t moved;  // re-keyed vertices whose smallest block member changed (renumbering)
    int64_t work_set;   // vertices re-keyed by a round of an incremental refinement
    int64_t graphs_on;  // graphs of a batch that refine next round (launch_graph_bases)
    // vertices re-keyed this round and their edges in the processed
    // direction, per kernel family: small, medium, hub
    int64_t keyed_v[3];
    int64_t keyed_e[3];
    int32_t dense_bad;  // a level-0 key outside [0, kDenseLabels) (launch_dense_labels)
    int64_t prev_count; // blocks at the level before
    // the fused rounds of small graphs (launch_fused_rounds): arrivals at the
    // grid's barrier, the last round run, the count before its first round and
    // after each one
    uint32_t arrived;
    int32_t last_round;
    int64_t start_count;
    int64_t round_count[kFusedRounds];
    uint32_t most_pairs;    // most distinct pairs of a vertex of the medium CTA kernel this round
    uint32_t exact_chunks;  // chunks of hubs that need their exact set (launch_hub_sketch)
    int64_t n_class[3]; // mid and medium vertices and hubs of the graph (launch_classes)
    uint32_t hub_at;    // hubs handed out (HubSink)
    uint32_t tiles[3 * 32];  // tile counts of launch_classes, up to 32 tiles
};

// Everything one refinement round reads and writes.
struct RoundParams {
    int64_t n;
    const int64_t* row;   // [n+1] CSR of the processed direction
    const int32_t* col;   // [m_proc] neighbour; bit 31 set for in-edges
    const int32_t* lab;   // [m_proc] edge label or nullptr (all labels 0)
    const int32_t* prev;  // [n] previous level (vertex labels at level 0)
    // Locality order (optional).  perm[v] is v's position in an order that puts
    // often-gathered vertices first; col then holds positions instead of ids and
    // gat holds the previous level in that order, each block named by its
    // smallest member instead of its rank (gat[perm[v]] = smallest member of
    // v's block; any injective naming of blocks gives the same partition), so
    // the per-edge gather of neighbour blocks hits a compact, cache-resident
    // head, and the renumbering rewrites gat only where a block's smallest
    // member changed.  perm == nullptr: col holds ids and the gather reads prev.
    const int32_t* perm;
    int32_t* gat;
    // Generic CSE rounds (Def. "cse"): the subject part of every key, one class
    // id (< n) per vertex; nullptr keys by the own previous block (stratified
    // bisimulation).
    const int32_t* own_key;
    // Incremental refinement (kb_refine_update): only vertices with their bit
    // set in vmask are re-keyed (nullptr: all); every other vertex keeps its old
    // grouping at this level: keep_old is the level's old row and old_min[b] the
    // smallest vertex of old block b.  The renumbering writes old_name[v], the
    // smallest vertex of v's old block, for every re-keyed vertex, and sets the
    // bits of its old and new block's names in taint where they differ.
    const uint32_t* vmask;
    const int32_t* keep_old;
    const uint32_t* old_min;
    uint32_t* old_name;
    uint32_t* taint;
    // Frozen blocks (stratified rounds, whose keys hold the own previous block):
    // a block that cannot change this round, because it has one member (a
    // vertex alone in its previous block stays alone) or because all its
    // members have no edges and it was formed by a signature round (their keys
    // are then (own block, empty set) alike).  Bit v of frozen: v is skipped by
    // the round kernels; frozen_min holds the minima of frozen blocks and
    // starts the round's bitmap of minima; a skipped vertex that is not a
    // minimum keeps its slot_of entry of the round that formed its block.  The
    // renumbering sets bit b of shared for the minimum b of every block of
    // several vertices (blocks of edgeless vertices aside: those are frozen
    // whatever their size), from joined: bit v for the vertex v that inserted
    // the table entry of such a block, set by the round kernels and cleared by
    // the renumbering.  All nullptr when every vertex is re-keyed.
    const uint32_t* frozen;
    const uint32_t* frozen_min;
    uint32_t* shared;
    uint32_t* joined;
    // Clean blocks (with frozen blocks).  minof[v] is the smallest member of
    // v's block at the level last assigned: the name its block goes by in the
    // next round's keys (prev and gather), unique over all graphs of a run.  The
    // renumbering writes it for re-keyed vertices whose block's smallest member
    // changed; a frozen vertex keeps it.  moved (when set) receives bit v for
    // every such vertex, counted in ctr->moved; under the locality order the bit
    // goes to v's position, which is what the neighbour ids hold.
    uint32_t* minof;
    uint32_t* moved;
    int32_t hub_threshold;
    int32_t small_max;    // largest degree of the small-vertex kernel (<= kSmallDegree, <= mid_max)
    int32_t mid_max;      // largest degree of the mid kernel (<= kMidDegree, <= hub_threshold)
    int32_t warp_verts;   // vertices per warp task of the small-vertex kernel; 0: by the graph's size
    int32_t hub_chunk;    // edges per hub-chunk CTA: 256, 512 or 1024
    int32_t med_split;    // medium vertices up to this degree take a warp, larger a CTA (1..kMaxMedSplit)
    int32_t hash_mode;
    uint32_t epoch;       // 1..255, tags this round's table entries
    uint64_t* table;      // [mask+1] block table: [epoch 8 | tag 24 | single bit, smallest member 32]
    uint64_t mask;
    int32_t* slot_of;     // [n] table slot of every vertex; 0x80000000|own for an empty signature
    uint64_t* emin;       // [n] smallest vertex with an empty signature per own block:
                          //     (ehigh << 32) | vertex, ehigh decreasing from round to round
    uint32_t ehigh;
    uint32_t* bitmap;     // [n/32+1] bit v set iff v is the smallest member of its block
    Counters* ctr;
    // mid (small_max < degree <= mid_max) and medium vertices (up to
    // hub_threshold), ascending
    const int32_t* mid_v;
    int64_t n_mid;
    const int32_t* med_v;
    int64_t n_med;
    // hubs (vertices with more than hub_threshold edges)
    int32_t n_hubs;
    const int32_t* hub_v;          // [n_hubs] ascending
    const int64_t* hub_chunk_off;  // [n_hubs+1]
    const int32_t* chunk_hub;      // [total chunks] hub index of every chunk
    const uint64_t* chunk_ext;     // [total chunks] (first edge << 16) | edges of every chunk
    const int64_t* hub_set_off;    // [n_hubs+1] open-addressing set per hub (hub_set_capacity slots)
    uint64_t* hub_sets;
    uint64_t* hub_acc;  // [n_hubs] sum of pair mixes over unique pairs
    uint32_t* hub_cnt;  // [n_hubs] unique pairs
    // Sketches first (kb_hub.cu): hub_exact[h] != 0 for the hubs that need their
    // exact set, whose chunks are in exact_list (ctr->exact_chunks of them); the
    // others that refine are alone in their new block.  nullptr: every hub does.
    uint32_t* hub_exact;
    int32_t* exact_list;
    uint32_t* hub_twin;      // [hub_twin_mask + 1] table of hub indices + 1
    uint32_t hub_twin_mask;
    // several graphs at once (batched refinement, serving); all null or 0 for one graph
    int32_t n_graphs;
    const int64_t* voff;       // [G+1] first vertex of every graph
    // vgraph: graph of every vertex, while keys need it: at a batch's level 0 and
    // in serving, where graphs may compute their level 0 among others' rounds.
    // (The names of blocks are unique over all graphs, so signature keys of
    // different graphs differ by themselves.)
    const int32_t* vgraph;
    const uint8_t* gmode;      // [G] 1: the graph computes its level 0 this round (serving), or nullptr
    const int32_t* vlab;       // [n] vertex labels read by graphs in level-0 mode, or nullptr (all 0)
    // Where the levels go: ids local to the graph (lgraph: graph of every vertex),
    // into one row, or (gout) to every graph's own row, nullptr for none.
    const int32_t* lgraph;
    int32_t* const* gout;
    const uint32_t* gbase_prev;   // [G+1] rank of every graph's first vertex at the previous level
    uint32_t* gbase_cur;          // [G+1] the same at this level (written by the renumbering)
};

__host__ __device__ __forceinline__ bool batched(const RoundParams& p) { return p.n_graphs > 0; }

// The subject part of vertex v's key in a signature round.
__host__ __device__ __forceinline__ int32_t own_of(const RoundParams& p, int64_t v) {
    return p.own_key ? p.own_key[v] : p.prev[v];
}

// The array the per-edge gather reads through col (see RoundParams::perm).
__host__ __device__ __forceinline__ const int32_t* gather_base(const RoundParams& p) {
    return p.perm ? p.gat : p.prev;
}

// Loads of what a kernel only reads: the previous level and the frozen bits.
// The fused kernel of small graphs writes them between its phases, so its
// translation unit (kb_fused.cu) asks for ordinary loads instead of the
// read-only path; device code is compiled per translation unit.
template <class T>
__device__ __forceinline__ T load_level(const T* x) {
#ifdef KB_LEVELS_WRITTEN
    return *x;
#else
    return __ldg(x);
#endif
}

// The previous block of neighbour word w (bit 31: direction).
__device__ __forceinline__ int32_t gather_block(const RoundParams& p, int32_t w) {
    return load_level(gather_base(p) + (w & 0x7fffffff));
}

// ---------------------------------------------------------------- hashing
// SplitMix64 output function (Steele, Lea & Flood, "Fast splittable
// pseudorandom number generators", OOPSLA 2014): a bijective 64-bit mixer.
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t x) {
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ULL;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebULL;
    x ^= x >> 31;
    return x;
}

// A signature pair (direction d, edge label l, neighbour block b) as one
// 64-bit word: label in bits 63..32, d in bit 31, b in bits 30..0.
__device__ __forceinline__ uint64_t pack_pair(int32_t label, uint32_t col_word, int32_t block) {
    return ((uint64_t)(uint32_t)label << 32) | (uint64_t)(col_word & 0x80000000u) | (uint64_t)(uint32_t)block;
}

__device__ __forceinline__ uint64_t pair_mix(uint64_t p) { return mix64(p ^ 0x9e3779b97f4a7c15ULL); }

// A hub's global dedup set: 1.5 x its degree (at most two thirds full), any
// size, home slot by multiply-shift range reduction of the pair mix.
__host__ __device__ __forceinline__ int64_t hub_set_capacity(int64_t degree) {
    const int64_t c = degree + degree / 2 + 4;
    return c < 64 ? 64 : (c & ~(int64_t)3);
}

__device__ __forceinline__ uint64_t hub_set_home(uint64_t pr, uint64_t cap) {
    return __umul64hi(pair_mix(pr), cap);
}

// Slot of (local vertex j, pair p) in a shared dedup set.
__device__ __forceinline__ uint32_t set_slot(uint64_t p, uint32_t j) {
    return (uint32_t)(mix64(p + 0x632be59bd9b4e019ULL * (uint64_t)(j + 1)) >> 20);
}

// Hash of a vertex key (own previous block, signature set).  The set enters
// through an order-independent sum of pair mixes over its distinct pairs and
// its size.  hash_mode 1 keeps only the own block (forces collisions).
__device__ __forceinline__ uint64_t vertex_hash(int32_t own, uint32_t cnt, uint64_t acc, int mode) {
    uint64_t base = mix64(((uint64_t)(uint32_t)own << 32) ^ 0x5851f42d4c957f2dULL);
    if (mode == 1) return base;
    return mix64(base ^ mix64(acc + 0xd6e8feb86659fd93ULL * ((uint64_t)cnt + 1)));
}

__device__ __forceinline__ uint32_t table_hi(uint64_t h, uint32_t epoch) {
    return (epoch << 24) | (uint32_t)(h >> 40);
}

// ---------------------------------------------------------------- launchers
// Signature rounds (kb_kernels.cu).  The round's bitmap of block minima starts
// as p.frozen_min (or empty).
void launch_clear_round(const RoundParams& p, cudaStream_t s);
// Empty the sets of the hubs that refine this round; clear the hubs' sums.
void launch_clear_hubs(const RoundParams& p, int64_t total_slots, cudaStream_t s);
// Clean blocks (RoundParams::minof).  After the renumbering of level i (minima
// in p.bitmap, names in p.minof, moved vertices in `moved`): mark =
// blocks of level i holding a vertex with an edge to a moved vertex (bit =
// the block's name; a vertex above max_scan edges counts as such).  Only vertices
// that are neither alone in their block (bitmap & ~shared) nor edgeless are
// scanned, and nothing when more than an eighth of the vertices moved.
// gactive (or nullptr): graphs that stopped are not scanned.  stop_stable: the
// pass does nothing after a round that kept the block count (a
// stable round under early stop is the last one).
void launch_dirty_blocks(const RoundParams& p, const uint32_t* edgeless, const uint32_t* moved,
                         int32_t max_scan, uint32_t* mark, const uint8_t* gactive, bool stop_stable,
                         cudaStream_t s);
// After the renumbering (stratified rounds): the frozen blocks of the next
// round.  A vertex is frozen when it is alone in its block (a minimum in bitmap
// without a mark in shared), edgeless (edgeless != null: from the first
// signature round on, a block holding an edgeless vertex holds only edgeless
// vertices with one previous block), or in a level-i block without a mark bit
// (mark != null, unless more than an eighth of the vertices moved).
struct FreezePass {
    int64_t n = 0;
    const uint32_t* bitmap = nullptr;    // block minima of the level
    uint32_t* shared = nullptr;          // in: minima of blocks of several vertices; out: exactly the frozen ones
    const uint32_t* edgeless = nullptr;
    const uint32_t* names = nullptr;     // RoundParams::minof
    const uint32_t* mark = nullptr;
    uint32_t* frozen = nullptr;          // out: frozen vertices, counted in ctr->frozen
    uint32_t* frozen_min = nullptr;      // out: the minima of frozen blocks
    uint32_t* moved_clear = nullptr;     // a bitmap to clear, or nullptr
    const uint32_t* classes[3] = {};     // mid, medium, hub: those not frozen are counted in ctr->class_on
                                         // (nullptr: an empty class)
    Counters* ctr = nullptr;
    // several graphs: all vertices of a graph that stopped (not in gactive) are
    // frozen, those of a graph that computed its level 0 in this step (gmode) are
    // not by the edgeless rule
    const int32_t* vgraph = nullptr;
    const uint8_t* gactive = nullptr;
    const uint8_t* gmode = nullptr;
    bool stop_stable = false;            // a round that kept the count is the last one: nothing to do after it
    int per_warp = 32;                   // bitmap words per warp (set by the launcher)
};
void launch_freeze_clean(const FreezePass& f, cudaStream_t s);
// Clear bits a..b-1 of a bitmap.
void launch_clear_bits(uint32_t* words, int64_t a, int64_t b, cudaStream_t s);
// The vertices this round re-keys (not in p.frozen) and their edges, per
// kernel family, into ctr->keyed_v / keyed_e (work accounting only).
void launch_round_work(const RoundParams& p, cudaStream_t s);
// Windows of consecutive vertices, or packed from the vertices that refine
// (kCompact: worth it when many are frozen; kSparse: nearly all are).
enum class SmallWindows { kConsecutive, kCompact, kSparse };
void launch_small_round(const RoundParams& p, bool level0, SmallWindows windows, cudaStream_t s);
int32_t default_task_vertices(int64_t n);  // per warp task, when the caller gives none
// The small, mid and medium vertices in one launch (kb_keys.cu).
void launch_keys(const RoundParams& p, cudaStream_t s);
void launch_mid_round(const RoundParams& p, cudaStream_t s);     // kb_medium.cu: after the small vertices,
void launch_medium_round(const RoundParams& p, cudaStream_t s);  //   after the mid ones
// Per-device kernel attributes (shared-memory carveouts); call once per device
// before the first launch and outside any stream capture.
void set_medium_kernel_attributes();
void launch_hub_sketch(const RoundParams& p, int64_t total_chunks, cudaStream_t s);  // kb_hub.cu
void launch_hub_chunk(const RoundParams& p, int64_t total_chunks, cudaStream_t s);
void launch_hub_final(const RoundParams& p, cudaStream_t s);
// Several graphs, after the rank scan: gbase_cur, and the stop test of every
// graph still in `active` (cleared when it stops; ctr->graphs_on counts the
// others).  `round`: the level just computed.
struct GraphStop {
    uint8_t* active = nullptr;        // [G]; nullptr: no test
    int round = 0;
    // a batch: stop at the graph's own k, or (early) at an unchanged count
    const int32_t* k = nullptr;       // [G]
    bool early = false;
    int32_t* last = nullptr;          // [G] receives the round
    // serving: mode 1 stops after this round, 2 when the count is prev_count's
    const uint8_t* mode = nullptr;    // [G]
    const int64_t* prev_count = nullptr;
};
// Rounds first..last (at most kFusedRounds) of one small graph in one cooperative
// launch (kb_fused.cu): p, f and the buffers as for the single passes, with the
// starting level's freeze pass done (or all_on: every vertex refines).
struct FusedRounds {
    RoundParams p;          // epoch and ehigh of round `first`
    FreezePass f;
    uint2* rank = nullptr;
    uint32_t* sums = nullptr;    // [CTAs] scratch of the rank scan
    int32_t* levels = nullptr;   // row i at levels + i * n, or
    int32_t* ping[2] = {nullptr, nullptr};  // in turn
    int64_t edges = 0;           // of the processed CSR
    int64_t total_chunks = 0;
    int first = 0, last = 0, k = 0;  // k: the call's last level
    // the starting level too, row first - 1, when its keys are small: they and the
    // label minima (launch_dense_labels), which are left empty
    const int32_t* key0 = nullptr;
    uint32_t* lmin = nullptr;
    bool stop_stable = false;    // stop at a round that keeps the count; its row and all up to k are copied
    bool all_on = false;
    uint32_t max_polls = kFusedPolls;
};
// CTAs that a cooperative launch may have (0: not available).
int fused_max_ctas();
// again: not the first launch since the counters were cleared.
cudaError_t launch_fused_rounds(const FusedRounds& a, int max_ctas, bool again, cudaStream_t s);
// Canonical renumbering: prefix of block minima, then ids.
// rank: (n/32 + 2) words, rank[w] = (minima before word w, minima bits of word w).
// The frozen, class_on and moved counters restart at 0; with frozen
// blocks moved vertices are counted, and mark (or nullptr) is cleared.
// stop_stable (frozen-block rounds under early stop): in a round that kept the
// block count (the last round) the ids are those of the previous level, and out
// is left for the caller to copy.
void launch_renumber(const RoundParams& p, uint2* rank, uint32_t* scan_tmp, int32_t* out, uint32_t* mark,
                     bool stop_stable, cudaStream_t s, const GraphStop& stop = GraphStop());
size_t scan_tmp_words(int64_t n_items);
// Level 0 of one graph whose keys (vertex labels, or a starting partition)
// are all in [0, kDenseLabels): the label partition straight from each
// label's smallest vertex, without the block table.  launch_dense_labels
// lowers lmin[label] (all ones for an unused label) to the label's smallest
// vertex (bit 31 set while it is the label's only one) and sets ctr->dense_bad if some key lies outside the range (the
// caller then takes the general path).  launch_dense_level0 then writes what
// the general level-0 pass writes: the minima bitmap and the shared-block
// marks of p, the rank words, ctr->count, the level (out), minof and the
// locality order's copy gat.  lpair: kDenseLabels (minimum, id) words of scratch.
// It leaves lmin all ones.
constexpr int kDenseLabels = 8192;
constexpr uint32_t kNoMember = 0xffffffffu;
void launch_dense_labels(int64_t n, const int32_t* key, uint32_t* lmin, Counters* ctr, cudaStream_t s);
void launch_dense_level0(const RoundParams& p, const int32_t* key, uint32_t* lmin, uint2* lpair, uint2* rank,
                         uint32_t* scan_tmp, int32_t* out, cudaStream_t s);
void launch_fill_i32(int32_t* out, int64_t n, int32_t value, cudaStream_t s);
// vgraph[v] = graph owning v
void launch_vertex_graph(const int64_t* voff, int32_t G, int64_t n, int32_t* vgraph, cudaStream_t s);

// Setup (kb_setup.cu)
// Neighbour ids in [0, n); with row also offsets monotone from 0 to m.
void launch_validate(int64_t n, int64_t m, const int64_t* row, const int32_t* col, Counters* ctr,
                     cudaStream_t s);
// in-degree histogram: deg[w] += 1 per edge (deg must be zeroed)
void launch_in_degree(int64_t m, const int32_t* col, int64_t* deg, cudaStream_t s);
// exclusive prefix of n int64 values into out[0..n] (out[n] = total); in and out may alias
void launch_scan_i64(const int64_t* in, int64_t n, int64_t* out, int64_t* tmp, cudaStream_t s);
size_t scan_i64_tmp(int64_t n);
// Build the processed CSR for IN (include_out = 0) or BOTH (include_out = 1):
//   row_p[v] = (include_out ? row[v] : 0) + in_prefix[v]
void launch_build_csr(int64_t n, int64_t m, const int64_t* row, const int32_t* col, const int32_t* lab,
                      const int64_t* in_prefix, int include_out, int64_t* row_p, int32_t* col_p,
                      int32_t* lab_p, int64_t* cursor, cudaStream_t s);
// Degree classes of the processed CSR: vertices without edges, mid, medium and
// hub vertices, a bitmap of (n >> 5) + 1 words each, pitch words apart.  The last
// three are counted in ctr->n_class and per tile in tile_counts (kClassLists
// words per tile, class_tiles(n) tiles).  check: report offsets out of order
// (kOrder), or also not from 0 to m (kAll), in ctr->err.
enum DegreeClass { kEdgeless, kMid, kMedium, kHub };
constexpr int kClassLists = 3;  // classes that are also listed
struct ClassBounds {
    int32_t small;   // largest degree of the small-vertex kernel
    int32_t mid;     // of the mid class
    int32_t medium;  // of the medium class
};
enum class CheckRows { kNone, kOrder, kAll };
// ids: two arrays whose entries have to lie in [0, n) (kErrInvalid).  hubs: room
// for the hubs and their degrees in any order (cap 0: none wanted).  The caller
// has cleared tile_counts and ctr.  One launch: on small graphs each costs more
// than its work (ids, offsets, hub list and its copies in one launch, both lists
// in one, and the bitmaps of a call cleared together: a whole call on 10^4
// vertices and 5 x 10^4 edges 185 -> 160 us, on 7 x 10^5 edges with host buffers
// 447 -> 403 us; on 10^8 edges 5070 -> 4990 us).
struct CheckIds {
    const int32_t* a[2] = {nullptr, nullptr};
    int64_t count[2] = {0, 0};
};
struct HubSink {
    int32_t* v = nullptr;
    int64_t* deg = nullptr;
    uint32_t cap = 0;
};
size_t class_tiles(int64_t n);
void launch_classes(int64_t n, int64_t m, const int64_t* row, const ClassBounds& bounds, uint32_t* bits, int64_t pitch,
                    uint32_t* tile_counts, CheckRows check, const CheckIds& ids, const HubSink& hubs, Counters* ctr,
                    cudaStream_t s);
// The vertices of one or two classes, ascending, at most cap of each, with their
// degrees unless deg is nullptr.
struct ClassList {
    DegreeClass cls = kMid;
    int64_t cap = 0;
    int32_t* out = nullptr;
    int64_t* deg = nullptr;
};
void launch_class_lists(int64_t n, const int64_t* row, const uint32_t* bits, int64_t pitch, const uint32_t* tile_counts,
                        const ClassList& a, const ClassList& b, cudaStream_t s);
// Hub and packed extent of every hub chunk (RoundParams::chunk_hub, chunk_ext).
void launch_chunk_ext(int64_t chunks, int32_t n_hubs, const int32_t* hub_v, const int64_t* chunk_off,
                      const int64_t* row, int32_t chunk, int32_t* chunk_hub, uint64_t* out, cudaStream_t s);
void launch_locality_order(int64_t n, int64_t m, const int32_t* col, uint32_t* cnt, unsigned long long* hist,
                           int32_t* perm, cudaStream_t s);
void launch_remap_cols(int64_t m, const int32_t* col, const int32_t* perm, int32_t* out, cudaStream_t s);
// Rank of every set bit of a bitmap: prefix[w] = set bits before word w, the
// total in ctr->count (kb_kernels.cu).
void launch_bitmap_rank(const uint32_t* bitmap, int64_t nw, uint32_t* scan_tmp, uint32_t* prefix, Counters* ctr,
                        cudaStream_t s);
// Summary graph (kb_summary.cu)
struct SummaryParams {
    int64_t n, m;
    const int64_t* row;         // [n+1] the caller's out-edge CSR
    const int32_t* col;         // [m]
    const int32_t* lab;         // [m] or nullptr (every label reads 0)
    int32_t dir;                // 0: x = source, y = target; 1: reversed
    const int32_t* lsrc;        // [n] block of x
    const int32_t* ldst;        // [n] block of y
    unsigned long long* table;  // [2 * cap] 16-byte slots (summary_insert_kernel); both words zero = empty
    uint64_t mask;              // cap - 1
    uint32_t* bitmap;           // [m/32+1] edges that are first occurrences
    Counters* ctr;
};
void launch_summary_insert(const SummaryParams& q, cudaStream_t s);
void launch_summary_emit(const SummaryParams& q, const uint32_t* prefix, int32_t* out_src, int32_t* out_label,
                         int32_t* out_dst, cudaStream_t s);
// fill out[i] = i (kb_kernels.cu)
void launch_iota_i32(int32_t* out, int64_t n, cudaStream_t s);
// ctr->diff |= (a != b) over n entries (kb_kernels.cu)
void launch_levels_differ(const int32_t* a, const int32_t* b, int64_t n, Counters* ctr, cudaStream_t s);
// Incremental refinement (kb_update.cu)
void launch_dirty_from_moved(int64_t n, int64_t m, const int64_t* row, const int32_t* col, const uint32_t* moved,
                             uint32_t* dirty, cudaStream_t s);
void launch_work_set(int64_t n, const int32_t* prev, const uint32_t* changed, const uint32_t* moved,
                     const uint32_t* dirty, uint32_t* flag, uint32_t* wmask, Counters* ctr, cudaStream_t s);
void launch_old_min(int64_t n, const int32_t* level, uint32_t* old_min, cudaStream_t s);
void launch_keep_bits(int64_t n, const uint32_t* wmask, const int32_t* old, const uint32_t* old_min, uint32_t* bitmap,
                      cudaStream_t s);
void launch_moved(int64_t n, const uint32_t* wmask, const uint32_t* old_name, const uint32_t* taint, uint32_t* moved,
                  Counters* ctr, cudaStream_t s);
// Level 0 without labels: {V} (out all 0), with RoundParams::old_name and taint.
void launch_one_block(const RoundParams& p, int32_t* out, cudaStream_t s);
void launch_check_ids(int64_t count, int64_t n, const int32_t* a, Counters* ctr, cudaStream_t s);
// Bits of the changed vertices; ctr->work_set += vertices in the blocks of
// `level` that hold one (touched: a zeroed bitmap of n bits).
void launch_changed(int64_t n, int64_t count, const int32_t* ids, const int32_t* level, uint32_t* bits,
                    uint32_t* touched, Counters* ctr, cudaStream_t s);
// Copy row src of the level store to the rows [first, last] of levels (src not among them).
void launch_copy_rows(int32_t* levels, int64_t n, int src, int first, int last, cudaStream_t s);

// ---- serving arena (kb_serve.cu)
// Copy vertices [src_vbase, src_vbase+n] and edges [src_ebase, src_ebase+m)
// of a CSR into an arena at dst_vbase / dst_ebase, rebasing row offsets and
// neighbour ids (the in-edge bit of a neighbour id is kept).  Labels may be
// null (written as 0).  When given, block names (RoundParams::minof) move too.
struct PlaceArgs {
    const int64_t* srow;
    const int32_t* scol;
    const int32_t* slab;
    const int32_t* svlab;
    const uint32_t* sname;
    int64_t* drow;
    int32_t* dcol;
    int32_t* dlab;
    int32_t* dvlab;
    uint32_t* dname;
    int64_t n, m;
    int64_t src_vbase, dst_vbase, src_ebase, dst_ebase;
};
void launch_place(const PlaceArgs& a, cudaStream_t s);
// From arrays that the device may read in host memory (source bases 0), checked;
// *verdict, cleared by the caller, becomes 1 when they are malformed.
void launch_place_checked(const PlaceArgs& a, int32_t* verdict, cudaStream_t s);
}  // namespace kb
