// Refinement-round kernels of the GB300 k-bisimulation library.
//
// One round (paper Alg. 1, one pass of the loop; Def. "signature"):
//   1. kb_small.cu / kb_medium.cu: every non-hub vertex gathers its (direction,
//      edge label, previous block of neighbour) pairs, drops duplicates, hashes
//      (own previous block, pair set) and finds or inserts its key in the
//      block table.  A hash match is accepted only after the full signature
//      compare (the paper's implementations trust the hash; Section 4.3 notes
//      BRS is only correct while hashes do not collide).
//   2. hub_chunk_kernel / hub_final_kernel: the same for vertices with more
//      than hub_threshold edges, split over many CTAs.
//   3. renumber: the block table keeps the smallest member of every block; a
//      bitmap marks those minima, its prefix count gives every block its
//      canonical id (rank of its smallest member).
//   4. freeze (stratified single-graph rounds): blocks that cannot change in
//      the next round -- one member, or formed by a round from edgeless
//      vertices -- are skipped by steps 1-2 there and keep their minima.
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_device.cuh"
#include "kb_internal.cuh"
#include "kb_round.cuh"

namespace kb {
namespace {

// A chunk per CTA, or (after sketches) the listed chunks in strides of the grid.
template <int kChunk>
__global__ void __launch_bounds__(kHubThreads) hub_chunk_kernel(const RoundParams p) {
    __shared__ HubChunkSmem<kChunk> sm;
    if (!p.exact_list) {
        hub_chunk<kChunk, kHubThreads>(p, sm, blockIdx.x);
        return;
    }
    const uint32_t total = p.ctr->exact_chunks;
    for (uint32_t i = blockIdx.x; i < total; i += gridDim.x) {
        hub_chunk<kChunk, kHubThreads>(p, sm, p.exact_list[i]);
        __syncthreads();  // the shared sets start afresh
    }
}

__global__ void __launch_bounds__(kHubFinalThreads) hub_final_kernel(const RoundParams p) {
    __shared__ HubFinalSmem sm;
    hub_final(p, sm, (int)blockIdx.x);
}

// ----------------------------------------------------------------------------
// Canonical renumbering
// ----------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_sum_u32(uint32_t x, uint32_t* tmp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    if (lane == 0) tmp[warp] = x;
    __syncthreads();
    uint32_t t = 0;
    if (warp == 0) {
        t = lane < (int)(blockDim.x >> 5) ? tmp[lane] : 0u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    }
    __syncthreads();
    return t;
}

// exclusive scan of one value per thread (blockDim = kScanThreads)
__device__ __forceinline__ uint32_t block_exscan_u32(uint32_t x, uint32_t* tmp, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) tmp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = tmp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        tmp[lane] = w;
    }
    __syncthreads();
    const uint32_t base = warp > 0 ? tmp[warp - 1] : 0u;
    *total = tmp[31];
    __syncthreads();
    return base + incl - x;
}

__global__ void __launch_bounds__(kScanThreads) popc_reduce_kernel(const uint32_t* bitmap, int64_t nw,
                                                                  uint32_t* block_sums) {
    __shared__ uint32_t tmp[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    uint32_t s = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = base + (int64_t)u * kScanThreads + threadIdx.x;
        if (i < nw) s += __popc(bitmap[i]);
    }
    s = block_sum_u32(s, tmp);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = s;
}

// Rank of every set bit: prefix[w] = set bits before word w, or with rank
// given instead, rank[w] = (prefix[w], bitmap[w]), so a rank lookup is one
// 8-byte load.  Every block finds the set bits before its tile by itself: from
// the tiles' sums (popc_reduce_kernel), or with block_sums null from the words
// of the tiles before it.  The last block writes the total (and, for several
// graphs, rank[nw]) and clears the counters that the passes after the
// renumbering add to.
__global__ void __launch_bounds__(kScanThreads) popc_scan_kernel(const uint32_t* bitmap, int64_t nw,
                                                                const uint32_t* block_sums, uint32_t* prefix,
                                                                uint2* rank, bool rank_total, Counters* ctr) {
    __shared__ uint32_t tmp[32];
    __shared__ uint32_t s_before;
    uint32_t before = 0;
    if (block_sums) {
        for (int64_t i = threadIdx.x; i < blockIdx.x; i += kScanThreads) before += block_sums[i];
    } else {
        for (int64_t i = threadIdx.x; i < (int64_t)blockIdx.x * kScanTile; i += kScanThreads) before += __popc(bitmap[i]);
    }
    before = block_sum_u32(before, tmp);
    if (threadIdx.x == 0) s_before = before;
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t w[kScanItems], c[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = base + u;
        w[u] = i < nw ? bitmap[i] : 0u;
        c[u] = (uint32_t)__popc(w[u]);
        s += c[u];
    }
    uint32_t total;
    uint32_t ex = block_exscan_u32(s, tmp, &total);  // its barriers publish s_before
    ex += s_before;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        const uint32_t all = s_before + total;
        ctr->prev_count = ctr->count;
        ctr->count = (int64_t)all;
        ctr->frozen = 0;
        for (int k = 0; k < 3; ++k) ctr->class_on[k] = 0;
        ctr->moved = 0;
        ctr->graphs_on = 0;
        ctr->most_pairs = 0;
        if (rank_total) rank[nw] = make_uint2(all, 0u);
    }
#pragma unroll
    for (int u = 0; u < kScanItems; ++u) {
        const int64_t i = base + u;
        if (i < nw) {
            if (rank)
                rank[i] = make_uint2(ex, w[u]);
            else
                prefix[i] = ex;
        }
        ex += c[u];
    }
}

// Up to this many tiles one launch does the scan, each block counting the words
// before its tile: the last of 8 reads 28,672 words (7 per thread and tile
// before it), less than the 3 us that the launch of a reduction costs.
constexpr int64_t kScanDirect = 8;

void rank_scan(const uint32_t* bitmap, int64_t nw, uint32_t* scan_tmp, uint32_t* prefix, uint2* rank, bool rank_total,
               Counters* ctr, cudaStream_t s) {
    const int64_t nb = (nw + kScanTile - 1) / kScanTile;
    const bool direct = nb <= kScanDirect;
    if (!direct) popc_reduce_kernel<<<(unsigned)nb, kScanThreads, 0, s>>>(bitmap, nw, scan_tmp);
    popc_scan_kernel<<<(unsigned)nb, kScanThreads, 0, s>>>(bitmap, nw, direct ? nullptr : scan_tmp, prefix, rank,
                                                           rank_total, ctr);
}

__global__ void __launch_bounds__(256) assign_kernel(const RoundParams p, const uint2* rank, int32_t* out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < p.n; v += stride) {
        uint32_t mn = (uint32_t)v;
        if (!vertex_active(p, v)) {
            mn = p.old_min[p.keep_old[v]];  // incremental: its old block stays
            if ((int64_t)mn >= p.n) mn = (uint32_t)v;
        } else {
            if (!((p.bitmap[v >> 5] >> (v & 31)) & 1u)) {
                mn = block_min(p, v);
                if ((int64_t)mn >= p.n) mn = (uint32_t)v;  // only after a reported device error
            }
            if (p.taint) note_old_name(p, v, mn);
        }
        const uint2 rw = rank[mn >> 5];
        const int32_t b = (int32_t)(rw.x + __popc(rw.y & ((1u << (mn & 31)) - 1u)));
        out[v] = b;
        if (p.perm) p.gat[p.perm[v]] = (int32_t)mn;  // the block by its smallest member
    }
}

__global__ void __launch_bounds__(256) assign_frozen_kernel(const RoundParams p, const uint2* rank, int32_t* out,
                                                             uint32_t* moved, uint32_t* mark, bool stop_stable) {
    // a round that kept the block count kept every block (blocks only split):
    // under early stop it is the last one, and the caller copies the level
    if (stop_stable && p.ctr->count == p.ctr->prev_count) return;
    __shared__ uint32_t s_moved;
    assign_frozen(p, rank, out, moved, mark, &s_moved);
}

__global__ void __launch_bounds__(256) dirty_blocks_kernel(const RoundParams p, const uint32_t* edgeless,
                                                            const uint32_t* moved, int32_t max_scan, uint32_t* mark,
                                                            int per_warp, const uint8_t* gactive, bool stop_stable) {
    if (!few_moved(p)) return;
    if (stop_stable && p.ctr->count == p.ctr->prev_count) return;  // the last round: nothing follows
    dirty_blocks(p, edgeless, moved, max_scan, mark, per_warp, gactive,
                 ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * per_warp);
}

__global__ void __launch_bounds__(256) freeze_clean_kernel(const FreezePass f) {
    __shared__ uint32_t s_clean[8][32];
    __shared__ uint32_t s_on[4];
    if (f.stop_stable && f.ctr->count == f.ctr->prev_count) return;  // the last round: nothing follows
    if (threadIdx.x < 4) s_on[threadIdx.x] = 0u;
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    freeze_clean(f, s_clean[warp], s_on, ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * f.per_warp);
    __syncthreads();
    add_frozen(f.ctr, s_on);
}

// The vertices a round re-keys (those not in frozen; all when frozen is null)
// and their processed edges, per kernel family: small (at most small_max
// edges), medium, hub (more than thr edges).
__global__ void __launch_bounds__(256) round_work_kernel(int64_t n, const int64_t* row, const uint32_t* frozen,
                                                          int32_t small_max, int32_t thr, Counters* ctr) {
    __shared__ unsigned long long s_sum[6][8];
    unsigned long long c[6] = {0, 0, 0, 0, 0, 0};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (frozen && ((frozen[v >> 5] >> (v & 31)) & 1u)) continue;
        const int64_t d = row[v + 1] - row[v];
        const int f = d <= small_max ? 0 : (d > thr ? 2 : 1);
        c[f] += 1;
        c[3 + f] += (unsigned long long)d;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c[k] += __shfl_xor_sync(kFull, c[k], o);
        if ((threadIdx.x & 31) == 0) s_sum[k][threadIdx.x >> 5] = c[k];
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        unsigned long long t = 0;
        for (int w = 0; w < 8; ++w) t += s_sum[threadIdx.x][w];
        int64_t* dst = threadIdx.x < 3 ? &ctr->keyed_v[threadIdx.x] : &ctr->keyed_e[threadIdx.x - 3];
        if (t) atomicAdd(reinterpret_cast<unsigned long long*>(dst), t);
    }
}

// Clear bits a..b-1 of a bitmap (partial words at the ends keep their other bits).
__global__ void clear_bits_kernel(uint32_t* words, int64_t a, int64_t b) {
    const int64_t w0 = a >> 5, w1 = (b - 1) >> 5;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t w = w0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w <= w1; w += stride) {
        uint32_t keep = 0u;
        if (w == w0 && (a & 31)) keep |= (1u << (a & 31)) - 1u;
        if (w == w1 && (b & 31)) keep |= ~((1u << (b & 31)) - 1u);
        words[w] &= keep;
    }
}

// Refill the sets of the hubs that refine this round with the empty pair, in
// tiles of kClearTile consecutive slots of all sets together (one hub's set
// can hold 10^8 slots; large tiles keep the per-tile search for the first hub
// rare).  Sets hold at least 64 slots, so a tile overlaps at most
// kClearTile / 64 + 1 hubs; they start at multiples of 4 slots, so a 16-byte
// store never straddles two sets.
constexpr int kClearTile = 65536;
constexpr int kClearHubs = kClearTile / 64 + 1;

__global__ void __launch_bounds__(256) clear_hub_sets_kernel(const RoundParams p, int64_t tile) {
    __shared__ int s_h0;
    __shared__ int64_t s_end[kClearHubs];
    __shared__ uint8_t s_ref[kClearHubs];
    const int64_t total = p.hub_set_off[p.n_hubs];
    const int64_t t0 = (int64_t)blockIdx.x * tile;
    const int64_t t1 = min(total, t0 + tile);
    if (threadIdx.x == 0) {
        int lo = 0, hi = p.n_hubs - 1;  // first hub whose set ends after t0
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (p.hub_set_off[mid + 1] > t0) hi = mid; else lo = mid + 1;
        }
        s_h0 = lo;
    }
    __syncthreads();
    bool any = false;
    for (int i = threadIdx.x; i < kClearHubs; i += blockDim.x) {
        const int h = s_h0 + i;
        const bool in = h < p.n_hubs && p.hub_set_off[h] < t1;
        s_end[i] = in ? p.hub_set_off[h + 1] : t1;
        s_ref[i] = in && hub_is_exact(p, h);
        any |= s_ref[i] != 0;
        if (!in) break;  // later entries keep their stale values: the walk below stops at this one
    }
    if (!__syncthreads_or(any)) return;
    ulonglong2* sets2 = reinterpret_cast<ulonglong2*>(p.hub_sets);
    const ulonglong2 e = make_ulonglong2(kEmptyPair, kEmptyPair);
    const bool pairs = (reinterpret_cast<uintptr_t>(sets2) & 15) == 0;  // (a caller's workspace may start at any 8 bytes)
    int j = 0;
    for (int64_t s = t0 + 2 * threadIdx.x; s < t1; s += 2 * blockDim.x) {
        while (j < kClearHubs - 1 && s_end[j] <= s) ++j;
        if (!s_ref[j]) continue;
        if (pairs)
            sets2[s >> 1] = e;
        else
            p.hub_sets[s] = p.hub_sets[s + 1] = kEmptyPair;
    }
}

// ----------------------------------------------------------------------------
// Level 0 over small labels.  A label's entry is its smallest vertex so far,
// with kSingleBit while it has only that one (all ones: none yet).  A shared
// entry is read before the atomicMin that would lower it: after a label's first
// members, a CTA's later (larger) vertices leave it alone.  Knowing here which
// labels have several members saves the assignment its marks of shared blocks
// (one atomic per label and CTA on the few words that hold the labels' smallest
// vertices): 171 -> 13 us for it at 2.5 x 10^6 vertices, 569 -> 113 us at
// 2 x 10^7 with the locality order (the minima pass itself 21 -> 31 us).
// ----------------------------------------------------------------------------
constexpr int kDenseThreads = 512;


// Lower an entry to `member`: a vertex, with kSingleBit when it is the only one
// its side has seen.
__device__ __forceinline__ void see_member(uint32_t* entry, uint32_t member) {
    const uint32_t old = atomicMin(entry, member);
    if (old != kNoMember && ((member | old) & kSingleBit))  // several members together: the entry loses the bit
        atomicMin(entry, min(member & kVertexMask, old & kVertexMask));
}

__device__ __forceinline__ void see_label(uint32_t* s_min, int64_t v, int32_t l, bool& bad) {
    if ((uint32_t)l >= (uint32_t)kDenseLabels) {
        bad = true;
        return;
    }
    if (s_min[l] > (uint32_t)v) see_member(&s_min[l], (uint32_t)v | kSingleBit);
}

__global__ void __launch_bounds__(kDenseThreads) dense_label_min_kernel(int64_t n, const int32_t* key, uint32_t* lmin,
                                                                         Counters* ctr) {
    __shared__ uint32_t s_min[kDenseLabels];
    for (int i = threadIdx.x; i < kDenseLabels; i += blockDim.x) s_min[i] = kNoMember;
    __syncthreads();
    bool bad = false;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if ((reinterpret_cast<uintptr_t>(key) & 15) == 0) {
        const int64_t n4 = n >> 2;  // four keys per 16-byte load
        const int4* k4 = reinterpret_cast<const int4*>(key);
        for (int64_t i = t; i < n4; i += stride) {
            const int4 q = __ldcs(k4 + i);
            see_label(s_min, 4 * i, q.x, bad);
            see_label(s_min, 4 * i + 1, q.y, bad);
            see_label(s_min, 4 * i + 2, q.z, bad);
            see_label(s_min, 4 * i + 3, q.w, bad);
        }
        done = n4 << 2;
    }
    for (int64_t v = done + t; v < n; v += stride) see_label(s_min, v, __ldcs(key + v), bad);
    if (bad) atomicOr(&ctr->dense_bad, 1);
    __syncthreads();
    for (int i = threadIdx.x; i < kDenseLabels; i += blockDim.x)
        if (s_min[i] != kNoMember && __ldcg(lmin + i) > (s_min[i] & kVertexMask)) see_member(&lmin[i], s_min[i]);
}

// Every used label's smallest vertex is a block minimum, marked as shared when
// the label has other members.
__global__ void dense_mark_kernel(const RoundParams p, const uint32_t* lmin) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= kDenseLabels) return;
    const uint32_t e = lmin[l];
    if (e == kNoMember) return;
    const uint32_t m = e & kVertexMask;
    atomicOr(&p.bitmap[m >> 5], 1u << (m & 31));
    if (p.shared && !(e & kSingleBit)) atomicOr(&p.shared[m >> 5], 1u << (m & 31));
}

// (smallest vertex, canonical id) of every used label; leaves the minima empty
// for the next level 0
__global__ void dense_ids_kernel(uint32_t* lmin, const uint2* rank, uint2* lpair) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= kDenseLabels) return;
    const uint32_t e = lmin[l], m = e & kVertexMask;
    uint32_t id = 0u;
    if (e != kNoMember) {
        lmin[l] = kNoMember;
        const uint2 rw = rank[m >> 5];
        id = rw.x + __popc(rw.y & ((1u << (m & 31)) - 1u));
    }
    lpair[l] = make_uint2(m, id);
}

// The level, minof and the locality order's copy.  The 64 KB label table stays
// in L1.
__global__ void __launch_bounds__(256) dense_assign_kernel(const RoundParams p, const int32_t* key,
                                                           const uint2* lpair, int32_t* out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < p.n; v += stride) {
        const uint32_t l = (uint32_t)__ldcs(key + v);
        if (l >= (uint32_t)kDenseLabels) {  // the keys changed since they were checked
            set_error(p.ctr, kErrInvalid);
            continue;
        }
        const uint2 e = __ldg(lpair + l);
        const uint32_t mn = e.x;
        if (p.taint) note_old_name(p, v, mn);
        out[v] = (int32_t)e.y;
        if (p.perm) p.gat[p.perm[v]] = (int32_t)mn;  // the block by its smallest member
        if (p.minof) p.minof[v] = mn;
    }
}

// Rank of every graph's first vertex (the first vertex of a graph is always the
// smallest member of its block), and the graphs' stop test (GraphStop).
__device__ __forceinline__ uint32_t rank_at(const RoundParams& p, const uint2* rank, int64_t x) {
    if (x >= p.n) return rank[(p.n >> 5) + 1].x;
    const uint2 rw = rank[x >> 5];
    return rw.x + __popc(rw.y & ((1u << (x & 31)) - 1u));
}

__global__ void graph_base_kernel(const RoundParams p, const uint2* rank, const GraphStop st) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g > p.n_graphs) return;
    const uint32_t base = rank_at(p, rank, p.voff[g]);
    p.gbase_cur[g] = base;
    if (!st.active || g == p.n_graphs || !st.active[g]) return;
    const uint32_t count = rank_at(p, rank, p.voff[g + 1]) - base;
    bool stop;
    if (st.k) {
        st.last[g] = st.round;
        stop = st.round >= st.k[g] || (st.early && count == p.gbase_prev[g + 1] - p.gbase_prev[g]);
    } else {
        stop = st.mode[g] == 1 || (st.mode[g] == 2 && (int64_t)count == st.prev_count[g]);
    }
    if (stop)
        st.active[g] = 0;
    else
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctr->graphs_on), 1ull);
}

// vgraph[v] = graph owning v, in tiles (a CTA per graph leaves most of the chip
// idle: 282 us for 16 graphs of 5 x 10^6 vertices together).
constexpr int kGraphPer = 8;
__global__ void __launch_bounds__(256) vertex_graph_kernel(const int64_t* voff, int64_t G, int64_t n, int32_t* vgraph) {
    __shared__ int32_t s_g[256 * kGraphPer];
    const int64_t v0 = (int64_t)blockIdx.x * 256 * kGraphPer;
    tile_sources<256, kGraphPer>(G, voff, v0, min(n, v0 + 256 * kGraphPer), s_g);
    for (int i = threadIdx.x; i < 256 * kGraphPer && v0 + i < n; i += 256) vgraph[v0 + i] = s_g[i];
}

__global__ void fill_i32_kernel(int32_t* out, int64_t n, int32_t value) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = value;
}

__global__ void iota_i32_kernel(int32_t* out, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = (int32_t)i;
}

__global__ void levels_differ_kernel(const int32_t* a, const int32_t* b, int64_t n, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool d = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) d |= a[i] != b[i];
    if (__any_sync(kFull, d) && (threadIdx.x & 31) == 0) atomicOr(&ctr->diff, 1);
}

int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 64) b = 152 * 64;
    return (int)b;
}

}  // namespace

void launch_clear_round(const RoundParams& p, cudaStream_t s) {
    const size_t bytes = sizeof(uint32_t) * (size_t)((p.n >> 5) + 1);
    if (p.frozen_min)
        cudaMemcpyAsync(p.bitmap, p.frozen_min, bytes, cudaMemcpyDeviceToDevice, s);
    else
        cudaMemsetAsync(p.bitmap, 0, bytes, s);
}

void launch_clear_hubs(const RoundParams& p, int64_t total_slots, cudaStream_t s) {
    if (p.n_hubs <= 0) return;
    cudaMemsetAsync(p.hub_acc, 0, sizeof(uint64_t) * (size_t)p.n_hubs, s);
    cudaMemsetAsync(p.hub_cnt, 0, sizeof(uint32_t) * (size_t)p.n_hubs, s);
    if (total_slots <= 0) return;
    if (!p.frozen && !p.hub_exact) {
        cudaMemsetAsync(p.hub_sets, 0xff, sizeof(uint64_t) * (size_t)total_slots, s);
        return;
    }
    // short tiles while the sets are small, so that every SM stores (18 us for
    // 3 x 10^5 slots in tiles of 65536, 5 us in tiles of 2048)
    const int64_t per = total_slots / (152 * 8);
    const int64_t tile = std::min<int64_t>(kClearTile, std::max<int64_t>(2048, (per + 1023) & ~(int64_t)1023));
    clear_hub_sets_kernel<<<(unsigned)((total_slots + tile - 1) / tile), 256, 0, s>>>(p, tile);
}

// Bitmap words per warp of the dirty and freeze passes: 32, fewer while that
// leaves SMs idle (a lane walks up to as many candidates as its warp has words:
// 17 and 11 us for 3 x 10^5 vertices on the 37 CTAs that 32 words give).
static int words_per_warp(int64_t nw) {
    return (int)std::min<int64_t>(32, std::max<int64_t>(1, nw / (152 * 32)));
}

void launch_dirty_blocks(const RoundParams& p, const uint32_t* edgeless, const uint32_t* moved,
                         int32_t max_scan, uint32_t* mark, const uint8_t* gactive, bool stop_stable,
                         cudaStream_t s) {
    if (p.n <= 0) return;
    const int64_t nw = (p.n >> 5) + 1;
    const int per = words_per_warp(nw);
    const int64_t warps = (nw + per - 1) / per;
    dirty_blocks_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(p, edgeless, moved, max_scan, mark, per,
                                                                     gactive, stop_stable);
}

void launch_freeze_clean(const FreezePass& f, cudaStream_t s) {
    if (f.n <= 0) return;
    const int64_t nw = (f.n >> 5) + 1;
    FreezePass g = f;
    g.per_warp = words_per_warp(nw);
    const int64_t warps = (nw + g.per_warp - 1) / g.per_warp;
    freeze_clean_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(g);
}

void launch_round_work(const RoundParams& p, cudaStream_t s) {
    if (p.n <= 0) return;
    const int g = grid_for(p.n, 256) < 1216 ? grid_for(p.n, 256) : 1216;
    round_work_kernel<<<g, 256, 0, s>>>(p.n, p.row, p.frozen, p.mid_max, p.hub_threshold, p.ctr);
}

void launch_clear_bits(uint32_t* words, int64_t a, int64_t b, cudaStream_t s) {
    if (b <= a) return;
    const int64_t w0 = a >> 5, w1 = (b - 1) >> 5;
    clear_bits_kernel<<<grid_for(w1 - w0 + 1, 256), 256, 0, s>>>(words, a, b);
}

void launch_hub_chunk(const RoundParams& p, int64_t total_chunks, cudaStream_t s) {
    if (p.n_hubs <= 0 || total_chunks <= 0) return;
    // after sketches few chunks may be left: a grid that fills the chip walks them
    const unsigned grid = (unsigned)(p.exact_list ? std::min<int64_t>(total_chunks, 152 * 12 * 4) : total_chunks);
    if (p.hub_chunk == 256)
        hub_chunk_kernel<256><<<grid, kHubThreads, 0, s>>>(p);
    else if (p.hub_chunk == 1024)
        hub_chunk_kernel<1024><<<grid, kHubThreads, 0, s>>>(p);
    else
        hub_chunk_kernel<kDefaultHubChunk><<<grid, kHubThreads, 0, s>>>(p);
}

void launch_hub_final(const RoundParams& p, cudaStream_t s) {
    if (p.n_hubs <= 0) return;
    hub_final_kernel<<<(unsigned)p.n_hubs, kHubFinalThreads, 0, s>>>(p);
}

size_t scan_tmp_words(int64_t n_items) { return (size_t)((n_items + kScanTile - 1) / kScanTile) + 1; }

void launch_bitmap_rank(const uint32_t* bitmap, int64_t nw, uint32_t* scan_tmp, uint32_t* prefix, Counters* ctr,
                        cudaStream_t s) {
    rank_scan(bitmap, nw, scan_tmp, prefix, nullptr, false, ctr, s);
}

void launch_renumber(const RoundParams& p, uint2* rank, uint32_t* scan_tmp, int32_t* out, uint32_t* mark,
                     bool stop_stable, cudaStream_t s, const GraphStop& stop) {
    const int64_t nw = (p.n >> 5) + 1;
    rank_scan(p.bitmap, nw, scan_tmp, nullptr, rank, batched(p), p.ctr, s);
    if (batched(p)) graph_base_kernel<<<(p.n_graphs + 1 + 255) / 256, 256, 0, s>>>(p, rank, stop);
    if (p.n <= 0) return;
    if (p.minof)
        assign_frozen_kernel<<<grid_for(p.n, 256), 256, 0, s>>>(p, rank, out, p.moved, mark, stop_stable);
    else
        assign_kernel<<<grid_for(p.n, 256), 256, 0, s>>>(p, rank, out);
}

void launch_dense_labels(int64_t n, const int32_t* key, uint32_t* lmin, Counters* ctr, cudaStream_t s) {
    if (n <= 0) return;
    int64_t grid = (n + kDenseThreads - 1) / kDenseThreads;
    if (grid > 152 * 4) grid = 152 * 4;  // each CTA flushes its label table once
    dense_label_min_kernel<<<(unsigned)grid, kDenseThreads, 0, s>>>(n, key, lmin, ctr);
}

void launch_dense_level0(const RoundParams& p, const int32_t* key, uint32_t* lmin, uint2* lpair, uint2* rank,
                         uint32_t* scan_tmp, int32_t* out, cudaStream_t s) {
    if (p.n <= 0) return;
    const int64_t nw = (p.n >> 5) + 1;
    dense_mark_kernel<<<(kDenseLabels + 255) / 256, 256, 0, s>>>(p, lmin);
    rank_scan(p.bitmap, nw, scan_tmp, nullptr, rank, false, p.ctr, s);
    dense_ids_kernel<<<(kDenseLabels + 255) / 256, 256, 0, s>>>(lmin, rank, lpair);
    dense_assign_kernel<<<grid_for(p.n, 256), 256, 0, s>>>(p, key, lpair, out);
}

void launch_vertex_graph(const int64_t* voff, int32_t G, int64_t n, int32_t* vgraph, cudaStream_t s) {
    if (G <= 0 || n <= 0) return;
    const int64_t tile = 256 * kGraphPer;
    vertex_graph_kernel<<<(unsigned)((n + tile - 1) / tile), 256, 0, s>>>(voff, G, n, vgraph);
}

void launch_iota_i32(int32_t* out, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    iota_i32_kernel<<<grid_for(n, 256), 256, 0, s>>>(out, n);
}

void launch_levels_differ(const int32_t* a, const int32_t* b, int64_t n, Counters* ctr, cudaStream_t s) {
    if (n <= 0) return;
    levels_differ_kernel<<<grid_for(n, 256), 256, 0, s>>>(a, b, n, ctr);
}

void launch_fill_i32(int32_t* out, int64_t n, int32_t value, cudaStream_t s) {
    if (n <= 0) return;
    fill_i32_kernel<<<grid_for(n, 256), 256, 0, s>>>(out, n, value);
}

}  // namespace kb
