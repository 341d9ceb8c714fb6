// Device helpers shared by the round kernels: the block-table protocol
// (probe, insert, join) and the bitmap of block minima.
#pragma once

#include "kb_internal.cuh"

namespace kb {

constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ void set_error(Counters* c, int32_t bit) { atomicOr(&c->err, bit); }

__device__ __forceinline__ uint64_t volatile_load(const uint64_t* p) {
    return *reinterpret_cast<const volatile uint64_t*>(p);
}

// Toggle membership of v in the set of block minima.  Every vertex that ever
// becomes the minimum of its slot is toggled on once and off once when a
// smaller member replaces it, so the final bitmap holds exactly the minima,
// whatever order the toggles land in.
__device__ __forceinline__ void toggle_min(uint32_t* bitmap, uint32_t v) {
    atomicXor(&bitmap[v >> 5], 1u << (v & 31));
}

// A table entry's low word holds the smallest member of its block so far; the
// bit above it is set while the block has only the vertex that inserted it.
constexpr uint32_t kSingleBit = 0x80000000u;
constexpr uint32_t kVertexMask = 0x7fffffffu;

// Lower the smallest member of slot `pos` (same epoch and tag as ours) to v.
// A block's minimum only decreases during a round, so an entry that another
// vertex joined already and whose minimum is at or below v needs no atomic:
// hot keys would otherwise take one serialised atomic per join.  The one join
// that finds the entry single records its inserter in p.joined: the
// renumbering turns that bit into the mark of the block's minimum, one atomic
// per shared block (marks sent by every other member, through a cache per
// CTA, were most of the renumbering: 450 -> 260 us in round 1 of the 2 x 10^8
// edge graph, 283 -> 99 us with 10^8 edges and one label class).
__device__ __forceinline__ void join_block(const RoundParams& p, uint64_t pos, uint32_t hi, uint32_t v) {
    const uint32_t seen = (uint32_t)volatile_load(&p.table[pos]);
    if (seen <= v) return;  // the single bit is above every vertex
    const uint32_t want = min(v, seen & kVertexMask);
    const uint32_t old = (uint32_t)atomicMin(reinterpret_cast<unsigned long long*>(&p.table[pos]),
                                             (unsigned long long)(((uint64_t)hi << 32) | want));
    const uint32_t prev_min = old & kVertexMask;
    if ((old & kSingleBit) && p.joined) atomicOr(&p.joined[prev_min >> 5], 1u << (prev_min & 31));
    if (want < prev_min) {
        toggle_min(p.bitmap, v);
        toggle_min(p.bitmap, prev_min);
    }
}

// Vertex v joins slot `pos`.
__device__ __forceinline__ void join_slot(const RoundParams& p, uint64_t pos, uint32_t hi, uint32_t v) {
    join_block(p, pos, hi, v);
    p.slot_of[v] = (int32_t)pos;
}

// Incremental refinement: vertex v's new block goes by `name`.  Where its old
// one went by another, both names are tainted (RoundParams::taint).
__device__ __forceinline__ void note_old_name(const RoundParams& p, int64_t v, uint32_t name) {
    const uint32_t old = p.old_min[p.keep_old[v]];
    p.old_name[v] = old;
    if (old == name) return;
    atomicOr(&p.taint[old >> 5], 1u << (old & 31));
    atomicOr(&p.taint[name >> 5], 1u << (name & 31));
}

__device__ __forceinline__ bool vertex_active(const RoundParams& p, int64_t v) {
    return !p.vmask || ((p.vmask[v >> 5] >> (v & 31)) & 1u);
}

// A graph in level-0 mode (serving: admitted this step) keys its vertices by
// (graph, label) and ignores its edges.
__device__ __forceinline__ bool vertex_level0(const RoundParams& p, int64_t v) {
    return p.gmode && p.gmode[p.vgraph[v]] == 1;
}

// In a frozen block (RoundParams::frozen): it keeps its previous block.
__device__ __forceinline__ bool vertex_frozen(const RoundParams& p, int64_t v) {
    return p.frozen && ((load_level(p.frozen + (v >> 5)) >> (v & 31)) & 1u);
}

// Active and refining by signature (not in level-0 mode, not frozen).
__device__ __forceinline__ bool vertex_refines(const RoundParams& p, int64_t v) {
    return vertex_active(p, v) && !vertex_level0(p, v) && !vertex_frozen(p, v);
}

// In multi-graph runs a representative must belong to the same graph.
__device__ __forceinline__ bool same_graph(const RoundParams& p, int64_t a, int64_t b) {
    return !p.vgraph || p.vgraph[a] == p.vgraph[b];
}

// Probe the block table from *pos.  Returns 0 when v inserted a new key,
// 1 with *rep set when a slot with our tag was found (a signature compare
// decides), 2 when the probe limit was hit.
__device__ __forceinline__ int probe_table(const RoundParams& p, uint64_t* pos_io, uint32_t hi, uint32_t v,
                                           uint32_t* rep) {
    uint64_t pos = *pos_io;
    for (int it = 0; it < kProbeLimit; ++it) {
        uint64_t cur = volatile_load(&p.table[pos]);
        if ((uint32_t)(cur >> 56) != p.epoch) {
            const uint64_t want = ((uint64_t)hi << 32) | kSingleBit | v;
            const uint64_t old = atomicCAS(reinterpret_cast<unsigned long long*>(&p.table[pos]),
                                           (unsigned long long)cur, (unsigned long long)want);
            if (old == cur) {
                p.slot_of[v] = (int32_t)pos;
                toggle_min(p.bitmap, v);
                *pos_io = pos;
                return 0;
            }
            cur = old;
            if ((uint32_t)(cur >> 56) != p.epoch) continue;
        }
        if ((uint32_t)(cur >> 32) == hi) {
            *rep = (uint32_t)cur & kVertexMask;
            *pos_io = pos;
            return 1;
        }
        pos = (pos + 1) & p.mask;
    }
    return 2;
}
// ---- tiles of consecutive edges
// Source vertex of edge e, the largest v with row[v] <= e, by a whole warp: each
// step reads 32 offsets at once and keeps one of 33 parts (a search by halves is
// 20 dependent loads, 12 us, that a tile's CTA has to wait for).
__device__ __forceinline__ int64_t edge_source(const int64_t* row, int64_t n, int64_t e) {
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = n;  // row[lo] <= e < row[hi]
    while (hi - lo > 1) {
        const int64_t at = lo + (lane + 1) * (hi - lo) / 33;
        const int c = __popc(__ballot_sync(kFull, row[at] <= e));  // ascending over the lanes
        const int64_t below = __shfl_sync(kFull, (long long)at, max(c - 1, 0));
        const int64_t above = __shfl_sync(kFull, (long long)at, min(c, 31));
        if (c > 0) lo = below;
        if (c < 32) hi = above;
    }
    return lo;
}

// Sources of the edges [e0, e1) of a tile of kThreads x kPer edges, for a whole
// CTA of kThreads: s_src[i] = source of edge e0 + i.  Two warps search for the
// first and last edge's source, every vertex between them that has edges marks
// its first one, and a running maximum fills the rest (a search per edge reads
// a dozen offsets each).  Where the sources lie far apart -- runs of edgeless
// vertices, or many more vertices than edges -- the walk over the vertices between
// them is longer than the searches (one CTA's 0.23 us per 256 vertices): beyond
// kWalkPerEdge vertices per edge of the tile every edge searches between the two.
// 10^7 vertices with 5 x 10^6 edgeless ones in one run, 10^6 edges: backward
// 4073 -> 1053 us, summary 9162 -> 183 us.  Begins and ends with a barrier.
constexpr int kWalkPerEdge = 8;

// (a call of its own, so that the tiles that walk keep their registers)
template <int kThreads, int kPer>
__device__ __noinline__ void search_sources(const int64_t* row, uint32_t span, int64_t lo, int64_t e0, int64_t e1,
                                            int32_t* s_src) {
    static_assert(kPer % 2 == 0, "a thread's searches run two by two");
#pragma unroll 1
    for (int u = 0; u < kPer; u += 2) {
        const int i = u * kThreads + threadIdx.x;
        const int64_t ea = min(e0 + i, e1 - 1), eb = min(e0 + i + kThreads, e1 - 1);
        uint32_t a = 0u, b = 0u;
        for (uint32_t step = 1u << (31 - __clz(span)); step > 0u; step >>= 1) {
            const bool in_a = step <= span - a && row[a + step] <= ea, in_b = step <= span - b && row[b + step] <= eb;
            if (in_a) a += step;
            if (in_b) b += step;
        }
        s_src[i] = (int32_t)(lo + a);
        s_src[i + kThreads] = (int32_t)(lo + b);
    }
}

template <int kThreads, int kPer>
__device__ __forceinline__ void tile_sources(int64_t n, const int64_t* row, int64_t e0, int64_t e1, int32_t* s_src) {
    __shared__ int64_t s_v[2];
    __shared__ int32_t s_warp[kThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();
    if (warp < 2) {
        const int64_t v = edge_source(row, n, warp ? e1 - 1 : e0);
        if (lane == 0) s_v[warp] = v;
    }
    for (int i = tid; i < kThreads * kPer; i += kThreads) s_src[i] = -1;
    __syncthreads();
    const int64_t lo = s_v[0];
    const uint32_t span = (uint32_t)(s_v[1] - lo);
    if (span > (uint32_t)(kWalkPerEdge * kThreads * kPer)) {  // uniform over the CTA
        search_sources<kThreads, kPer>(row + lo, span, lo, e0, e1, s_src);
        __syncthreads();
        return;
    }
    for (int64_t v = lo + tid; v <= s_v[1]; v += kThreads) {
        const int64_t a = row[v], b = row[v + 1];
        if (b > a && b > e0 && a < e1) s_src[max(a, e0) - e0] = (int32_t)v;
    }
    __syncthreads();
    int32_t run[kPer], mx = -1;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        mx = max(mx, s_src[tid * kPer + u]);
        run[u] = mx;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(kFull, mx, o);
        if (lane >= o) mx = max(mx, y);
    }
    if (lane == 31) s_warp[warp] = mx;
    int32_t before = __shfl_up_sync(kFull, mx, 1);
    if (lane == 0) before = -1;
    __syncthreads();
    for (int i = 0; i < warp; ++i) before = max(before, s_warp[i]);
#pragma unroll
    for (int u = 0; u < kPer; ++u) s_src[tid * kPer + u] = max(run[u], before);
    __syncthreads();
}

}  // namespace kb
