// Kernel for the vertices with at most kSmallDegree edges in the processed
// direction (the large majority of vertices in power-law graphs), and for
// level 0 (no edges; the key is the vertex label or a starting partition).
//
// One lane per vertex: it loads four neighbours, labels and blocks at a time,
// keeps its distinct pairs (set semantics, Def. "signature") in a column of
// shared memory, sums their mixes, probes the table and, on a tag match, derives
// the representative's pairs and looks each up among its own (the full
// signature compare).  Representatives are small vertices too, as larger ones
// enter the table after this kernel; where the classes share a launch
// (kb_fused.cu, kb_keys.cu) they may be of any degree, so the compare has no limit.  Neighbouring lanes read neighbouring edges, so
// the lines that one lane's load brings serve the others from L1.
//
// What bounds it: random 4-8 byte accesses (blocks, table, representatives) and
// the instructions around them.  One edge per lane, with vertices packed into
// windows of 32 edges by warp scans and matches, issued 730 warp instructions
// per window of about six vertices and filled 55-61% of the issue slots; a lane
// per vertex needs about a fifth of them and has four loads in flight per lane.
// Round 1: 2871 -> 895 us with 10^8 power-law edges (and 207 us more in the mid
// kernel, which takes 9 to 32 edges), 2733 -> 1385 us with 2 x 10^8 (+ 415 us),
// 1795 -> 733 us on a batch of 5.5 x 10^7 Erdos-Renyi edges (+ 160 us).  Vertices
// of up to 16 edges in this kernel lose (7311 against 6938 us for a whole call
// when this was tried): their pairs take the L1 that the random loads need.
//
// Hot keys.  In power-law graphs millions of vertices share a key (all
// edgeless vertices with the same label, all vertices with one edge to the
// same hub block), and a global atomic per vertex on the same word serialises.
// So joins are aggregated per CTA: a shared map keyed by the table slot (or by
// the own block of an empty signature) keeps the smallest joining vertex, and
// the CTA applies one global atomicMin per key when it finishes.  New-block
// owners toggle their minimum bits once per window (one atomicXor per bitmap
// word).  The XOR toggling of block minima is order independent, so the
// aggregation leaves the result unchanged.
#pragma once

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {

constexpr int kSmallThreads = 256;
constexpr int kSmallMinBlocks = 5;  // 48 registers, nothing spills; 6 CTAs per SM spill and cost a tenth of a whole call
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int64_t kResidentWarps = 152 * kSmallMinBlocks * kSmallWarps;  // warps the chip holds at once
// Joins a CTA can aggregate (1 x its vertices at the default task size; a
// join that finds no room goes to global memory at once).  Shared memory comes
// out of the SM's L1, which the many outstanding random loads need, so no more;
// 512 and 256 entries lose 2% and 7% of a whole call to hot keys.
constexpr int kMapBits = 10;
constexpr int kMapCap = 1 << kMapBits;
constexpr uint64_t kMapEmpty = ~0ull;
// Longest task: packed windows keep a vertex's place in its task in 16 bits.
constexpr int32_t kMaxTaskVerts = 65536;
constexpr uint64_t kEmptyKeyBit = 1ull << 63;  // map key of an empty-signature join: bit 63 | own

// Task of a round in which few vertices refine: four times as long, so that fewer
// warps walk windows that are nearly empty, up to the 4096 vertices that
// launch_small_round takes there; a caller's longer task stays as it is.
__host__ __device__ constexpr int32_t sparse_task(int32_t verts) {
    return verts >= 4096 ? verts : (verts * 4 < 4096 ? verts * 4 : 4096);
}
static_assert(sparse_task(kMaxTaskVerts) == kMaxTaskVerts && sparse_task(4095) == 4096 && sparse_task(32) == 128,
              "a task never grows past what its windows can address");

struct JoinMap {
    uint64_t key[kMapCap];
    uint32_t hi[kMapCap];
    uint32_t vmin[kMapCap];
};

// Record that v joins `key`; false when the map has no room (the caller then
// joins globally right away).
__device__ __forceinline__ bool map_join(JoinMap& M, uint64_t key, uint32_t hi, uint32_t v) {
    uint32_t slot = ((uint32_t)key * 2654435761u ^ (uint32_t)(key >> 63)) >> (32 - kMapBits);
    for (int t = 0; t < 32; ++t) {
        uint64_t cur = M.key[slot];
        if (cur == kMapEmpty) {
            cur = atomicCAS(reinterpret_cast<unsigned long long*>(&M.key[slot]), (unsigned long long)kMapEmpty,
                            (unsigned long long)key);
            if (cur == kMapEmpty) {
                M.hi[slot] = hi;
                cur = key;
            }
        }
        if (cur == key) {
            atomicMin(&M.vmin[slot], v);
            return true;
        }
        slot = (slot + 1) & (kMapCap - 1);
    }
    return false;
}

// A CTA's smallest joining vertex of one key, with minimum toggles.  Edgeless
// blocks (vertices with the key (own block, empty set), grouped by the own
// block exactly) keep their smallest vertex of this round in emin[own]; entries
// of earlier rounds carry a larger high word and lose every atomicMin.
__device__ __forceinline__ void flush_join(const RoundParams& p, uint64_t key, uint32_t hi, uint32_t v) {
    if (key & kEmptyKeyBit) {
        const int32_t own = (int32_t)(uint32_t)key;
        const uint64_t want = ((uint64_t)p.ehigh << 32) | v;
        const uint64_t seen = volatile_load(&p.emin[own]);
        if ((uint32_t)(seen >> 32) == p.ehigh && (uint32_t)seen <= v) return;  // minima only decrease
        const uint64_t old = atomicMin(reinterpret_cast<unsigned long long*>(&p.emin[own]), (unsigned long long)want);
        if ((uint32_t)(old >> 32) != p.ehigh) {
            toggle_min(p.bitmap, v);
        } else if (v < (uint32_t)old) {
            toggle_min(p.bitmap, v);
            toggle_min(p.bitmap, (uint32_t)old);
        }
    } else {
        join_block(p, key, hi, v);
    }
}

template <bool kLevel0, bool kCompact>
struct SmallSmem {
    uint64_t pairs[kLevel0 ? 1 : kSmallDegree][kLevel0 ? 1 : kSmallThreads];
    JoinMap map;
    unsigned long long l0[kLevel0 ? 256 : 1];
    uint16_t off[kSmallWarps][kCompact ? 32 : 1];
};

// A CTA's share of the round: its warps take the task first and, with kLoop, first +
// stride, .. of p.warp_verts vertices each (a kernel with a warp per task has no
// loop: it would cost it registers, and spills).  Begins without and ends with all warps past
// the join map (a caller that goes on to use sm waits for the CTA).
template <bool kLevel0, bool kCompact, bool kLoop>
__device__ __forceinline__ void small_body(const RoundParams& p, SmallSmem<kLevel0, kCompact>& sm, int64_t first,
                                           int64_t stride) {
    JoinMap& M = sm.map;
    unsigned long long* s_l0 = sm.l0;
    const int lane = threadIdx.x & 31;
    uint64_t* pairs = &sm.pairs[0][kLevel0 ? 0 : threadIdx.x];  // this lane's distinct pairs, kSmallThreads apart
    for (int i = threadIdx.x; i < kMapCap; i += kSmallThreads) {
        M.key[i] = kMapEmpty;
        M.vmin[i] = 0xffffffffu;
    }
    if (kLevel0)
        for (int i = threadIdx.x; i < 256; i += kSmallThreads) s_l0[i] = ~0ull;
    __syncthreads();

    for (int64_t vb = first * p.warp_verts; vb < p.n; vb += stride * p.warp_verts) {
        const int64_t ve = min(p.n, vb + p.warp_verts);

        // A window holds up to 32 vertices of the task, one per lane: consecutive
        // ones, or (kCompact, when many vertices are frozen) the next ones that
        // refine this round among the next kLook, so that frozen and inactive
        // vertices take no lane.  The next window is picked, and its row offsets
        // and own blocks loaded, before the current one works.
        constexpr int kLook = kCompact ? 128 : 32;
        const int span = (int)(ve - vb);  // task vertices (at most kMaxTaskVerts)
        int pf_off = -1;  // next window: this lane's vertex as an offset from vb (-1: none)
        int pf_next = 0;  // and where the window after it starts
        int64_t pf_a = 0;
        int32_t pf_d = 0, pf_own = 0;
        auto pick = [&](int c) {
            if (!kCompact) {  // the next 32 vertices
                pf_off = c + lane < span ? c + lane : -1;
                pf_next = c + 32;
            } else {  // the next 32 that refine, among the next kLook
                unsigned bk[kLook / 32];
#pragma unroll
                for (int k = 0; k < kLook / 32; ++k) {
                    const int u = c + 32 * k + lane;
                    bk[k] = __ballot_sync(kFull, u < span && vertex_active(p, vb + u) && !vertex_frozen(p, vb + u));
                }
                // every candidate hands its offset to the lane of its rank
                uint16_t* offs = sm.off[threadIdx.x >> 5];
                int total = 0;
#pragma unroll
                for (int k = 0; k < kLook / 32; ++k) {
                    const int r = total + __popc(bk[k] & ((1u << lane) - 1u));
                    if (((bk[k] >> lane) & 1u) && r < 32) offs[r] = (uint16_t)(c + 32 * k + lane);
                    total += __popc(bk[k]);
                }
                __syncwarp();
                const int o = offs[lane], last = offs[31];
                __syncwarp();
                pf_off = lane < total ? o : -1;
                pf_next = total > 32 ? last + 1 : c + kLook;
            }
            if (pf_off >= 0) {
                const int64_t pv = vb + pf_off;
                pf_own = (!kLevel0 && p.own_key) ? p.own_key[pv] : (p.prev ? p.prev[pv] : 0);
                if (!kLevel0) {
                    pf_a = p.row[pv];
                    pf_d = (int32_t)min(p.row[pv + 1] - pf_a, (int64_t)0x7fffffff);
                }
            }
        };
        pick(0);
        for (int wc = 0; wc < span;) {
            const int64_t v0 = vb + wc;  // first vertex of a window of consecutive vertices (not kCompact)
            const int64_t v = vb + pf_off;  // meaningful when this lane has a vertex
            const int64_t a = pf_a;
            int d = pf_d;
            int32_t own = pf_own;
            bool l0 = kLevel0;
            bool pending = pf_off >= 0 && (kCompact || (vertex_active(p, v) && !vertex_frozen(p, v)));
            if (!kLevel0 && pending && vertex_level0(p, v)) {
                l0 = true;
                own = p.vlab ? p.vlab[v] : 0;
            }
            if (kLevel0 || l0) d = 0;
            pending = pending && d <= p.small_max;
            wc = pf_next;
            if (wc < span) pick(wc);

            // this lane's distinct pairs and the sum of their mixes, four edges at a time
            int cnt = 0;
            uint64_t acc = 0;
            if (!kLevel0) {
                const int de = pending ? d : 0;
                for (int k = 0; __any_sync(kFull, k < de); k += 4) {
                    int32_t w[4], l[4], b[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        w[u] = l[u] = 0;
                        if (k + u < de) {
                            w[u] = __ldg(p.col + a + k + u);
                            if (p.lab) l[u] = __ldg(p.lab + a + k + u);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (k + u < de) b[u] = gather_block(p, w[u]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (k + u >= de) break;
                        const uint64_t x = pack_pair(l[u], (uint32_t)w[u], b[u]);
                        bool seen = false;
                        for (int t = 0; t < cnt; ++t) seen |= pairs[t * kSmallThreads] == x;
                        if (!seen) {
                            pairs[cnt * kSmallThreads] = x;
                            acc += pair_mix(x);
                            ++cnt;
                        }
                    }
                }
            }

            bool inserted = false;
            uint64_t pos = 0;
            uint32_t hi = 0;
            if (pending) {
                if (!l0 && d == 0) {
                    // (own block, empty set): grouped by the own block exactly
                    const uint64_t key = kEmptyKeyBit | (uint32_t)own;
                    if (!map_join(M, key, 0u, (uint32_t)v)) flush_join(p, key, 0u, (uint32_t)v);
                    p.slot_of[v] = (int32_t)(0x80000000u | (uint32_t)own);
                    pending = false;
                } else {
                    // at level 0 of a multi-graph run the key is (graph, label)
                    const uint32_t c2 = (l0 && p.vgraph) ? (uint32_t)p.vgraph[v] : (uint32_t)cnt;
                    const uint64_t h = vertex_hash(own, c2, acc, p.hash_mode);
                    pos = h & p.mask;
                    hi = table_hi(h, p.epoch);
                }
            }
            // Level 0 of one graph: the key is the label alone, so a slot that a
            // lane of this CTA found (or claimed) for a label serves later lanes
            // with the same label without a probe or a compare (a direct-mapped
            // cache of (label, slot) words).
            uint32_t l0c = 0;
            bool resolved = false;
            if (kLevel0 && !batched(p)) {
                l0c = ((uint32_t)own * 2654435761u) >> 24;
                if (pending) {
                    const unsigned long long e = s_l0[l0c];
                    if (e != ~0ull && (uint32_t)(e >> 32) == (uint32_t)own) {
                        pos = (uint32_t)e;
                        if (!map_join(M, pos, hi, (uint32_t)v)) flush_join(p, pos, hi, (uint32_t)v);
                        p.slot_of[v] = (int32_t)pos;
                        pending = false;
                    }
                }
            }
            for (int probes = 0; __any_sync(kFull, pending); ++probes) {
                if (!pending) continue;
                if (probes > kProbeLimit) {
                    set_error(p.ctr, kErrTableFull);
                    pending = false;
                    continue;
                }
                const uint64_t cur = volatile_load(&p.table[pos]);
                if ((uint32_t)(cur >> 56) != p.epoch) {
                    const unsigned long long want = ((uint64_t)hi << 32) | kSingleBit | (uint32_t)v;
                    if (atomicCAS(reinterpret_cast<unsigned long long*>(&p.table[pos]), (unsigned long long)cur, want) != cur)
                        continue;  // taken
                    p.slot_of[v] = (int32_t)pos;
                    inserted = true;
                    pending = false;
                    continue;
                }
                bool eq = false;
                if ((uint32_t)(cur >> 32) == hi) {
                    // full signature compare with the representative: its key and its
                    // row offsets are loaded together
                    const uint32_t rep = (uint32_t)cur & kVertexMask;
                    const int32_t* keys = (l0 && !kLevel0) ? p.vlab : ((!kLevel0 && p.own_key) ? p.own_key : p.prev);
                    const int32_t rkey = keys ? load_level(keys + rep) : 0;
                    int64_t rb = 0, re = 0;
                    if (!l0) {
                        rb = p.row[rep];
                        re = p.row[(int64_t)rep + 1];
                    }
                    eq = same_graph(p, rep, v) && rkey == own;
                    if (!l0 && eq) {
                        unsigned found = 0;
                        for (int64_t e0 = rb; e0 < re && eq; e0 += 4) {
                            uint64_t x[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                x[u] = 0;
                                if (e0 + u < re) {
                                    const int32_t w = __ldg(p.col + e0 + u);
                                    const int32_t l = p.lab ? __ldg(p.lab + e0 + u) : 0;
                                    x[u] = pack_pair(l, (uint32_t)w, gather_block(p, w));
                                }
                            }
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (e0 + u >= re) break;
                                unsigned hit = 0;
                                for (int t = 0; t < cnt; ++t)
                                    if (pairs[t * kSmallThreads] == x[u]) hit = 1u << t;
                                if (!hit) eq = false;
                                found |= hit;
                            }
                        }
                        if (found != (1u << cnt) - 1u) eq = false;
                    }
                }
                if (eq) {
                    if (!map_join(M, pos, hi, (uint32_t)v)) flush_join(p, pos, hi, (uint32_t)v);
                    p.slot_of[v] = (int32_t)pos;
                    pending = false;
                    resolved = true;
                } else {
                    pos = (pos + 1) & p.mask;
                }
            }
            if (kLevel0 && !batched(p) && (resolved || inserted))
                s_l0[l0c] = ((unsigned long long)(uint32_t)own << 32) | (uint32_t)pos;
            // new-block owners of this window: one atomicXor per bitmap word (the
            // window's vertices lie in at most kLook / 32 + 1 words)
            if (!kCompact) {
                const uint32_t sh = (uint32_t)(v0 & 31);
                const int64_t w0 = v0 >> 5;
                const unsigned m = __ballot_sync(kFull, inserted);
                if (lane == 0 && m) {
                    atomicXor(&p.bitmap[w0], m << sh);
                    if (sh && (m >> (32 - sh))) atomicXor(&p.bitmap[w0 + 1], m >> (32 - sh));
                }
            } else {
                unsigned todo = __ballot_sync(kFull, inserted);
                while (todo) {
                    const int64_t w = __shfl_sync(kFull, (long long)(v >> 5), __ffs(todo) - 1);
                    const bool mine = inserted && (v >> 5) == w;
                    const unsigned bits = __reduce_or_sync(kFull, mine ? 1u << (v & 31) : 0u);
                    if (lane == 0) atomicXor(&p.bitmap[w], bits);
                    todo &= ~__ballot_sync(kFull, mine);
                }
            }
        }
        if (!kLoop) break;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kMapCap; i += kSmallThreads) {
        const uint64_t key = M.key[i];
        if (key != kMapEmpty) flush_join(p, key, M.hi[i], M.vmin[i]);
    }
}

}  // namespace kb
