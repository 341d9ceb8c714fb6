// Device bodies of the hub, renumbering, dirty and freeze passes of a round,
// shared by their kernels (kb_kernels.cu) and the fused kernel of small graphs
// (kb_fused.cu).
#pragma once

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {

// ----------------------------------------------------------------------------
// Hub chunks: kChunk edges of one hub per CTA.  Chunk-local dedup in shared
// memory, then the chunk's distinct pairs go into the hub's global set; pairs
// new to the hub (the CAS that placed them found the slot empty) are counted
// and summed into its hash.
// ----------------------------------------------------------------------------
// Whether hub h takes part in the exact path this round.
__device__ __forceinline__ bool hub_is_exact(const RoundParams& p, int h) {
    return p.hub_exact ? p.hub_exact[h] != 0u : vertex_refines(p, p.hub_v[h]);
}

template <int kChunk>
struct HubChunkSmem {
    uint64_t pair[kChunk];
    uint64_t fresh[kChunk];
    uint32_t set[2 * kChunk];  // the chunk's dedup set
    int nuniq, nnew;
    uint64_t accsum;
};

// (a caller that goes on to use sm waits for the CTA)
template <int kChunk, int kThreads>
__device__ __forceinline__ void hub_chunk(const RoundParams& p, HubChunkSmem<kChunk>& sm, int64_t c) {
    constexpr int kHubSetCap = 2 * kChunk;
    uint64_t *s_pair = sm.pair, *s_new = sm.fresh;
    uint32_t* s_set = sm.set;

    const int tid = threadIdx.x;
    // every thread reads the chunk's hub and packed extent (one broadcast word each)
    const int h = p.chunk_hub[c];
    const uint64_t ext = p.chunk_ext[c];
    const int64_t e0 = (int64_t)(ext >> 16);
    const int E = (int)(ext & 0xffffu);
    if (!hub_is_exact(p, h)) return;  // uniform over the CTA
    if (tid == 0) {
        sm.nuniq = 0;
        sm.nnew = 0;
        sm.accsum = 0ull;
    }
    for (int i = tid; i < kHubSetCap; i += kThreads) s_set[i] = 0u;

    for (int base = 0; base < E; base += 4 * kThreads) {
        int32_t w[4], l[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int le = base + u * kThreads + tid;
            if (le < E) {
                w[u] = __ldcs(p.col + e0 + le);
                l[u] = p.lab ? __ldcs(p.lab + e0 + le) : 0;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int le = base + u * kThreads + tid;
            if (le < E) b[u] = gather_block(p, w[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int le = base + u * kThreads + tid;
            if (le < E) s_pair[le] = pack_pair(l[u], (uint32_t)w[u], b[u]);
        }
    }
    __syncthreads();

    // chunk-local distinct pairs, compacted into s_new with one shared atomic per warp
    for (int base = 0; base < E; base += kThreads) {
        const int le = base + tid;
        bool isu = false;
        uint64_t pr = 0;
        if (le < E) {
            pr = s_pair[le];
            uint32_t slot = set_slot(pr, 0u) & (kHubSetCap - 1);
            while (true) {
                uint32_t cur = s_set[slot];
                if (cur == 0u) {
                    const uint32_t old = atomicCAS(&s_set[slot], 0u, (uint32_t)(le + 1));
                    if (old == 0u) {
                        isu = true;
                        break;
                    }
                    cur = old;
                }
                if (s_pair[(int)cur - 1] == pr) break;
                slot = (slot + 1) & (kHubSetCap - 1);
            }
        }
        const unsigned b = __ballot_sync(kFull, isu);
        int wbase = 0;
        if ((tid & 31) == 0 && b) wbase = atomicAdd(&sm.nuniq, __popc(b));
        wbase = __shfl_sync(kFull, wbase, 0);
        if (isu) s_new[wbase + __popc(b & ((1u << (tid & 31)) - 1u))] = pr;
    }
    __syncthreads();

    // insert into the hub's global set
    const int nu = sm.nuniq;
    uint64_t* gset = p.hub_sets + p.hub_set_off[h];
    const uint64_t gcap = (uint64_t)(p.hub_set_off[h + 1] - p.hub_set_off[h]);
    uint64_t lacc = 0;
    uint32_t lnew = 0;
    // Up to kChunk / kThreads pairs per thread: the first probe of every
    // pair is a CAS issued before waiting on any, then the rare collisions are
    // finished one by one.
    constexpr int kPer = kChunk / kThreads;
    uint64_t prs[kPer], slots[kPer], olds[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * kThreads;
        if (i < nu) {
            prs[u] = s_new[i];
            slots[u] = hub_set_home(prs[u], gcap);
            olds[u] = atomicCAS(reinterpret_cast<unsigned long long*>(&gset[slots[u]]),
                                (unsigned long long)kEmptyPair, (unsigned long long)prs[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = tid + u * kThreads;
        if (i >= nu) continue;
        const uint64_t pr = prs[u];
        uint64_t slot = slots[u], old = olds[u];
        bool placed = false;
        for (uint64_t t = 0; t < gcap; ++t) {
            if (old == kEmptyPair) {
                lacc += pair_mix(pr);
                ++lnew;
                placed = true;
                break;
            }
            if (old == pr) {
                placed = true;
                break;
            }
            slot = slot + 1 == gcap ? 0 : slot + 1;
            old = atomicCAS(reinterpret_cast<unsigned long long*>(&gset[slot]), (unsigned long long)kEmptyPair,
                            (unsigned long long)pr);
        }
        // sets hold 1.5 x the hub's degree: a pair that finds no slot means
        // corrupted sets (reported as a device check failure)
        if (!placed) set_error(p.ctr, kErrHubSet);
    }
    // CTA sums of the pairs new to the hub: hash and count
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lacc += __shfl_xor_sync(kFull, lacc, o);
        lnew += __shfl_xor_sync(kFull, lnew, o);
    }
    if ((tid & 31) == 0 && lnew) {
        atomicAdd(reinterpret_cast<unsigned long long*>(&sm.accsum), (unsigned long long)lacc);
        atomicAdd(&sm.nnew, (int)lnew);
    }
    __syncthreads();
    if (tid == 0 && sm.nnew) {
        atomicAdd(&p.hub_cnt[h], (uint32_t)sm.nnew);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.hub_acc[h]), (unsigned long long)sm.accsum);
    }
}

__device__ __forceinline__ bool hub_set_contains(const uint64_t* gset, uint64_t gcap, uint64_t pr) {
    uint64_t slot = hub_set_home(pr, gcap);
    for (uint64_t t = 0; t < gcap; ++t) {
        const uint64_t cur = gset[slot];
        if (cur == pr) return true;
        if (cur == kEmptyPair) return false;
        slot = slot + 1 == gcap ? 0 : slot + 1;
    }
    return false;
}

// ----------------------------------------------------------------------------
// Hub keys: one CTA per hub finds or inserts the hub's key, comparing the full
// signature against the representative of any slot with a matching tag.
// ----------------------------------------------------------------------------
struct HubFinalSmem {
    uint64_t pair[kMaxHubThreshold];
    uint32_t set[2 * kMaxHubThreshold];
    int kind;
    uint32_t rep;
    uint64_t pos;
    int ok, cnt_r;
};

// (a caller that goes on to use sm waits for the CTA)
__device__ __forceinline__ void hub_final(const RoundParams& p, HubFinalSmem& sm, int h) {
    uint64_t* s_pair = sm.pair;
    uint32_t* s_set = sm.set;
    const int tid = threadIdx.x;
    const int32_t v = p.hub_v[h];
    if (!vertex_refines(p, v)) return;
    if (!hub_is_exact(p, h)) {  // its sketch says that it is alone in its new block
        if (tid == 0) toggle_min(p.bitmap, (uint32_t)v);
        return;
    }
    const int32_t own = own_of(p, v);
    const uint32_t cnt = p.hub_cnt[h];
    const uint64_t hv = vertex_hash(own, cnt, p.hub_acc[h], p.hash_mode);
    const uint32_t hi = table_hi(hv, p.epoch);
    const uint64_t* gset = p.hub_sets + p.hub_set_off[h];
    const uint64_t gcap = (uint64_t)(p.hub_set_off[h + 1] - p.hub_set_off[h]);
    if (tid == 0) sm.pos = hv & p.mask;

    for (int iter = 0; iter < kProbeLimit; ++iter) {
        __syncthreads();
        if (tid == 0) {
            uint64_t pos = sm.pos;
            uint32_t rep = 0;
            sm.kind = probe_table(p, &pos, hi, (uint32_t)v, &rep);
            sm.pos = pos;
            sm.rep = rep;
            sm.ok = 1;
            sm.cnt_r = 0;
        }
        __syncthreads();
        const int kind = sm.kind;
        if (kind == 0) return;
        if (kind == 2) {
            if (tid == 0) set_error(p.ctr, kErrTableFull);
            return;
        }
        const uint32_t r = sm.rep;
        bool ok = same_graph(p, r, v) && (own_of(p, r) == own);
        const int64_t rb = p.row[r], re = p.row[r + 1];
        if (ok && re - rb > p.hub_threshold) {
            // representative is a hub: compare distinct counts, then look its
            // distinct pairs (the filled slots of its set) up in our set
            int lo = 0, hi2 = p.n_hubs;
            while (hi2 - lo > 1) { int mid = (lo + hi2) >> 1; if (p.hub_v[mid] <= (int32_t)r) lo = mid; else hi2 = mid; }
            const uint32_t cnt_r = p.hub_cnt[lo];
            ok = (cnt_r == cnt);
            if (ok) {
                // its set holds exactly its distinct pairs (and empty slots)
                const uint64_t* rset = p.hub_sets + p.hub_set_off[lo];
                const int64_t rcap = p.hub_set_off[lo + 1] - p.hub_set_off[lo];
                bool all = true;
                for (int64_t i = tid; i < rcap && all; i += kHubFinalThreads) {
                    const uint64_t pr = rset[i];
                    if (pr != kEmptyPair && !hub_set_contains(gset, gcap, pr)) all = false;
                }
                if (!all) sm.ok = 0;
            } else if (tid == 0) {
                sm.ok = 0;
            }
        } else if (ok) {
            // representative is a small vertex: derive its pairs, count its
            // distinct pairs in shared memory and look each up in our set
            const int d = (int)(re - rb);
            for (int i = tid; i < 2 * kMaxHubThreshold; i += kHubFinalThreads) s_set[i] = 0u;
            __syncthreads();
            bool all = true;
            for (int i = tid; i < d; i += kHubFinalThreads) {
                const int32_t w = __ldg(p.col + rb + i);
                const int32_t l = p.lab ? __ldg(p.lab + rb + i) : 0;
                const uint64_t pr = pack_pair(l, (uint32_t)w, gather_block(p, w));
                s_pair[i] = pr;
                if (!hub_set_contains(gset, gcap, pr)) all = false;
            }
            __syncthreads();
            for (int i = tid; i < d; i += kHubFinalThreads) {
                const uint64_t pr = s_pair[i];
                uint32_t slot = set_slot(pr, 0u) & (2 * kMaxHubThreshold - 1);
                while (true) {
                    uint32_t cur = s_set[slot];
                    if (cur == 0u) {
                        const uint32_t old = atomicCAS(&s_set[slot], 0u, (uint32_t)(i + 1));
                        if (old == 0u) { atomicAdd(&sm.cnt_r, 1); break; }
                        cur = old;
                    }
                    if (s_pair[(int)cur - 1] == pr) break;
                    slot = (slot + 1) & (2 * kMaxHubThreshold - 1);
                }
            }
            if (!all) sm.ok = 0;
            __syncthreads();
            if (tid == 0 && (uint32_t)sm.cnt_r != cnt) sm.ok = 0;
        } else if (tid == 0) {
            sm.ok = 0;
        }
        __syncthreads();
        if (tid == 0) {
            if (sm.ok) {
                join_slot(p, sm.pos, hi, (uint32_t)v);
                sm.kind = 0;
            } else {
                sm.pos = (sm.pos + 1) & p.mask;
            }
        }
        __syncthreads();
        if (sm.kind == 0) return;
    }
    if (tid == 0) set_error(p.ctr, kErrTableFull);
}

// The smallest member of v's block when v is not that member.
__device__ __forceinline__ uint32_t block_min(const RoundParams& p, int64_t v) {
    const uint32_t sl = (uint32_t)p.slot_of[v];
    if (sl & 0x80000000u) return (uint32_t)p.emin[(sl & 0x7fffffffu) % (uint32_t)p.n];
    return (uint32_t)p.table[(uint64_t)sl & p.mask] & kVertexMask;
}

// Canonical ids of a stratified round with frozen blocks (RoundParams::minof;
// one graph, or several at once): assign_kernel's work with every lane of a warp
// on one bitmap word (a warp-uniform loop), so that the moved vertices (re-keyed
// vertices whose smallest block member changed) leave as one word per warp.
// Frozen vertices keep minof, and their blocks keep their shared marks (the
// freeze pass carries them over); the mark of a re-keyed block comes from the
// vertex that inserted its table entry (RoundParams::joined).  moved may be null
// (the starting level); mark, when given, is cleared for the dirty pass.
// Vertices in strides of the grid; begins and ends with a barrier of the CTA.
__device__ __forceinline__ void assign_frozen(const RoundParams& p, const uint2* rank, int32_t* out, uint32_t* moved,
                                              uint32_t* mark, uint32_t* s_moved) {
    if (threadIdx.x == 0) *s_moved = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    uint32_t n_moved = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < p.n; base += stride) {
        const int64_t v = base + lane;
        bool mv = false;
        const uint32_t joined = p.joined[base >> 5];
        if (v < p.n) {
            const bool fz = vertex_frozen(p, v);
            // a frozen block keeps its members and smallest member; a graph that
            // computed its level 0 here has no previous level
            const bool history = fz || (moved && !vertex_level0(p, v));
            const uint32_t before = history ? p.minof[v] : 0u;
            uint32_t mn = (uint32_t)v;
            if (fz)
                mn = before;
            else if (!((p.bitmap[v >> 5] >> (v & 31)) & 1u))
                mn = block_min(p, v);
            if ((int64_t)mn >= p.n) mn = (uint32_t)v;  // only after a reported device error
            if ((joined >> lane) & 1u) atomicOr(&p.shared[mn >> 5], 1u << (mn & 31));
            const uint2 rw = rank[mn >> 5];
            uint32_t b = rw.x + __popc(rw.y & ((1u << (mn & 31)) - 1u));
            if (!p.lgraph) {
                out[v] = (int32_t)b;
            } else {
                const int32_t g = p.lgraph[v];
                b -= p.gbase_cur[g];
                if (!p.gout)
                    out[v] = (int32_t)b;
                else if (p.gout[g])
                    p.gout[g][v - p.voff[g]] = (int32_t)b;
            }
            // the locality order's copy of the level names every block by its
            // smallest member too
            if (!history || before != mn) {
                mv = history;
                if (p.perm) p.gat[p.perm[v]] = (int32_t)mn;
                p.minof[v] = mn;
            }
        }
        if (joined) {  // read by every lane above
            __syncwarp();
            if (lane == 0) p.joined[base >> 5] = 0u;
        }
        if (mark && lane == 0) mark[base >> 5] = 0u;
        if (moved) {
            const unsigned w = __ballot_sync(kFull, mv);
            if (p.perm) {
                if (mv) atomicOr(&moved[p.perm[v] >> 5], 1u << (p.perm[v] & 31));
            } else if (lane == 0) {
                moved[base >> 5] = w;
            }
            n_moved += __popc(w);
        }
    }
    if (!moved) return;  // uniform over the grid
    if (lane == 0 && n_moved) atomicAdd(s_moved, n_moved);
    __syncthreads();
    if (threadIdx.x == 0 && *s_moved)
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctr->moved), (unsigned long long)*s_moved);
}

// Vertices of bitmap word w that are neither alone in their block nor
// edgeless (and exist).
__device__ __forceinline__ uint32_t candidate_word(const uint32_t* bitmap, const uint32_t* shared,
                                                   const uint32_t* edgeless, int64_t w, int64_t n) {
    uint32_t c = ~(bitmap[w] & ~shared[w]);
    if (edgeless) c &= ~edgeless[w];
    const int64_t first = w * 32;
    if (first + 32 > n) c &= n > first ? ((1u << (uint32_t)(n - first)) - 1u) : 0u;
    return c;
}

// A warp takes up to 32 consecutive bitmap words (1024 vertices; fewer while
// the graph is too small to fill the chip with that) and deals their candidate
// vertices (candidate_word) to its lanes, 32 at a time: *v receives
// the vertex of rank r among them, or -1.  excl / c are this lane's word's
// exclusive candidate prefix and candidate bits.
__device__ __forceinline__ int64_t dealt_vertex(int64_t w0, uint32_t excl, uint32_t c, int r, int total) {
    int src = 0;  // the last lane with excl <= r, by halves
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
        if ((int)__shfl_sync(kFull, excl, src + step) <= r) src += step;
    uint32_t x = __shfl_sync(kFull, c, src);
    int k = r - (int)__shfl_sync(kFull, excl, src);  // the set bit of rank k in x, by halves
    int at = 0;
#pragma unroll
    for (int width = 16; width > 0; width >>= 1) {
        const int low = __popc(x & ((1u << width) - 1u));
        if (k >= low) {
            k -= low;
            x >>= width;
            at += width;
        }
    }
    return r < total ? (w0 + src) * 32 + at : -1;
}

// A level-i block X can split in the next round only if one of its members
// has an edge to a vertex whose smallest block member changed this round.
// For X to split, two members u, v with equal signatures over level i-1 must
// differ over level i: u has an edge (label l) into a level-i part C of some
// level-(i-1) block B, and v has its label-l edges into B only outside C, in
// another part C'.  So B split, and C or C' lacks B's smallest member: the
// members of that part changed smallest member, and u or v has an edge to
// one of them.  Mark (by the block's name) the blocks that hold such a member; a
// vertex with more than max_scan edges marks its block unread.  When more
// than an eighth of the vertices moved, nothing is scanned: the freeze pass
// then takes every block as marked.
__device__ __forceinline__ bool few_moved(const RoundParams& p) { return p.ctr->moved * 8 <= p.n; }

// (One warp's words, from w0 on.)
__device__ __forceinline__ void dirty_blocks(const RoundParams& p, const uint32_t* edgeless, const uint32_t* moved,
                                             int32_t max_scan, uint32_t* mark, int per_warp, const uint8_t* gactive,
                                             int64_t w0) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (p.n >> 5) + 1;
    if (w0 >= nw) return;  // uniform over the warp
    const uint32_t c =
        lane < per_warp && w0 + lane < nw ? candidate_word(p.bitmap, p.shared, edgeless, w0 + lane, p.n) : 0u;
    uint32_t incl = __popc(c);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = (int)__shfl_sync(kFull, incl, 31);
    const uint32_t excl = incl - __popc(c);
    for (int t = 0; t < total; t += 32) {
        const int64_t v = dealt_vertex(w0, excl, c, t + lane, total);
        if (v < 0 || (gactive && !gactive[p.lgraph[v]])) continue;
        const int64_t a = p.row[v], e_end = p.row[v + 1];
        // a graph that computed its level 0 here has no history: all dirty
        bool dirty = e_end - a > max_scan || vertex_level0(p, v);
        for (int64_t e0 = a; e0 < e_end && !dirty; e0 += 4) {
            int32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = e0 + u < e_end ? (__ldg(p.col + e0 + u) & 0x7fffffff) : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (w[u] >= 0 && ((moved[w[u] >> 5] >> (w[u] & 31)) & 1u)) dirty = true;
        }
        if (dirty) {
            const uint32_t b = p.minof[v];
            const uint32_t mb = 1u << (b & 31);
            if (!(__ldcg(mark + (b >> 5)) & mb)) atomicOr(&mark[b >> 5], mb);
        }
    }
}

// The frozen blocks of the next round (see FreezePass).  frozen_min holds the
// minima of frozen blocks, and the shared marks of exactly those minima are
// kept for the next round (their blocks keep their members; the others are
// marked afresh).  A warp takes up to 32 bitmap words and deals the candidates
// whose block it must look up to its lanes, as dirty_blocks_kernel does.
// (One warp's words, from w0 on; s_clean: a word per lane of this warp; s_on:
// frozen vertices and refining mid and medium vertices and hubs of the CTA.)
__device__ __forceinline__ void freeze_clean(const FreezePass& f, uint32_t* s_clean, uint32_t* s_on, int64_t w0) {
    Counters* ctr = f.ctr;
    const int64_t n = f.n;
    const int per_warp = f.per_warp;
    const uint32_t* bitmap = f.bitmap;
    uint32_t* shared = f.shared;
    const uint32_t* edgeless = f.edgeless;
    const uint32_t* mark = f.mark;
    const int lane = threadIdx.x & 31;
    const int64_t nw = (n >> 5) + 1;
    if (w0 >= nw) return;  // uniform over the warp
    if (mark && ctr->moved * 8 > n) mark = nullptr;  // the dirty pass scanned nothing
    const int64_t w = w0 + lane;
    const bool own = lane < per_warp && w < nw;
    uint32_t b = 0, sh = 0, e = 0, c = 0;
    if (own) {
        b = bitmap[w];
        sh = shared[w];
        e = edgeless ? edgeless[w] : 0u;
        c = mark ? candidate_word(bitmap, shared, edgeless, w, n) : 0u;
    }
    uint32_t off = 0;  // vertices of graphs that stopped
    if (f.gactive && own) {
        const int64_t first = w * 32, last = min(n, first + 32) - 1;
        if (first <= last) {
            const int32_t g0 = f.vgraph[first], g1 = f.vgraph[last];
            if (g0 == g1) {
                off = f.gactive[g0] ? 0u : 0xffffffffu;
            } else {
                for (int64_t v = first; v <= last; ++v)
                    if (!f.gactive[f.vgraph[v]]) off |= 1u << (v - first);
            }
        }
        c &= ~off;
    }
    if (f.gmode && edgeless) {
        // serving: a graph that computed its level 0 in this step has not had
        // its edgeless blocks formed by a round yet
        for (int j = 0; j < 32; ++j) {
            const uint32_t ej = __shfl_sync(kFull, e, j);
            const int64_t vj = (w0 + j) * 32 + lane;
            const bool lvl0 = vj < n && ((ej >> lane) & 1u) && f.gmode[f.vgraph[vj]] == 1;
            const uint32_t drop = __ballot_sync(kFull, lvl0);
            if (lane == j) {
                e &= ~drop;
                // their blocks are looked up (and marked dirty) instead; without
                // marks nothing but singletons is frozen
                if (mark) c |= drop & ~(b & ~sh);
            }
        }
    }
    s_clean[lane] = 0u;
    __syncwarp();
    uint32_t incl = __popc(c);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = (int)__shfl_sync(kFull, incl, 31);
    const uint32_t excl = incl - __popc(c);
    for (int t = 0; t < total; t += 32) {
        const int64_t v = dealt_vertex(w0, excl, c, t + lane, total);
        if (v < 0) continue;
        const uint32_t l = (uint32_t)f.names[v];
        if (!((mark[l >> 5] >> (l & 31)) & 1u)) atomicOr(&s_clean[(v >> 5) - w0], 1u << (v & 31));
    }
    __syncwarp();
    if (own) {
        // no bit past the last vertex survives (rank scans count whole words)
        const uint32_t valid = w * 32 + 32 <= n ? 0xffffffffu : (n > w * 32 ? (1u << (uint32_t)(n - w * 32)) - 1u : 0u);
        const uint32_t single = b & ~sh & valid;
        const uint32_t cl = s_clean[lane];
        const uint32_t keep = (e | cl | off) & valid;
        const uint32_t fz = single | keep;
        const uint32_t fm = single | (b & keep);
        f.frozen[w] = fz;
        f.frozen_min[w] = fm;
        shared[w] = sh & fm;
        if (f.moved_clear) f.moved_clear[w] = 0u;
        if (fz) atomicAdd(&s_on[0], (uint32_t)__popc(fz));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t on = f.classes[k] ? f.classes[k][w] & ~fz : 0u;
            if (on) atomicAdd(&s_on[1 + k], (uint32_t)__popc(on));
        }
    }
    __syncwarp();  // s_clean is read no more
}


// A CTA's counts of freeze_clean (after a barrier).
__device__ __forceinline__ void add_frozen(Counters* ctr, const uint32_t* s_on) {
    if (threadIdx.x < 4 && s_on[threadIdx.x]) {
        int64_t* dst = threadIdx.x == 0 ? &ctr->frozen : &ctr->class_on[threadIdx.x - 1];
        atomicAdd(reinterpret_cast<unsigned long long*>(dst), (unsigned long long)s_on[threadIdx.x]);
    }
}

}  // namespace kb
