// Hubs that are alone in their key.  Most hubs of a power-law graph share their
// signature with no other vertex, and finding that out does not need their
// exact pair sets (hub_chunk_kernel), only a sketch that equal sets share:
//
//   * kSketchMins minima: a pair's mix picks one of them and lowers it;
//   * a bitmap of kSketchBits bits with one bit per pair.
//
// Both ignore duplicates and the order of the edges, so no set is kept, and both
// are merged over a hub's chunks with atomics that mostly find nothing to do.
// A hub with more bits set than any vertex that is not a hub has distinct pairs
// this round can share its signature with hubs only, and those have the same
// sketch.  Such a hub whose (own block,
// sketch) hash no other one has is alone in its new block.  All others --
// hubs with few distinct pairs, hubs whose hash occurs twice (equal sketches, or
// a collision) -- go on to the exact sets and the full signature compare, so the
// sketch never decides that two vertices are equal.
//
// The exact sets cost a returning CAS on 12 bytes of set per edge for every pair
// that is new to its chunk; the sketch is bound by the gather of the neighbours'
// blocks.  1.1 x 10^8 hub edges of the 2 x 10^8-edge graph: exact sets, their
// clearing and the hub keys 1848 us, sketches (408 us, 821 with one chunk per
// CTA) and what is left for the exact path 543 us.  On the first round of 10^8
// edges in one block every hub has few distinct pairs: there the sketches add
// 140 us to 500, and the second round gets back 400.
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {
namespace {

constexpr int kSketchMins = 32;
constexpr int kSketchBits = 8192;
constexpr int kSketchWords = kSketchMins + kSketchBits / 32;
constexpr int kPerLane = kSketchWords / 32;
static_assert(kSketchMins == 32 && kSketchWords % 32 == 0, "one minimum per lane");
static_assert(sizeof(uint32_t) * kSketchWords <= sizeof(uint64_t) * 3 * kSketchMinThreshold / 2,
              "a hub's sketch lies in the memory of its exact set");

__device__ __forceinline__ uint32_t* sketch_of(const RoundParams& p, int h) {
    return reinterpret_cast<uint32_t*>(p.hub_sets + p.hub_set_off[h]);
}

// Word i of an empty sketch.
__device__ __forceinline__ uint32_t empty_word(int i) { return i < kSketchMins ? 0xffffffffu : 0u; }

__global__ void __launch_bounds__(256) sketch_clear_kernel(const RoundParams p) {
    const int lane = threadIdx.x & 31;
    const int h = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (h >= p.n_hubs || !vertex_refines(p, p.hub_v[h])) return;
    uint32_t* s = sketch_of(p, h);
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) s[i * 32 + lane] = empty_word(i * 32 + lane);
}

// Merge a CTA's sketch of (part of) hub h into the hub's.
__device__ __forceinline__ void merge_sketch(const RoundParams& p, int h, const uint32_t* mine) {
    uint32_t* s = sketch_of(p, h);
    for (int i = threadIdx.x; i < kSketchWords; i += kHubThreads) {
        const uint32_t x = mine[i], seen = __ldcg(s + i);
        if (i < kSketchMins) {
            if (x < seen) atomicMin(s + i, x);
        } else if (x & ~seen) {
            atomicOr(s + i, x);
        }
    }
}

// kSketchChunks chunks per CTA; consecutive ones are mostly of one hub, so that
// clearing and merging the CTA's sketch is rare.
constexpr int kSketchChunks = 4;
__global__ void __launch_bounds__(kHubThreads) hub_sketch_kernel(const RoundParams p, int64_t total_chunks) {
    __shared__ uint32_t s_sketch[kSketchWords];
    constexpr int U = 4;
    const int tid = threadIdx.x;
    const int64_t c0 = (int64_t)blockIdx.x * kSketchChunks, c1 = min(total_chunks, c0 + kSketchChunks);
    int cur = -1;  // the hub in s_sketch
    for (int64_t c = c0; c < c1; ++c) {
        const int h = p.chunk_hub[c];
        const uint64_t ext = p.chunk_ext[c];
        const int64_t e0 = (int64_t)(ext >> 16);
        const int E = (int)(ext & 0xffffu);
        if (!vertex_refines(p, p.hub_v[h])) continue;  // uniform over the CTA
        if (h != cur) {
            if (cur >= 0) {
                __syncthreads();
                merge_sketch(p, cur, s_sketch);
                __syncthreads();
            }
            for (int i = tid; i < kSketchWords; i += kHubThreads) s_sketch[i] = empty_word(i);
            cur = h;
            __syncthreads();
        }
        for (int base = 0; base < E; base += U * kHubThreads) {
            int32_t w[U], l[U], b[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int le = base + u * kHubThreads + tid;
                w[u] = l[u] = 0;
                if (le < E) {
                    w[u] = __ldcs(p.col + e0 + le);
                    if (p.lab) l[u] = __ldcs(p.lab + e0 + le);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (base + u * kHubThreads + tid < E) b[u] = gather_block(p, w[u]);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (base + u * kHubThreads + tid >= E) continue;
                const uint64_t x = pair_mix(pack_pair(l[u], (uint32_t)w[u], b[u]));
                const uint32_t m = (uint32_t)(x >> 32), bit = (uint32_t)(x >> 5) & (kSketchBits - 1);
                uint32_t* mn = s_sketch + (x & (kSketchMins - 1));
                if (m < *mn) atomicMin(mn, m);
                uint32_t* word = s_sketch + kSketchMins + (bit >> 5);
                if (!((*word >> (bit & 31)) & 1u)) atomicOr(word, 1u << (bit & 31));
            }
        }
    }
    if (cur < 0) return;  // uniform over the CTA
    __syncthreads();
    merge_sketch(p, cur, s_sketch);
}

// Send hub h to the exact path (once): its chunks join the list.
__device__ __forceinline__ void make_exact(const RoundParams& p, int h) {
    const int lane = threadIdx.x & 31;
    int first = -1;
    const int64_t c0 = p.hub_chunk_off[h];
    const int nc = (int)(p.hub_chunk_off[h + 1] - c0);
    if (lane == 0 && atomicExch(&p.hub_exact[h], 1u) == 0u) first = (int)atomicAdd(&p.ctr->exact_chunks, (uint32_t)nc);
    first = __shfl_sync(kFull, first, 0);
    if (first < 0) return;
    for (int i = lane; i < nc; i += 32) p.exact_list[first + i] = (int32_t)(c0 + i);
}

// A warp per hub: its sketch's hash, and the hubs that need their exact set.
__global__ void __launch_bounds__(256) hub_alone_kernel(const RoundParams p) {
    const int lane = threadIdx.x & 31;
    const int h = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (h >= p.n_hubs) return;  // uniform over the warp
    const int32_t v = p.hub_v[h];
    if (!vertex_refines(p, v)) return;
    const uint32_t* s = sketch_of(p, h);
    uint64_t acc = 0;
    uint32_t bits = 0;
#pragma unroll
    for (int i = 0; i < kPerLane; ++i) {
        const int k = i * 32 + lane;
        const uint32_t x = s[k];
        if (k >= kSketchMins) bits += __popc(x);
        acc += mix64(((uint64_t)(k + 1) << 32) | x);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(kFull, (unsigned long long)acc, o);
        bits += __shfl_xor_sync(kFull, bits, o);
    }
    // distinct pairs of a vertex that is not a hub: counted by the medium CTA
    // kernel, at most the degree for those of the other kernels
    const uint32_t most = max(p.ctr->most_pairs, (uint32_t)max(p.mid_max, min(p.med_split, p.hub_threshold)));
    if (bits <= most) {
        make_exact(p, h);
        return;
    }
    // hubs with equal hashes meet in a table of hub indices
    const uint64_t hash = vertex_hash(own_of(p, v), bits, acc, 0);
    int other = -1;
    if (lane == 0) {
        p.hub_acc[h] = hash;
        __threadfence();  // the hash before the index that leads to it
        uint32_t slot = (uint32_t)hash & p.hub_twin_mask;
        while (true) {  // at most half full
            const uint32_t old = atomicCAS(&p.hub_twin[slot], 0u, (uint32_t)h + 1u);
            if (old == 0u) break;
            __threadfence();  // the index before the hash that it leads to: a stale one would hide a twin
            if (volatile_load(&p.hub_acc[old - 1u]) == hash) {
                other = (int)old - 1;
                break;
            }
            slot = (slot + 1) & p.hub_twin_mask;
        }
    }
    other = __shfl_sync(kFull, other, 0);
    if (other >= 0) {
        make_exact(p, h);
        make_exact(p, other);
    }
}

}  // namespace

void launch_hub_sketch(const RoundParams& p, int64_t total_chunks, cudaStream_t s) {
    if (p.n_hubs <= 0 || total_chunks <= 0) return;
    cudaMemsetAsync(p.hub_exact, 0, sizeof(uint32_t) * (size_t)p.n_hubs, s);
    cudaMemsetAsync(p.hub_twin, 0, sizeof(uint32_t) * ((size_t)p.hub_twin_mask + 1), s);
    cudaMemsetAsync(&p.ctr->exact_chunks, 0, sizeof(uint32_t), s);
    const unsigned warps = (unsigned)(((int64_t)p.n_hubs * 32 + 255) / 256);
    sketch_clear_kernel<<<warps, 256, 0, s>>>(p);
    hub_sketch_kernel<<<(unsigned)((total_chunks + kSketchChunks - 1) / kSketchChunks), kHubThreads, 0, s>>>(p, total_chunks);
    hub_alone_kernel<<<warps, 256, 0, s>>>(p);
}

}  // namespace kb
