// Summary graph of a partition pair (Sec. "Graph Summaries for Bisimulation":
// one summary vertex per block, a labelled summary edge from block b to block c
// when the vertices of b have an edge with that label into c).
//
// Every edge v -> w with label l gives the triple (lsrc[x], l, ldst[y]), with
// x -> y the edge in the processed direction.  The distinct triples are found
// with one open-addressing table of 16-byte slots, each a triple and its smallest
// edge index so far, read and replaced whole (128-bit load and CAS; the triple
// itself is the key, so no compare against a representative is needed).  Output
// order is first occurrence in the edge list: the edges that hold their triple's
// slot are marked in an edge bitmap, ranked by a popcount prefix scan, and every
// first edge writes its triple at its rank.
//
//   insert  CTA tiles of kSumTile consecutive edges; lanes of a warp holding the
//           same triple elect the lowest (its edge comes first) to look it up.
//           A slot that has the triple with a smaller edge needs no atomic, and
//           a warp's new triples are marked with one: its edges share a bitmap
//           word.  An edge that loses its slot to a smaller one is unmarked;
//   emit    the edges again, in order: every first occurrence re-derives its
//           triple and writes it at its rank (consecutive writes per warp).
//
// What bounds the insert: one random sector per edge for the table and one for
// the target's block.  2 x 10^7 power-law edges: 1739 us (and 167 us of marking)
// with a separate array of smallest edges, a CAS per edge and a pass over the
// table that marked them, 893 us this way.  Two or four looks at the table
// in flight per lane, or tiles of 2,048 edges, lose to the registers they take
// (1465, 2057 and 1413 against 1351 us for the whole call).
#include <cuda_runtime.h>

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {
namespace {

constexpr int kSumThreads = 256;
constexpr int kSumPer = 4;
constexpr int kSumTile = kSumThreads * kSumPer;

// Atomic 128-bit compare-and-swap of a 16-byte aligned slot (lo at the lower
// address); returns the slot's previous contents.
__device__ __forceinline__ void cas128(unsigned long long* slot, unsigned long long clo, unsigned long long chi,
                                       unsigned long long nlo, unsigned long long nhi, unsigned long long* olo,
                                       unsigned long long* ohi) {
    asm volatile(
        "{\n\t.reg .b128 d, c, n;\n\t"
        "mov.b128 c, {%2, %3};\n\t"
        "mov.b128 n, {%4, %5};\n\t"
        "atom.global.cas.b128 d, [%6], c, n;\n\t"
        "mov.b128 {%0, %1}, d;\n\t}"
        : "=l"(*olo), "=l"(*ohi)
        : "l"(clo), "l"(chi), "l"(nlo), "l"(nhi), "l"(slot)
        : "memory");
}

__device__ __forceinline__ void load128(const unsigned long long* slot, unsigned long long* lo, unsigned long long* hi) {
    asm volatile(
        "{\n\t.reg .b128 d;\n\t"
        "ld.relaxed.gpu.global.b128 d, [%2];\n\t"
        "mov.b128 {%0, %1}, d;\n\t}"
        : "=l"(*lo), "=l"(*hi)
        : "l"(slot)
        : "memory");
}

__global__ void __launch_bounds__(kSumThreads, 6) summary_insert_kernel(const SummaryParams q) {
    __shared__ int32_t s_src[kSumTile];
    if (q.ctr->err) return;  // malformed offsets or ids: nothing may be indexed by them
    const int lane = threadIdx.x & 31;
    const int64_t e0 = (int64_t)blockIdx.x * kSumTile;
    int32_t w[kSumPer];
    uint32_t l[kSumPer];
#pragma unroll
    for (int u = 0; u < kSumPer; ++u) {
        const int64_t e = e0 + u * kSumThreads + threadIdx.x;
        w[u] = e < q.m ? __ldcs(q.col + e) : 0;
        l[u] = q.lab && e < q.m ? (uint32_t)__ldcs(q.lab + e) : 0u;
    }
    tile_sources<kSumThreads, kSumPer>(q.n, q.row, e0, min(q.m, e0 + kSumTile), s_src);
    int32_t bx[kSumPer], by[kSumPer];
#pragma unroll
    for (int u = 0; u < kSumPer; ++u) {
        const int i = u * kSumThreads + threadIdx.x;
        const int64_t v = max(s_src[i], 0);  // past the last edge: any vertex
        bx[u] = __ldg(q.lsrc + (q.dir == 0 ? v : (int64_t)w[u]));
        by[u] = __ldg(q.ldst + (q.dir == 0 ? (int64_t)w[u] : v));
    }
#pragma unroll
    for (int u = 0; u < kSumPer; ++u) {
        const int64_t e = e0 + u * kSumThreads + threadIdx.x;
        const bool ok = e < q.m;
        // a slot: label and source block, then the edge's index + 1 and the
        // target block; all zero while empty
        const unsigned long long lo = ((unsigned long long)l[u] << 32) | (uint32_t)bx[u];
        const unsigned long long hi = ((unsigned long long)(e + 1) << 32) | (uint32_t)by[u];
        // lanes with the same triple: the lowest one (smallest edge) goes
        const unsigned grp = __match_any_sync(kFull, lo) & __match_any_sync(kFull, (unsigned)by[u]) &
                             __ballot_sync(kFull, ok);
        bool mark = false;
        if (ok && lane == __ffs(grp) - 1) {
            uint64_t pos = mix64(lo ^ mix64((unsigned long long)(uint32_t)by[u] ^ 0x2545f4914f6cdd1dULL)) & q.mask;
            int it = 0;
            for (; it < kProbeLimit; ++it) {
                unsigned long long* slot = q.table + 2 * pos;
                unsigned long long slo, shi;
                load128(slot, &slo, &shi);
                bool mine = slo == lo && (uint32_t)shi == (uint32_t)hi && shi != 0ull;
                if (shi != 0ull && !mine) {
                    pos = (pos + 1) & q.mask;
                    continue;
                }
                if (mine && shi <= hi) break;  // an earlier edge has it
                unsigned long long olo, ohi;
                cas128(slot, slo, shi, lo, hi, &olo, &ohi);
                if (olo == slo && ohi == shi) {
                    mark = true;
                    if (mine) {  // a later edge had it
                        const uint64_t old = (shi >> 32) - 1;
                        atomicXor(&q.bitmap[old >> 5], 1u << (old & 31));
                    }
                    break;
                }
            }
            if (it == kProbeLimit) set_error(q.ctr, kErrTableFull);
        }
        const unsigned marks = __ballot_sync(kFull, mark);  // e & 31 == lane: tiles and warps are 32-aligned
        if (lane == 0 && marks) atomicXor(&q.bitmap[e >> 5], marks);
    }
}

// Walks the edges again in their order: a first occurrence re-derives its
// triple and writes it at its rank, so a warp's writes are consecutive.
__global__ void __launch_bounds__(kSumThreads) summary_emit_kernel(const SummaryParams q, const uint32_t* prefix,
                                                                   int32_t* out_src, int32_t* out_label,
                                                                   int32_t* out_dst) {
    __shared__ int32_t s_src[kSumTile];
    const int lane = threadIdx.x & 31;
    const int64_t e0 = (int64_t)blockIdx.x * kSumTile;
    uint32_t words[kSumPer];
    int32_t w[kSumPer];
    uint32_t l[kSumPer];
    bool any = false;
#pragma unroll
    for (int u = 0; u < kSumPer; ++u) {
        const int64_t e = e0 + u * kSumThreads + threadIdx.x;
        words[u] = e < q.m ? q.bitmap[e >> 5] : 0u;
        const bool first = (words[u] >> lane) & 1u;
        w[u] = first ? __ldcs(q.col + e) : 0;
        l[u] = first && q.lab ? (uint32_t)__ldcs(q.lab + e) : 0u;
        any |= words[u] != 0u;
    }
    if (!__syncthreads_or(any)) return;
    tile_sources<kSumThreads, kSumPer>(q.n, q.row, e0, min(q.m, e0 + kSumTile), s_src);
#pragma unroll
    for (int u = 0; u < kSumPer; ++u) {
        if (!((words[u] >> lane) & 1u)) continue;
        const int i = u * kSumThreads + threadIdx.x;
        const int64_t v = s_src[i];
        const uint32_t r = prefix[(e0 + i) >> 5] + (uint32_t)__popc(words[u] & ((1u << lane) - 1u));
        out_src[r] = __ldg(q.lsrc + (q.dir == 0 ? v : (int64_t)w[u]));
        out_label[r] = (int32_t)l[u];
        out_dst[r] = __ldg(q.ldst + (q.dir == 0 ? (int64_t)w[u] : v));
    }
}

}  // namespace

void launch_summary_insert(const SummaryParams& q, cudaStream_t s) {
    if (q.m <= 0) return;
    summary_insert_kernel<<<(unsigned)((q.m + kSumTile - 1) / kSumTile), kSumThreads, 0, s>>>(q);
}

void launch_summary_emit(const SummaryParams& q, const uint32_t* prefix, int32_t* out_src, int32_t* out_label,
                         int32_t* out_dst, cudaStream_t s) {
    if (q.m <= 0) return;
    summary_emit_kernel<<<(unsigned)((q.m + kSumTile - 1) / kSumTile), kSumThreads, 0, s>>>(q, prefix, out_src, out_label,
                                                                                          out_dst);
}

}  // namespace kb
