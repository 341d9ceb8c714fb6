// Incremental refinement after edge insertions and deletions
// (kb_refine_update).  The paper leaves incremental k-bisimulation as future
// work (Sec. "Conclusion and Future Work": one changed edge can change ids in
// every later round).  Here a round re-keys only a work set W and keeps the
// old grouping of every other vertex:
//
//   dirty(i)  = changed edge lists, vertices whose block changed as a set at
//               level i-1 ("moved"), and vertices with an edge to a moved one;
//   W(i)      = every vertex of a level-(i-1) block that holds a dirty vertex.
//
// A vertex moved when its old and its new block differ as sets.  Both go by
// their smallest member: a vertex whose two names differ taints both, and the
// vertices of tainted blocks moved (a block without a tainted name neither lost
// nor gained a member).  So only vertices that changed name cost an atomic; the
// ranges of new ids per old block and of old ids per new block that this
// replaces were four arrays to fill and four atomics per vertex (115 of 463 us
// of kernels in an update of 10^6 vertices).
//
// Keys hold the own previous block, so a level-i block lies inside one
// level-(i-1) block: blocks are either inside W or outside it.  Outside W,
// edge lists, neighbour blocks and own blocks are unchanged as sets, so two
// such vertices are equivalent now exactly when they were before.  Every
// level is then renumbered canonically in full.
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {
namespace {

constexpr int kT = 256;
constexpr int kPer = 4;
constexpr int kTile = kT * kPer;

__device__ __forceinline__ bool bit(const uint32_t* b, int64_t v) { return (b[v >> 5] >> (v & 31)) & 1u; }

__device__ __forceinline__ void set_bit(uint32_t* b, int64_t v) {
    const uint32_t m = 1u << (v & 31);
    if (!(__ldcg(b + (v >> 5)) & m)) atomicOr(&b[v >> 5], m);
}

int grid_of(int64_t items, int threads) {
    const int64_t b = (items + threads - 1) / threads;
    return (int)(b < 1 ? 1 : (b > 152 * 64 ? 152 * 64 : b));
}

// Sum of one value per thread of a 256-thread CTA, added to *out.
__device__ __forceinline__ void add_cta(unsigned long long c, int64_t* out) {
    __shared__ unsigned long long s_sum[kT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < kT / 32; ++w) t += s_sum[w];
        if (t) atomicAdd(reinterpret_cast<unsigned long long*>(out), t);
    }
}

// dirty[v] |= moved[y] over every edge v -> y of the processed CSR, in tiles of
// consecutive edges (two searches give a tile's source range).
__device__ __forceinline__ int64_t source_in(const int64_t* row, int64_t lo, int64_t hi, int64_t e) {
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (row[mid] <= e) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(kT) dirty_from_moved_kernel(int64_t n, int64_t m, const int64_t* row,
                                                              const int32_t* col, const uint32_t* moved,
                                                              uint32_t* dirty) {
    __shared__ int64_t s_v[2];
    const int64_t tiles = (m + kTile - 1) / kTile;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t e0 = t * kTile;
        bool hit[kPer], any = false;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int64_t e = e0 + u * kT + threadIdx.x;
            hit[u] = e < m && bit(moved, __ldcs(col + e) & 0x7fffffff);
            any |= hit[u];
        }
        if (!__syncthreads_or(any)) continue;  // most tiles have no edge to a moved vertex
        if (threadIdx.x < 64) {
            const int64_t v = edge_source(row, n, threadIdx.x < 32 ? e0 : min(m, e0 + kTile) - 1);
            if ((threadIdx.x & 31) == 0) s_v[threadIdx.x >> 5] = v;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kPer; ++u)
            if (hit[u]) set_bit(dirty, source_in(row, s_v[0], s_v[1], e0 + u * kT + threadIdx.x));
        __syncthreads();  // s_v is no longer read
    }
}

// flag bit b for every level-(i-1) block b holding a dirty vertex (in any of
// the three bitmaps; dirty may be null)
__global__ void flag_blocks_kernel(int64_t n, const int32_t* prev, const uint32_t* changed, const uint32_t* moved,
                                   const uint32_t* dirty, uint32_t* flag) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t nw = (n + 31) >> 5;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nw; w += stride) {
        uint32_t x = changed[w] | moved[w] | (dirty ? dirty[w] : 0u);
        for (; x; x &= x - 1) {
            const int64_t v = w * 32 + __ffs(x) - 1;
            if (v < n) set_bit(flag, prev[v]);
        }
    }
}

// W = vertices of flagged blocks, one bitmap word per warp; |W| into ctr->work_set
__global__ void __launch_bounds__(kT) work_set_kernel(int64_t n, const int32_t* prev, const uint32_t* flag,
                                                      uint32_t* wmask, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {
        const int64_t v = base + threadIdx.x;  // blockDim is a multiple of 32: a warp covers one word
        const bool in = v < n && bit(flag, prev[v]);
        const unsigned b = __ballot_sync(kFull, in);
        if ((threadIdx.x & 31) == 0 && (v >> 5) <= ((n - 1) >> 5)) wmask[v >> 5] = b;
        c += in;
    }
    add_cta(c, &ctr->work_set);
}

// old_min[b] = smallest vertex of block b of `level`
__global__ void old_min_kernel(int64_t n, const int32_t* level, uint32_t* old_min) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        uint32_t* m = old_min + level[v];
        if (__ldcg(m) > (uint32_t)v) atomicMin(m, (uint32_t)v);
    }
}

// the kept blocks' smallest members into the bitmap of block minima
__global__ void keep_bits_kernel(int64_t n, const uint32_t* wmask, const int32_t* old, const uint32_t* old_min,
                                 uint32_t* bitmap) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {
        const int64_t v = base + threadIdx.x;
        const bool mn = v < n && !bit(wmask, v) && old_min[old[v]] == (uint32_t)v;
        const unsigned b = __ballot_sync(kFull, mn);
        if ((threadIdx.x & 31) == 0 && b) atomicOr(&bitmap[v >> 5], b);
    }
}

// moved: a vertex of W (wmask; null: all) whose old block's name is tainted;
// counted in ctr->moved
__global__ void __launch_bounds__(kT) moved_mark_kernel(int64_t n, const uint32_t* wmask, const uint32_t* old_name,
                                                        const uint32_t* taint, uint32_t* moved, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {
        const int64_t v = base + threadIdx.x;
        const bool mv = v < n && (!wmask || bit(wmask, v)) && bit(taint, old_name[v]);
        const unsigned w = __ballot_sync(kFull, mv);
        if ((threadIdx.x & 31) == 0 && (v >> 5) <= ((n - 1) >> 5)) moved[v >> 5] = w;
        c += mv;
    }
    add_cta(c, &ctr->moved);
}

// Every vertex is in one block now, named by vertex 0.
__global__ void one_block_kernel(const RoundParams p, int32_t* out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < p.n; v += stride) {
        note_old_name(p, v, 0u);
        out[v] = 0;
    }
}

__global__ void check_ids_kernel(int64_t count, int64_t n, const int32_t* a, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride)
        bad |= a[i] < 0 || (int64_t)a[i] >= n;
    if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(&ctr->err, kErrInvalid);
}

// The changed vertices' bits, and their blocks of `level` into touched.  Ids out
// of [0, n) are reported (those of level by check_ids_kernel) and skipped.
__global__ void set_changed_kernel(int64_t n, int64_t count, const int32_t* ids, const int32_t* level, uint32_t* bits,
                                   uint32_t* touched, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
        const int32_t v = ids[i];
        if (v < 0 || (int64_t)v >= n) {
            atomicOr(&ctr->err, kErrInvalid);
            continue;
        }
        atomicOr(&bits[v >> 5], 1u << (v & 31));
        const int32_t b = level[v];
        if (b >= 0 && (int64_t)b < n) atomicOr(&touched[b >> 5], 1u << (b & 31));
    }
}

// ctr->work_set += vertices whose block of `level` is touched.
__global__ void __launch_bounds__(kT) touched_size_kernel(int64_t n, const int32_t* level, const uint32_t* touched,
                                                          Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int32_t b = level[v];
        c += b >= 0 && (int64_t)b < n && bit(touched, b);
    }
    add_cta(c, &ctr->work_set);
}

int few(int64_t n) { return std::min(grid_of(n, kT), 1216); }  // one atomic per CTA

}  // namespace

void launch_dirty_from_moved(int64_t n, int64_t m, const int64_t* row, const int32_t* col, const uint32_t* moved,
                             uint32_t* dirty, cudaStream_t s) {
    if (n <= 0 || m <= 0) return;
    cudaMemsetAsync(dirty, 0, sizeof(uint32_t) * (size_t)((n >> 5) + 1), s);
    const int64_t tiles = (m + kTile - 1) / kTile;
    dirty_from_moved_kernel<<<grid_of(tiles * kT, kT), kT, 0, s>>>(n, m, row, col, moved, dirty);
}

void launch_work_set(int64_t n, const int32_t* prev, const uint32_t* changed, const uint32_t* moved,
                     const uint32_t* dirty, uint32_t* flag, uint32_t* wmask, Counters* ctr, cudaStream_t s) {
    if (n <= 0) return;
    cudaMemsetAsync(flag, 0, sizeof(uint32_t) * (size_t)((n >> 5) + 1), s);
    cudaMemsetAsync(&ctr->work_set, 0, sizeof(int64_t), s);
    flag_blocks_kernel<<<grid_of((n + 31) >> 5, kT), kT, 0, s>>>(n, prev, changed, moved, dirty, flag);
    work_set_kernel<<<few(n), kT, 0, s>>>(n, prev, flag, wmask, ctr);
}

void launch_old_min(int64_t n, const int32_t* level, uint32_t* old_min, cudaStream_t s) {
    if (n <= 0) return;
    cudaMemsetAsync(old_min, 0xff, sizeof(uint32_t) * (size_t)n, s);
    old_min_kernel<<<grid_of(n, kT), kT, 0, s>>>(n, level, old_min);
}

void launch_keep_bits(int64_t n, const uint32_t* wmask, const int32_t* old, const uint32_t* old_min, uint32_t* bitmap,
                      cudaStream_t s) {
    if (n > 0) keep_bits_kernel<<<grid_of(n, kT), kT, 0, s>>>(n, wmask, old, old_min, bitmap);
}

void launch_moved(int64_t n, const uint32_t* wmask, const uint32_t* old_name, const uint32_t* taint, uint32_t* moved,
                  Counters* ctr, cudaStream_t s) {
    if (n > 0) moved_mark_kernel<<<few(n), kT, 0, s>>>(n, wmask, old_name, taint, moved, ctr);
}

void launch_one_block(const RoundParams& p, int32_t* out, cudaStream_t s) {
    if (p.n > 0) one_block_kernel<<<grid_of(p.n, kT), kT, 0, s>>>(p, out);
}

void launch_check_ids(int64_t count, int64_t n, const int32_t* a, Counters* ctr, cudaStream_t s) {
    if (count > 0) check_ids_kernel<<<grid_of(count, kT), kT, 0, s>>>(count, n, a, ctr);
}

void launch_changed(int64_t n, int64_t count, const int32_t* ids, const int32_t* level, uint32_t* bits,
                    uint32_t* touched, Counters* ctr, cudaStream_t s) {
    if (count > 0) set_changed_kernel<<<grid_of(count, kT), kT, 0, s>>>(n, count, ids, level, bits, touched, ctr);
    if (n > 0) touched_size_kernel<<<few(n), kT, 0, s>>>(n, level, touched, ctr);
}

}  // namespace kb
