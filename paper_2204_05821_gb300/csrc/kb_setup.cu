// Per-call setup kernels: input validation, the in-edge / both-direction CSR
// the backward and two-sided equivalences read (paper Defs. "bw-bisim" and
// "vertex-labeled-bw-bisimulation" use in-neighbours, N^-(v) of Section 3.1),
// hub discovery, an int64 prefix scan and level-row copies.
#include <cuda_runtime.h>

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {
namespace {

int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

__global__ void validate_kernel(int64_t n, int64_t m, const int64_t* row, const int32_t* col, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (row) {
        if (t0 == 0 && (row[0] != 0 || row[n] != m)) bad = true;
        for (int64_t v = t0; v < n; v += stride)
            if (row[v + 1] < row[v]) bad = true;
    }
    for (int64_t e = t0; e < m; e += stride) {
        const int32_t w = col[e];
        if (w < 0 || (int64_t)w >= n) bad = true;
    }
    if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(&ctr->err, kErrInvalid);
}

// ---- in-edge CSR
// Edges in tiles of kCsrTile consecutive ones per CTA.  Both passes count the
// targets of a tile in a shared hash table and send one global atomic per
// distinct target: a hub that receives a tenth of all edges would otherwise
// serialise as many atomics on one address.  (25 x 10^6 power-law edges in both
// directions: 747 us of counting and 2086 us of placing with one atomic and one
// binary search over all offsets per edge.)
constexpr int kCsrThreads = 256;
constexpr int kCsrPer = 8;
constexpr int kCsrTile = kCsrThreads * kCsrPer;
constexpr int kCsrSlots = 2 * kCsrTile;
constexpr uint32_t kNoTarget = 0xffffffffu;

// A tile's targets: (target, edges of the tile) words, the target's word empty
// or claimed by a CAS.
__device__ __forceinline__ int tile_slot(uint2* tab, uint32_t w) {
    uint32_t slot = (w * 2654435761u) >> 20;
    static_assert(kCsrSlots == 1 << 12, "the multiplicative hash keeps 12 bits");
    while (true) {
        const uint32_t old = atomicCAS(&tab[slot].x, kNoTarget, w);
        if (old == kNoTarget || old == w) return (int)slot;
        slot = (slot + 1) & (kCsrSlots - 1);
    }
}

__device__ __forceinline__ void clear_tile(uint2* tab) {
    for (int i = threadIdx.x; i < kCsrSlots; i += kCsrThreads) tab[i] = make_uint2(kNoTarget, 0u);
}

__global__ void __launch_bounds__(kCsrThreads) in_degree_kernel(int64_t m, const int32_t* col, int64_t* deg) {
    __shared__ uint2 tab[kCsrSlots];
    const int64_t e0 = (int64_t)blockIdx.x * kCsrTile;
    uint32_t w[kCsrPer];
#pragma unroll
    for (int u = 0; u < kCsrPer; ++u) {
        const int64_t e = e0 + u * kCsrThreads + threadIdx.x;
        w[u] = e < m ? (uint32_t)__ldcs(col + e) : kNoTarget;
    }
    clear_tile(tab);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kCsrPer; ++u)
        if (w[u] != kNoTarget) atomicAdd(&tab[tile_slot(tab, w[u])].y, 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < kCsrSlots; i += kCsrThreads) {
        const uint2 t = tab[i];
        if (t.x != kNoTarget) atomicAdd(reinterpret_cast<unsigned long long*>(&deg[t.x]), (unsigned long long)t.y);
    }
}

__global__ void rows_kernel(int64_t n, const int64_t* row, const int64_t* in_prefix, int include_out,
                            int64_t* row_p, int64_t* cursor) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += stride) {
        const int64_t r = (include_out ? row[v] : 0) + in_prefix[v];
        row_p[v] = r;
        if (v < n) cursor[v] = r + (include_out ? row[v + 1] - row[v] : 0);
    }
}

// Writes every edge at its target's cursor (and, for both directions, at its
// place among the source's out-edges, e + in_prefix[source]).
__global__ void __launch_bounds__(kCsrThreads) place_edges_kernel(int64_t n, int64_t m, const int64_t* row,
                                                                  const int32_t* col, const int32_t* lab,
                                                                  int include_out, const int64_t* in_prefix,
                                                                  int32_t* col_p, int32_t* lab_p, int64_t* cursor) {
    __shared__ uint2 tab[kCsrSlots];  // (target, edges), then the target's first position in the tile
    __shared__ int32_t s_src[kCsrTile];
    const int tid = threadIdx.x;
    const int64_t e0 = (int64_t)blockIdx.x * kCsrTile;
    const int64_t e1 = min(m, e0 + kCsrTile);
    uint32_t w[kCsrPer];
    int32_t l[kCsrPer];
#pragma unroll
    for (int u = 0; u < kCsrPer; ++u) {
        const int64_t e = e0 + u * kCsrThreads + tid;
        w[u] = e < e1 ? (uint32_t)__ldcs(col + e) : kNoTarget;
        l[u] = lab && e < e1 ? __ldcs(lab + e) : 0;
    }
    clear_tile(tab);
    __syncthreads();
    uint32_t at[kCsrPer];  // slot << 16 | edges of the tile with this target before this one
#pragma unroll
    for (int u = 0; u < kCsrPer; ++u) {
        at[u] = 0;
        if (w[u] == kNoTarget) continue;
        const int slot = tile_slot(tab, w[u]);
        at[u] = ((uint32_t)slot << 16) | atomicAdd(&tab[slot].y, 1u);
    }
    __syncthreads();
    for (int i = tid; i < kCsrSlots; i += kCsrThreads) {
        const uint2 t = tab[i];
        if (t.x == kNoTarget) continue;
        const unsigned long long first =
            atomicAdd(reinterpret_cast<unsigned long long*>(&cursor[t.x]), (unsigned long long)t.y);
        tab[i] = make_uint2((uint32_t)first, (uint32_t)(first >> 32));
    }
    tile_sources<kCsrThreads, kCsrPer>(n, row, e0, e1, s_src);
#pragma unroll
    for (int u = 0; u < kCsrPer; ++u) {
        if (w[u] == kNoTarget) continue;
        const int i = u * kCsrThreads + tid;
        const int64_t v = s_src[i];
        if (include_out) {
            const int64_t q = e0 + i + in_prefix[v];
            col_p[q] = (int32_t)w[u];
            if (lab_p) lab_p[q] = l[u];
        }
        const uint2 t = tab[at[u] >> 16];
        const int64_t q = (int64_t)(((uint64_t)t.y << 32) | t.x) + (at[u] & 0xffffu);
        col_p[q] = (int32_t)((uint32_t)v | 0x80000000u);
        if (lab_p) lab_p[q] = l[u];
    }
}

// Hub and extent of every hub chunk; the extent is packed as (first edge << 16)
// | edge count, so a chunk CTA reads one word instead of a chain of four
// dependent loads.
__global__ void chunk_ext_kernel(int64_t chunks, int32_t n_hubs, const int32_t* hub_v, const int64_t* chunk_off,
                                 const int64_t* row, int32_t chunk, int32_t* chunk_hub, uint64_t* out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks; c += stride) {
        int32_t h = 0, hi = n_hubs;  // chunk_off[h] <= c < chunk_off[hi]
        while (hi - h > 1) {
            const int32_t mid = (h + hi) >> 1;
            if (chunk_off[mid] <= c) h = mid; else hi = mid;
        }
        const int32_t v = hub_v[h];
        const int64_t e0 = row[v] + (c - chunk_off[h]) * (int64_t)chunk;
        const int64_t len = min((int64_t)chunk, row[(int64_t)v + 1] - e0);
        chunk_hub[c] = h;
        out[c] = ((uint64_t)e0 << 16) | (uint64_t)len;
    }
}

// ---- locality order (see RoundParams::perm)
// How often each vertex is gathered: its occurrences in the processed col,
// counted over runs of 32 edges taken every `stride` edges (all edges when
// stride == 32).
__global__ void count_targets_kernel(int64_t m, const int32_t* col, int64_t stride, uint32_t* cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t runs = (m + stride - 1) / stride;
    for (int64_t r = warp; r < runs; r += nwarps) {
        const int64_t e = r * stride + lane;
        if (e < m) atomicAdd(&cnt[col[e] & 0x7fffffff], 1u);
    }
}

// 256 classes, about 8 per octave of the count; class 0 = never gathered.
__device__ __forceinline__ int hot_class(uint32_t c) {
    if (c == 0) return 0;
    const int e = 31 - __clz(c);
    const int frac = e >= 3 ? (int)((c >> (e - 3)) & 7u) : (int)((c << (3 - e)) & 7u);
    return min(255, 1 + e * 8 + frac);
}

__global__ void class_hist_kernel(int64_t n, const uint32_t* cnt, unsigned long long* hist) {
    __shared__ uint32_t h[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        atomicAdd(&h[hot_class(cnt[v])], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], (unsigned long long)h[i]);
}

// cursor[k] = vertices in classes above k (hotter classes come first).
__global__ void class_base_kernel(const unsigned long long* hist, unsigned long long* cursor) {
    __shared__ unsigned long long s[256];
    const int k = threadIdx.x;
    s[k] = hist[k];
    __syncthreads();
    if (k == 0) {
        unsigned long long run = 0;
        for (int j = 255; j >= 0; --j) {
            const unsigned long long c = s[j];
            s[j] = run;
            run += c;
        }
    }
    __syncthreads();
    cursor[k] = s[k];
}

// perm[v] = position of v in the class order; one atomic per class and warp.
__global__ void class_scatter_kernel(int64_t n, const uint32_t* cnt, unsigned long long* cursor, int32_t* perm) {
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x; b < n; b += stride) {
        const int64_t v = b + threadIdx.x;
        const bool ok = v < n;
        const int k = ok ? hot_class(cnt[v]) : 256 + lane;  // lanes past the end match nobody
        const unsigned grp = __match_any_sync(kFull, k);
        const int leader = __ffs(grp) - 1;
        unsigned long long base = 0;
        if (ok && lane == leader) base = atomicAdd(&cursor[k], (unsigned long long)__popc(grp));
        base = __shfl_sync(kFull, base, leader);
        if (ok) perm[v] = (int32_t)(base + __popc(grp & ((1u << lane) - 1u)));
    }
}

// Neighbour ids -> positions in the order, keeping the direction bit.
__global__ void remap_cols_kernel(int64_t m, const int32_t* col, const int32_t* perm, int32_t* out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
        const int32_t w = col[e];
        out[e] = (int32_t)((uint32_t)perm[w & 0x7fffffff] | ((uint32_t)w & 0x80000000u));
    }
}

// ---- degree classes
// One pass over the row offsets: a bitmap per class (DegreeClass) says which one
// a vertex's degree falls in (no bit: 1 .. bounds.small edges), counted per tile
// of kListTile vertices and in ctr.  A CTA counts its classes before it touches
// global memory (an atomic per warp on one counter was 130 us of the pass over
// 10^7 vertices).
constexpr int kListTile = 131072;  // vertices whose words one CTA of the list kernel turns into ids
constexpr int kClassPer = 4096;    // vertices per CTA of the class kernel, at most; a divisor of kListTile

// The CTAs past the class_ctas first ones check ids (CheckIds) meanwhile.
__global__ void __launch_bounds__(256) classes_kernel(int64_t n, int64_t m, const int64_t* row, ClassBounds bounds,
                                                      uint32_t* bits, int64_t pitch, uint32_t* tile_counts, int per,
                                                      CheckRows check, unsigned class_ctas, CheckIds ids, HubSink hubs,
                                                      Counters* ctr) {
    if (blockIdx.x >= class_ctas) {
        const int64_t stride = (int64_t)(gridDim.x - class_ctas) * 256;
        const int64_t t0 = (int64_t)(blockIdx.x - class_ctas) * 256 + threadIdx.x;
        bool wrong = false;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int32_t* a = ids.a[k];
            const int64_t count = ids.count[k];
            int64_t i = t0;
            for (; i + 7 * stride < count; i += 8 * stride) {  // eight loads in flight
                int32_t x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = __ldcs(a + i + u * stride);
#pragma unroll
                for (int u = 0; u < 8; ++u) wrong |= x[u] < 0 || (int64_t)x[u] >= n;
            }
            for (; i < count; i += stride) wrong |= a[i] < 0 || (int64_t)a[i] >= n;
        }
        if (__any_sync(kFull, wrong) && (threadIdx.x & 31) == 0) atomicOr(&ctr->err, kErrInvalid);
        return;
    }
    __shared__ uint32_t s_n[kClassLists];
    if (threadIdx.x < kClassLists) s_n[threadIdx.x] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t v0 = (int64_t)blockIdx.x * per;
    const int64_t nw = (n >> 5) + 1;
    bool bad = check == CheckRows::kAll && blockIdx.x == 0 && threadIdx.x == 0 && (row[0] != 0 || row[n] != m);
    uint32_t c[kClassLists] = {0, 0, 0};
#pragma unroll 4
    for (int i = 0; i < per / 256; ++i) {
        const int64_t v = v0 + i * 256 + threadIdx.x;
        const int64_t d = v < n ? row[v + 1] - row[v] : 1;
        bad |= d < 0;
        const bool mid = v < n && d > bounds.small && d <= bounds.mid, hub = v < n && d > bounds.medium;
        if (hub && hubs.cap) {
            const uint32_t at = atomicAdd(&ctr->hub_at, 1u);
            if (at < hubs.cap) {
                hubs.v[at] = (int32_t)v;
                hubs.deg[at] = d;
            }
        }
        unsigned w[1 + kClassLists];
        w[kEdgeless] = __ballot_sync(kFull, d == 0);
        w[kMid] = __ballot_sync(kFull, mid);
        w[kMedium] = __ballot_sync(kFull, v < n && d > bounds.small && !mid && !hub);
        w[kHub] = __ballot_sync(kFull, hub);
        if (lane == 0 && (v >> 5) < nw) {
#pragma unroll
            for (int k = 0; k <= kClassLists; ++k) bits[k * pitch + (v >> 5)] = w[k];
        }
#pragma unroll
        for (int k = 0; k < kClassLists; ++k) c[k] += __popc(w[k + 1]);
    }
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < kClassLists; ++k)
            if (c[k]) atomicAdd(&s_n[k], c[k]);
    }
    if (check != CheckRows::kNone && bad) atomicOr(&ctr->err, kErrInvalid);
    __syncthreads();
    if (threadIdx.x < kClassLists && s_n[threadIdx.x]) {
        atomicAdd(&tile_counts[kClassLists * (v0 / kListTile) + threadIdx.x], s_n[threadIdx.x]);
        atomicAdd(reinterpret_cast<unsigned long long*>(&ctr->n_class[threadIdx.x]),
                  (unsigned long long)s_n[threadIdx.x]);
    }
}

// ---- int64 exclusive scan (reduce, scan of block sums, down-sweep)
constexpr int kT = 1024;
constexpr int kItems = 4;
constexpr int kTile = kT * kItems;

__device__ __forceinline__ int64_t block_exscan_i64(int64_t x, int64_t* tmp, int64_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) tmp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int64_t w = tmp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        tmp[lane] = w;
    }
    __syncthreads();
    const int64_t base = warp > 0 ? tmp[warp - 1] : 0;
    *total = tmp[31];
    __syncthreads();
    return base + incl - x;
}

// The set bits of a class bitmap as ascending vertex ids (with their degrees
// when deg is given): a CTA takes the words of one tile and finds its place from
// the counts of the tiles before it.  Nothing is written at or past cap.
static_assert(kListTile == kT * 4 * 32, "four words per thread");
struct TwoLists {
    ClassList l[2];
};
__global__ void __launch_bounds__(kT) class_list_kernel(int64_t n, const int64_t* row, const uint32_t* all_bits,
                                                        int64_t pitch, const uint32_t* all_counts,
                                                        const TwoLists lists) {
    __shared__ int64_t tmp[32];
    const ClassList& L = lists.l[blockIdx.y];
    const uint32_t* bits = all_bits + L.cls * pitch;
    const uint32_t* tile_counts = all_counts + L.cls - 1;
    const int64_t cap = L.cap;
    int32_t* out = L.out;
    int64_t* deg = L.deg;
    if (tile_counts[kClassLists * (int64_t)blockIdx.x] == 0) return;  // uniform over the CTA
    int64_t before = 0, base;
    for (int64_t t = threadIdx.x; t < blockIdx.x; t += kT) before += tile_counts[kClassLists * t];
    block_exscan_i64(before, tmp, &base);
    const int64_t nw = (n >> 5) + 1;
    const int64_t w0 = (int64_t)blockIdx.x * (kListTile / 32) + (int64_t)threadIdx.x * 4;
    uint32_t w[4];
    int64_t c = 0, total;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        w[u] = w0 + u < nw ? bits[w0 + u] : 0u;
        c += __popc(w[u]);
    }
    int64_t at = base + block_exscan_i64(c, tmp, &total);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        while (w[u]) {
            const int64_t v = (w0 + u) * 32 + (__ffs(w[u]) - 1);
            w[u] &= w[u] - 1;
            if (at < cap) {
                out[at] = (int32_t)v;
                if (deg) deg[at] = row[v + 1] - row[v];
            }
            ++at;
        }
    }
}

__global__ void __launch_bounds__(kT) scan_reduce_kernel(const int64_t* in, int64_t n, int64_t* sums) {
    __shared__ int64_t tmp[32];
    const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kItems;
    int64_t s = 0;
#pragma unroll
    for (int u = 0; u < kItems; ++u)
        if (base + u < n) s += in[base + u];
    int64_t total;
    block_exscan_i64(s, tmp, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kT) scan_sums_kernel(int64_t* sums, int64_t nb) {
    __shared__ int64_t tmp[32];
    int64_t carry = 0;
    for (int64_t b = 0; b < nb; b += kT) {
        const int64_t i = b + threadIdx.x;
        const int64_t x = i < nb ? sums[i] : 0;
        int64_t total;
        const int64_t ex = block_exscan_i64(x, tmp, &total);
        if (i < nb) sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void __launch_bounds__(kT) scan_down_kernel(const int64_t* in, int64_t n, const int64_t* sums,
                                                        int64_t* out) {
    __shared__ int64_t tmp[32];
    const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kItems;
    int64_t c[kItems];
    int64_t s = 0;
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        c[u] = base + u < n ? in[base + u] : 0;
        s += c[u];
    }
    int64_t total;
    int64_t ex = block_exscan_i64(s, tmp, &total) + sums[blockIdx.x];
    __syncthreads();  // every thread has read its inputs before any output is written (in may alias out)
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
        if (base + u < n) out[base + u] = ex;
        ex += c[u];
    }
}

// rows consecutive rows of n entries, each a copy of src, which is read once
template <typename T>
__global__ void __launch_bounds__(256) copy_rows_kernel(const T* src, int64_t n, int rows, T* dst) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const T x = __ldcs(src + i);
        for (int r = 0; r < rows; ++r) dst[(int64_t)r * n + i] = x;
    }
}

__global__ void write_total_kernel(const int64_t* sums, int64_t nb, int64_t* out, int64_t n) { out[n] = sums[nb]; }

}  // namespace

void launch_validate(int64_t n, int64_t m, const int64_t* row, const int32_t* col, Counters* ctr, cudaStream_t s) {
    validate_kernel<<<grid_for(n > m ? n : m, 256), 256, 0, s>>>(n, m, row, col, ctr);
}

void launch_in_degree(int64_t m, const int32_t* col, int64_t* deg, cudaStream_t s) {
    if (m <= 0) return;
    in_degree_kernel<<<(unsigned)((m + kCsrTile - 1) / kCsrTile), kCsrThreads, 0, s>>>(m, col, deg);
}

size_t scan_i64_tmp(int64_t n) { return (size_t)((n + kTile - 1) / kTile) + 2; }

void launch_scan_i64(const int64_t* in, int64_t n, int64_t* out, int64_t* tmp, cudaStream_t s) {
    const int64_t nb = (n + kTile - 1) / kTile;
    if (nb > 0) scan_reduce_kernel<<<(unsigned)nb, kT, 0, s>>>(in, n, tmp);
    scan_sums_kernel<<<1, kT, 0, s>>>(tmp, nb);
    if (nb > 0) scan_down_kernel<<<(unsigned)nb, kT, 0, s>>>(in, n, tmp, out);
    write_total_kernel<<<1, 1, 0, s>>>(tmp, nb, out, n);
}

void launch_build_csr(int64_t n, int64_t m, const int64_t* row, const int32_t* col, const int32_t* lab,
                      const int64_t* in_prefix, int include_out, int64_t* row_p, int32_t* col_p, int32_t* lab_p,
                      int64_t* cursor, cudaStream_t s) {
    rows_kernel<<<grid_for(n + 1, 256), 256, 0, s>>>(n, row, in_prefix, include_out, row_p, cursor);
    if (m > 0)
        place_edges_kernel<<<(unsigned)((m + kCsrTile - 1) / kCsrTile), kCsrThreads, 0, s>>>(
            n, m, row, col, lab, include_out, in_prefix, col_p, lab_p, cursor);
}

void launch_chunk_ext(int64_t chunks, int32_t n_hubs, const int32_t* hub_v, const int64_t* chunk_off,
                      const int64_t* row, int32_t chunk, int32_t* chunk_hub, uint64_t* out, cudaStream_t s) {
    if (chunks <= 0) return;
    chunk_ext_kernel<<<grid_for(chunks, 256), 256, 0, s>>>(chunks, n_hubs, hub_v, chunk_off, row, chunk, chunk_hub, out);
}

size_t class_tiles(int64_t n) { return (size_t)((n + kListTile - 1) / kListTile); }

void launch_classes(int64_t n, int64_t m, const int64_t* row, const ClassBounds& bounds, uint32_t* bits, int64_t pitch,
                    uint32_t* tile_counts, CheckRows check, const CheckIds& ids, const HubSink& hubs, Counters* ctr,
                    cudaStream_t s) {
    if (n <= 0) return;
    int per = 256;  // short CTAs on small graphs (11 us for 10^5 vertices in CTAs of 4096, 4 us in CTAs of 256)
    while (per < kClassPer && n > (int64_t)per * 152 * 8) per *= 2;
    // (n >> 5) + 1 words: the last one may lie past the last vertex
    const unsigned ctas = (unsigned)((n + per) / per);
    const int64_t most = ids.count[0] > ids.count[1] ? ids.count[0] : ids.count[1];
    const unsigned id_ctas = most > 0 ? (unsigned)grid_for(most, 256) : 0u;
    classes_kernel<<<ctas + id_ctas, 256, 0, s>>>(n, m, row, bounds, bits, pitch, tile_counts, per, check, ctas, ids,
                                                  hubs, ctr);
}

void launch_class_lists(int64_t n, const int64_t* row, const uint32_t* bits, int64_t pitch, const uint32_t* tile_counts,
                        const ClassList& a, const ClassList& b, cudaStream_t s) {
    TwoLists l;
    int lists = 0;
    for (const ClassList* x : {&a, &b})
        if (x->cap > 0) l.l[lists++] = *x;
    if (n <= 0 || !lists) return;
    class_list_kernel<<<dim3((unsigned)class_tiles(n), (unsigned)lists), kT, 0, s>>>(n, row, bits, pitch, tile_counts, l);
}

void launch_locality_order(int64_t n, int64_t m, const int32_t* col, uint32_t* cnt, unsigned long long* hist,
                           int32_t* perm, cudaStream_t s) {
    if (n <= 0) return;
    cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * (size_t)n, s);
    cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * 512, s);
    if (m > 0) {
        // every edge up to 2^26 edges, then one run of 32 in every 256
        const int64_t stride = m <= ((int64_t)1 << 26) ? 32 : 256;
        const int64_t runs = (m + stride - 1) / stride;
        count_targets_kernel<<<grid_for(runs * 32, 256), 256, 0, s>>>(m, col, stride, cnt);
    }
    class_hist_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, cnt, hist);
    class_base_kernel<<<1, 256, 0, s>>>(hist, hist + 256);
    class_scatter_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, cnt, hist + 256, perm);
}

void launch_remap_cols(int64_t m, const int32_t* col, const int32_t* perm, int32_t* out, cudaStream_t s) {
    if (m <= 0) return;
    remap_cols_kernel<<<grid_for(m, 256), 256, 0, s>>>(m, col, perm, out);
}

void launch_copy_rows(int32_t* levels, int64_t n, int src, int first, int last, cudaStream_t s) {
    if (n <= 0 || last < first) return;
    int32_t* from = levels + (size_t)src * (size_t)n;
    int32_t* to = levels + (size_t)first * (size_t)n;
    if (((reinterpret_cast<uintptr_t>(levels) | (uintptr_t)(4 * n)) & 15) == 0)  // every row starts on 16 bytes
        copy_rows_kernel<<<grid_for(n / 4, 256), 256, 0, s>>>(reinterpret_cast<const int4*>(from), n / 4, last - first + 1,
                                                              reinterpret_cast<int4*>(to));
    else
        copy_rows_kernel<<<grid_for(n, 256), 256, 0, s>>>(from, n, last - first + 1, to);
}

}  // namespace kb
