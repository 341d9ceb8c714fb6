// Device helpers of the serving arena: placing a request's CSR (and moving
// it during compaction) with vertex and edge ids rebased.
#include <cuda_runtime.h>

#include "kb_device.cuh"
#include "kb_internal.cuh"

namespace kb {
namespace {

int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 16) b = 152 * 16;
    return (int)b;
}

__global__ void place_vertices_kernel(const PlaceArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= a.n; i += stride) {
        a.drow[a.dst_vbase + i] = a.srow[a.src_vbase + i] - a.src_ebase + a.dst_ebase;
        if (i == a.n) continue;
        a.dvlab[a.dst_vbase + i] = a.svlab ? a.svlab[a.src_vbase + i] : 0;
        if (a.sname) a.dname[a.dst_vbase + i] = a.sname[a.src_vbase + i] - (uint32_t)a.src_vbase + (uint32_t)a.dst_vbase;
    }
}

__global__ void place_edges_kernel(const PlaceArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < a.m; j += stride) {
        const uint32_t c = (uint32_t)a.scol[a.src_ebase + j];
        const uint32_t w = (c & 0x7fffffffu) - (uint32_t)a.src_vbase + (uint32_t)a.dst_vbase;
        a.dcol[a.dst_ebase + j] = (int32_t)((c & 0x80000000u) | w);
        a.dlab[a.dst_ebase + j] = a.slab ? a.slab[a.src_ebase + j] : 0;
    }
}

// A request's CSR from its caller's pinned arrays straight to the arena's tail,
// checked on the way: one pass over the link instead of a copy to device memory,
// a check and a placing pass.  *verdict becomes 1 when the CSR is malformed; what
// was placed then is never used (nothing here indexes by what it reads), and the
// offset in front of it, the end of its predecessor, is written from the arguments
// only.  Bound by the link: 210 GB/s, which 32 CTAs reach as well as 1,216 or the
// copy engine (268 MB of 16 requests: copies, checks and placing in turn 2360 us,
// the next request's copies overlapped 1920 us, this kernel
// 1585 us).
constexpr int kAdmitThreads = 256;
constexpr int kAdmitUnroll = 8;  // loads in flight per thread and array

__global__ void __launch_bounds__(kAdmitThreads) place_checked_kernel(const PlaceArgs a, int32_t* verdict) {
    const int64_t stride = (int64_t)gridDim.x * kAdmitThreads;
    const int64_t t0 = (int64_t)blockIdx.x * kAdmitThreads + threadIdx.x;
    bool bad = false;
    for (int64_t j0 = t0; j0 < a.m; j0 += kAdmitUnroll * stride) {
        int32_t c[kAdmitUnroll], l[kAdmitUnroll];
#pragma unroll
        for (int u = 0; u < kAdmitUnroll; ++u) {
            const int64_t j = j0 + u * stride;
            c[u] = j < a.m ? __ldcs(a.scol + j) : 0;
            l[u] = a.slab && j < a.m ? __ldcs(a.slab + j) : 0;
        }
#pragma unroll
        for (int u = 0; u < kAdmitUnroll; ++u) {
            const int64_t j = j0 + u * stride;
            if (j >= a.m) continue;
            if (c[u] < 0 || (int64_t)c[u] >= a.n) bad = true;
            a.dcol[a.dst_ebase + j] = (int32_t)((uint32_t)c[u] + (uint32_t)a.dst_vbase);
            a.dlab[a.dst_ebase + j] = l[u];
        }
    }
    // offsets: every lane reads its vertex's, and the next one's from its neighbour
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = t0 - lane; i0 < a.n; i0 += stride) {  // uniform over the warp
        const int64_t i = i0 + lane;
        const int64_t r = i < a.n ? __ldcs(a.srow + i) : 0;
        const int32_t v = a.svlab && i < a.n ? __ldcs(a.svlab + i) : 0;
        int64_t next = __shfl_down_sync(kFull, (long long)r, 1);
        if (i >= a.n) continue;
        if (lane == 31 || i + 1 == a.n) next = __ldcs(a.srow + i + 1);
        if (next < r || (i == 0 && r != 0) || (i + 1 == a.n && next != a.m)) bad = true;
        a.drow[a.dst_vbase + i] = i == 0 ? a.dst_ebase : r + a.dst_ebase;
        if (i + 1 == a.n) a.drow[a.dst_vbase + a.n] = a.m + a.dst_ebase;
        a.dvlab[a.dst_vbase + i] = v;
    }
    if (bad) atomicOr(verdict, 1);
}

}  // namespace

void launch_place_checked(const PlaceArgs& a, int32_t* verdict, cudaStream_t s) {
    const int64_t work = a.n + a.m / kAdmitUnroll + 1;
    const int64_t ctas = (work + kAdmitThreads - 1) / kAdmitThreads;
    place_checked_kernel<<<(unsigned)(ctas < 152 * 4 ? ctas : 152 * 4), kAdmitThreads, 0, s>>>(a, verdict);
}

void launch_place(const PlaceArgs& a, cudaStream_t s) {
    place_vertices_kernel<<<grid_for(a.n + 1, 256), 256, 0, s>>>(a);
    if (a.m > 0) place_edges_kernel<<<grid_for(a.m, 256), 256, 0, s>>>(a);
}

}  // namespace kb
