// Launches of the small-vertex kernel (kb_small.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_small.cuh"

namespace kb {
namespace {

template <bool kLevel0, bool kCompact>
__global__ void __launch_bounds__(kSmallThreads, kSmallMinBlocks) small_round_kernel(const RoundParams p) {
    __shared__ SmallSmem<kLevel0, kCompact> sm;
    small_body<kLevel0, kCompact, false>(p, sm, (int64_t)blockIdx.x * kSmallWarps + (threadIdx.x >> 5), 0);
}

}  // namespace

// Vertices per warp task when the caller gives none: the vertices spread over
// two waves of resident warps, between lo and hi.  A warp walks its task window
// after window, each a chain of dependent loads (offsets, neighbours, blocks,
// table, representative), so a graph that fills only part of the chip with
// tasks of 128 is bound by the length of that chain (104 against 18 us for a
// round of 10^4 vertices when windows held six of them).  From about 1.6 x 10^6
// vertices on every task has 128.
static int64_t task_vertices(int64_t n, int64_t lo, int64_t hi) {
    const int64_t per = (n + 2 * kResidentWarps - 1) / (2 * kResidentWarps);
    return std::min(hi, std::max(lo, (per + 7) & ~(int64_t)7));
}

int32_t default_task_vertices(int64_t n) { return (int32_t)task_vertices(n, 32, kDefaultWarpVerts); }

void launch_small_round(const RoundParams& p, bool level0, SmallWindows windows, cudaStream_t s) {
    if (p.n <= 0) return;
    const bool compact = windows != SmallWindows::kConsecutive;
    int64_t wv = p.warp_verts > 0 ? p.warp_verts : default_task_vertices(p.n);
    // few vertices refine: long warp tasks, so that far fewer CTAs set up and
    // flush a join map for a handful of vertices each
    if (windows == SmallWindows::kSparse) wv = task_vertices(p.n, kDefaultWarpVerts, 4096);
    const int64_t per_cta = wv * kSmallWarps;
    const int64_t blocks = (p.n + per_cta - 1) / per_cta;
    RoundParams q = p;
    q.warp_verts = (int32_t)wv;
    if (level0)
        small_round_kernel<true, false><<<(unsigned)blocks, kSmallThreads, 0, s>>>(q);
    else if (compact)
        small_round_kernel<false, true><<<(unsigned)blocks, kSmallThreads, 0, s>>>(q);
    else
        small_round_kernel<false, false><<<(unsigned)blocks, kSmallThreads, 0, s>>>(q);
}

}  // namespace kb
