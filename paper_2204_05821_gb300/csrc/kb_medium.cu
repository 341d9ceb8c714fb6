// Launches of the mid and medium kernels (kb_medium.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_medium.cuh"

namespace kb {
namespace {

__global__ void __launch_bounds__(kMidWarps * 32) mid_round_kernel(const RoundParams p, int32_t per_task) {
    __shared__ uint64_t s_set[kMidWarps * 4][kMidCap];
    __shared__ uint32_t s_mark[kMidWarps * 4][kMidCap / 32];
    mid_task(p, s_set, s_mark, ((int64_t)blockIdx.x * kMidWarps + (threadIdx.x >> 5)) * per_task, per_task);
}

template <int kCap, int kWarps>
__global__ void __launch_bounds__(kWarps * 32) medium_round_kernel(const RoundParams p, int32_t dlo, int32_t dhi,
                                                                    int32_t per_task) {
    __shared__ MediumSmem<kCap, kWarps> sm;
    medium_task<kCap, kWarps>(p, sm, dlo, dhi, ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * per_task, per_task);
}

template <int kCap, int kThreads>
__global__ void __launch_bounds__(kThreads) medium_cta_kernel(const RoundParams p, int32_t dlo, int32_t dhi,
                                                              int32_t per_task) {
    __shared__ MediumCtaSmem<kCap, kThreads> sm;
    medium_cta_task<kCap, kThreads>(p, sm, dlo, dhi, (int64_t)blockIdx.x * per_task, per_task);
}

}  // namespace

// The CTA kernel's 17.5 KB set per CTA would let the SM give nearly all of its
// L1 to shared memory (12 CTAs by registers); at 60% of the maximum carveout 7
// CTAs run and the rest stays L1, which the kernel's many outstanding random
// loads need (2e9-edge graph: 8.2 -> 6.5 ms per round for the medium class).
void set_medium_kernel_attributes() {
    cudaFuncSetAttribute(medium_cta_kernel<2 * kMaxHubThreshold, kMedCtaThreads>,
                         cudaFuncAttributePreferredSharedMemoryCarveout, 60);
}

// List entries per task: enough tasks to fill the chip (13 CTAs of the warp
// kernel fit an SM by shared memory, 7 of the CTA kernel), at most one entry per
// lane.  A task takes its vertices one after another, so a short list in tasks
// of 32 ran on a few warps: 137 us (warp kernel) and 43 us (CTA kernel) on a
// power-law graph of 7 x 10^5 edges, 18 and 15 us with short tasks.
static int32_t task_entries(int64_t n_med, int64_t tasks) {
    return (int32_t)std::min<int64_t>(kMedTask, (n_med + tasks - 1) / tasks);
}

void launch_mid_round(const RoundParams& p, cudaStream_t s) {
    if (p.n_mid <= 0) return;
    const int32_t per = task_entries(p.n_mid, 152 * 6 * kMidWarps * 2);
    const int64_t ctas = (p.n_mid + (int64_t)per * kMidWarps - 1) / ((int64_t)per * kMidWarps);
    mid_round_kernel<<<(unsigned)ctas, kMidWarps * 32, 0, s>>>(p, per);
}

void launch_medium_round(const RoundParams& p, cudaStream_t s) {
    if (p.n_med <= 0) return;
    const int32_t thr = std::min(p.hub_threshold, (int32_t)kMaxHubThreshold);
    const int32_t split = std::min(std::max(p.med_split, 1), (int32_t)kMedSplit);
    const int32_t lo = p.mid_max;
    if (lo < std::min(thr, split)) {
        constexpr int kW = 4;
        const int32_t per = task_entries(p.n_med, 152 * 13 * kW);
        const int64_t ctas = (p.n_med + (int64_t)per * kW - 1) / ((int64_t)per * kW);
        medium_round_kernel<2 * kMedSplit, kW>
            <<<(unsigned)ctas, kW * 32, 0, s>>>(p, lo, std::min(thr, split), per);
    }
    if (thr > split) {
        const int32_t per = task_entries(p.n_med, 152 * 7 * 2);
        medium_cta_kernel<2 * kMaxHubThreshold, kMedCtaThreads>
            <<<(unsigned)((p.n_med + per - 1) / per), kMedCtaThreads, 0, s>>>(p, std::max(lo, split), thr, per);
    }
}

}  // namespace kb
