// The keys of the small, mid and medium vertices of a round in one launch: a
// block takes tasks of one class, so the classes overlap instead of draining one
// after another.  Their full signature compares take representatives of any
// degree, but the small vertices go first and the others by rising degree, as in
// launches of their own: a lane walks its representative's edges four at a time, and
// a block is represented by its smallest vertex so far.  With the largest first,
// 5 x 10^6 vertices with ids by falling degree and one edge label took 26.1 ms for
// 2.6 (2.4 and 2.1 with random ids; 18.6 with one edge per lane).  So that the long
// tasks at the end do not run alone, they are short: eight entries for a CTA's (with
// up to 32, ids by falling degree and 32 labels: 10^6 vertices 326 for 214 us).  What bounds a class here is what bounds it alone (random accesses; on a
// small graph the chain of dependent loads); what this saves is the draining.  One
// round of 4.8 x 10^5 edges: small 22 us, then mid 14 us; together a whole call
// takes 99 us instead of 119 (with one reset kernel for three clears).
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_medium.cuh"
#include "kb_small.cuh"

namespace kb {
namespace {

constexpr int kKeyThreads = 256;
constexpr int kKeyWarps = kKeyThreads / 32;
static_assert(kKeyThreads == kSmallThreads && kKeyWarps == kMidWarps, "the bodies' CTAs have one size");

union KeySmem {
    SmallSmem<false, false> small;
    MidSmem mid;
    MediumSmem<2 * kMedSplit, kKeyWarps> medium;
    MediumCtaSmem<2 * kMaxHubThreshold, kKeyThreads> medium_cta;
    __device__ KeySmem() {}
};

// CTAs and entries (vertices) per task of each class; dlo, dhi as for the single
// kernels.  Classes follow one another in the grid by rising degree.
struct KeySplit {
    unsigned small_ctas = 0, mid_ctas = 0, medium_ctas = 0, cta_ctas = 0;
    int32_t cta_per = 0, medium_per = 0, mid_per = 0;
    int32_t split = 0, thr = 0;
};

__global__ void __launch_bounds__(kKeyThreads, 4) keys_kernel(const RoundParams p, const KeySplit k) {
    __shared__ __align__(16) unsigned char raw[sizeof(KeySmem)];
    KeySmem& sm = *reinterpret_cast<KeySmem*>(raw);
    const int warp = threadIdx.x >> 5;
    unsigned b = blockIdx.x;
    if (b < k.small_ctas) {
        small_body<false, false, false>(p, sm.small, (int64_t)b * kKeyWarps + warp, 0);
        return;
    }
    b -= k.small_ctas;
    if (b < k.mid_ctas) {
        mid_task(p, sm.mid.set, sm.mid.mark, ((int64_t)b * kKeyWarps + warp) * k.mid_per, k.mid_per);
        return;
    }
    b -= k.mid_ctas;
    if (b < k.medium_ctas) {
        medium_task<2 * kMedSplit, kKeyWarps>(p, sm.medium, p.mid_max, min(k.thr, k.split),
                                              ((int64_t)b * kKeyWarps + warp) * k.medium_per, k.medium_per);
        return;
    }
    b -= k.medium_ctas;
    medium_cta_task<2 * kMaxHubThreshold, kKeyThreads>(p, sm.medium_cta, max(p.mid_max, k.split), k.thr,
                                                       (int64_t)b * k.cta_per, k.cta_per);
}

unsigned ctas_for(int64_t entries, int64_t per_cta) { return (unsigned)((entries + per_cta - 1) / per_cta); }

}  // namespace

void launch_keys(const RoundParams& p, cudaStream_t s) {
    if (p.n <= 0) return;
    KeySplit k;
    k.thr = std::min(p.hub_threshold, (int32_t)kMaxHubThreshold);
    k.split = std::min(std::max(p.med_split, 1), (int32_t)kMedSplit);
    const int64_t resident = 152 * 4;
    auto entries = [](int64_t n, int64_t tasks) { return (int32_t)std::min<int64_t>(kMedTask, (n + tasks - 1) / tasks); };
    if (p.n_mid > 0) {
        k.mid_per = entries(p.n_mid, resident * kKeyWarps);
        k.mid_ctas = ctas_for(p.n_mid, (int64_t)k.mid_per * kKeyWarps);
    }
    if (p.n_med > 0 && p.mid_max < std::min(k.thr, k.split)) {
        k.medium_per = entries(p.n_med, resident * kKeyWarps * 4);
        k.medium_ctas = ctas_for(p.n_med, (int64_t)k.medium_per * kKeyWarps);
    }
    if (p.n_med > 0 && k.thr > k.split) {
        k.cta_per = std::min(8, entries(p.n_med, resident * 8));
        k.cta_ctas = ctas_for(p.n_med, k.cta_per);
    }
    RoundParams q = p;
    if (q.warp_verts <= 0) q.warp_verts = default_task_vertices(p.n);
    k.small_ctas = ctas_for(p.n, (int64_t)q.warp_verts * kKeyWarps);
    keys_kernel<<<k.small_ctas + k.mid_ctas + k.medium_ctas + k.cta_ctas, kKeyThreads, 0, s>>>(q, k);
}

}  // namespace kb
