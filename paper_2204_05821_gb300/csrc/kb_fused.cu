// All rounds of a small graph in one cooperative kernel, and the starting level
// before them when its keys are small.
//
// A round is a chain of six or seven short passes, each of which takes a few
// microseconds on a small graph, about as long as launching it and draining the
// one before; then the host reads the count and decides.  Here the passes are
// phases between barriers of the whole grid, the stop test runs on the device and
// the rows behind a stable round are copied at once, so a call has one launch and
// one round trip for up to kFusedRounds rounds.  The small, mid and medium
// vertices and the hub chunks share one phase: their full signature compares take
// representatives of any degree.
//
// What bounds it: the chain of dependent loads in each phase and some 2 us per
// barrier, five to seven a round.  Whole calls, one launch per pass against this
// kernel: 10^4 vertices and 5 x 10^4 edges: 248 -> 183 us; a graph of
// 7 x 10^5 edges with host buffers: 525 -> 450 us; 3 x 10^5 vertices to their
// fixpoint in 11 rounds: 1066 -> 847 us.  The starting level's four passes in here
// too: 159 -> 147 us for the first (with fewer setup operations since).  Three CTAs per SM (a CTA per 256
// vertices or 1024 edges) as the occupancy allows: the last took 885 us with two and
// 1209 us with one.
//
// The grid is launched cooperatively, so all its CTAs run at once and the
// barrier's wait ends; it has a limit all the same, after which the kernel
// reports an error and returns, and the call runs again with one kernel per pass
// (as it does when the device refuses the launch).
#define KB_LEVELS_WRITTEN
#include <cuda_runtime.h>

#include <algorithm>

#include "kb_medium.cuh"
#include "kb_round.cuh"
#include "kb_small.cuh"

namespace kb {
namespace {

constexpr int kFusedThreads = 256;
constexpr int kFusedWarps = kFusedThreads / 32;
static_assert(kFusedThreads == kSmallThreads && kFusedWarps == kMidWarps && kFusedThreads == kHubFinalThreads,
              "the bodies' CTAs have one size");
// Bitmap words up to which the rank scan counts the words before a CTA's own
// instead of exchanging sums across a barrier (hierarchy of 3 x 10^5 vertices:
// 847 against 893 us with 9,376 words).
constexpr int64_t kDirectWords = 16384;

union FusedSmem {
    SmallSmem<false, false> small;
    SmallSmem<false, true> compact;
    MidSmem mid;
    MediumSmem<2 * kMedSplit, kFusedWarps> medium;
    MediumCtaSmem<2 * kMaxHubThreshold, kFusedThreads> medium_cta;
    HubChunkSmem<kMaxHubChunk> chunk1024;
    HubChunkSmem<kDefaultHubChunk> chunk512;
    HubChunkSmem<kMaxHubChunk / 4> chunk256;
    HubFinalSmem hub;
    struct {
        uint32_t warp[kFusedWarps], word, clean[kFusedWarps][32], on[4];
    } pass;
    __device__ FusedSmem() {}
};

// Wait for the whole grid; false when the limit ran out (or did for another CTA).
// A CTA passes only when all of them arrived, so what it reads next is whole
// even if others gave up meanwhile; it ends at the next barrier.
__device__ __forceinline__ bool grid_barrier(Counters* ctr, uint32_t& target, uint32_t max_polls) {
    target += gridDim.x;
    __shared__ int s_go;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&ctr->arrived, 1u);
        volatile uint32_t* arrived = &ctr->arrived;
        uint32_t polls = 0;
        while ((int32_t)(*arrived - target) < 0 && ++polls < max_polls) {
        }
        s_go = polls < max_polls && !(*(volatile int32_t*)&ctr->err & kErrWait);
        if (polls >= max_polls) atomicOr(&ctr->err, kErrWait);
        __threadfence();
    }
    __syncthreads();
    return s_go != 0;
}

// Sum of one value per thread, for every thread.
__device__ __forceinline__ uint32_t cta_sum(uint32_t x, uint32_t* s_warp) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = x;
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (int i = 0; i < kFusedWarps; ++i) t += s_warp[i];
    return t;
}

template <int kChunk>
__device__ __forceinline__ void all_chunks(const RoundParams& p, HubChunkSmem<kChunk>& sm, int64_t total) {
    for (int64_t c = blockIdx.x; c < total; c += gridDim.x) {
        __syncthreads();
        hub_chunk<kChunk, kFusedThreads>(p, sm, c);
    }
}

__global__ void __launch_bounds__(kFusedThreads, 3) fused_rounds_kernel(const FusedRounds a) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    FusedSmem& sm = *reinterpret_cast<FusedSmem*>(s_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n = a.p.n, nw = (n >> 5) + 1;
    Counters* ctr = a.p.ctr;
    const int64_t warps = (int64_t)gridDim.x * kFusedWarps, my_warp = (int64_t)blockIdx.x * kFusedWarps + warp;
    const int64_t thread = (int64_t)blockIdx.x * kFusedThreads + tid, threads = warps * 32;
    uint32_t target = 0;

    for (int i = a.key0 ? a.first - 1 : a.first; i <= a.last; ++i) {
        const bool level0 = i < a.first;
        RoundParams p = a.p;
        p.epoch = a.p.epoch + (uint32_t)(i - a.first);
        p.ehigh = a.p.ehigh - (uint32_t)(i - a.first);
        int32_t* out = a.levels ? a.levels + (int64_t)i * n : (i & 1 ? a.ping[1] : a.ping[0]);
        // what the freeze pass before counted decides which classes have work
        const bool all = a.all_on && i == a.first;
        const int64_t frozen = all ? 0 : *(volatile int64_t*)&ctr->frozen;
        bool on[3];
        for (int c = 0; c < 3; ++c) on[c] = all || *(volatile int64_t*)&ctr->class_on[c] > 0;
        const bool hubs = p.n_hubs > 0 && on[2] && !level0;

        // ---- keys
        if (level0) {  // every label's smallest vertex, shared when the label has others
            for (int64_t l = thread; l < kDenseLabels; l += threads) {
                const uint32_t e = a.lmin[l];
                if (e == kNoMember) continue;
                const uint32_t m = e & kVertexMask;
                atomicOr(&p.bitmap[m >> 5], 1u << (m & 31));
                if (!(e & kSingleBit)) atomicOr(&p.shared[m >> 5], 1u << (m & 31));
            }
        } else if (frozen * 4 > n) {
            if ((n - frozen) * 64 < n) p.warp_verts = sparse_task(p.warp_verts);  // few vertices refine
            small_body<false, true, true>(p, sm.compact, my_warp, warps);
        } else {
            small_body<false, false, true>(p, sm.small, my_warp, warps);
        }
        if (p.n_mid > 0 && on[0] && !level0) {
            __syncthreads();
            const int32_t per = (int32_t)min((int64_t)kMedTask, (p.n_mid + warps - 1) / warps);
            for (int64_t t = my_warp * per; t < p.n_mid; t += warps * per) mid_task(p, sm.mid.set, sm.mid.mark, t, per);
        }
        if (p.n_med > 0 && on[1] && !level0) {
            const int32_t thr = min(p.hub_threshold, (int32_t)kMaxHubThreshold);
            const int32_t split = min(max(p.med_split, 1), (int32_t)kMedSplit);
            if (p.mid_max < min(thr, split)) {
                __syncthreads();
                const int32_t per = (int32_t)min((int64_t)kMedTask, (p.n_med + warps - 1) / warps);
                for (int64_t t = my_warp * per; t < p.n_med; t += warps * per)
                    medium_task<2 * kMedSplit, kFusedWarps>(p, sm.medium, p.mid_max, min(thr, split), t, per);
            }
            if (thr > split) {
                __syncthreads();
                const int32_t per = (int32_t)min((int64_t)kMedTask, (p.n_med + gridDim.x - 1) / gridDim.x);
                for (int64_t t = (int64_t)blockIdx.x * per; t < p.n_med; t += (int64_t)gridDim.x * per)
                    medium_cta_task<2 * kMaxHubThreshold, kFusedThreads>(p, sm.medium_cta, max(p.mid_max, split), thr, t, per);
            }
        }
        if (hubs) {
            if (p.hub_chunk == 256)
                all_chunks<256>(p, sm.chunk256, a.total_chunks);
            else if (p.hub_chunk == 1024)
                all_chunks<1024>(p, sm.chunk1024, a.total_chunks);
            else
                all_chunks<kDefaultHubChunk>(p, sm.chunk512, a.total_chunks);
            if (!grid_barrier(ctr, target, a.max_polls)) return;
            for (int h = blockIdx.x; h < p.n_hubs; h += gridDim.x) {
                __syncthreads();
                hub_final(p, sm.hub, h);
            }
        }
        if (!grid_barrier(ctr, target, a.max_polls)) return;

        // ---- ranks of the block minima: a CTA per run of words
        const int64_t run = ((nw + gridDim.x - 1) / gridDim.x + 3) & ~(int64_t)3;
        const int64_t wa = min(nw, (int64_t)blockIdx.x * run), wb = min(nw, wa + run);
        uint32_t before = 0;
        const uint4* words = reinterpret_cast<const uint4*>(p.bitmap);
        // (a caller's workspace may start at any 8 bytes)
        if (nw <= kDirectWords && (reinterpret_cast<uintptr_t>(words) & 15) == 0) {  // every CTA counts the words before its own
#pragma unroll 4
            for (int64_t w = tid; w < wa >> 2; w += kFusedThreads) {  // (wa is nw or a multiple of 4)
                const uint4 x = words[w];
                before += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
            }
        } else {
            uint32_t own = 0;
            for (int64_t w = wa + tid; w < wb; w += kFusedThreads) own += __popc(p.bitmap[w]);
            own = cta_sum(own, sm.pass.warp);
            if (tid == 0) a.sums[blockIdx.x] = own;
            if (!grid_barrier(ctr, target, a.max_polls)) return;
            for (int b = tid; b < (int)blockIdx.x; b += kFusedThreads) before += a.sums[b];
        }
        uint32_t base = cta_sum(before, sm.pass.warp);
        for (int64_t w0 = wa; w0 < wb; w0 += kFusedThreads) {
            const int64_t w = w0 + tid;
            const uint32_t x = w < wb ? p.bitmap[w] : 0u;
            uint32_t incl = __popc(x);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            __syncthreads();
            if (lane == 31) sm.pass.warp[warp] = incl;
            __syncthreads();
            uint32_t at = base + incl - __popc(x), total = 0;
            for (int j = 0; j < kFusedWarps; ++j) {
                if (j < warp) at += sm.pass.warp[j];
                total += sm.pass.warp[j];
            }
            if (w < wb) a.rank[w] = make_uint2(at, x);
            base += total;
        }
        if (wa < wb && wb == nw && tid == 0) {
            if (i == a.first) ctr->start_count = ctr->count;
            ctr->prev_count = ctr->count;
            ctr->count = (int64_t)base;
            if (!level0) ctr->round_count[i - a.first] = (int64_t)base;
            ctr->last_round = i;
            ctr->frozen = 0;
            for (int c = 0; c < 3; ++c) ctr->class_on[c] = 0;
            ctr->moved = 0;
            ctr->most_pairs = 0;
        }
        if (!grid_barrier(ctr, target, a.max_polls)) return;

        // ---- ids; under early stop a round that kept the count is the last one
        const bool stable = a.stop_stable && !level0 &&
                            *(volatile int64_t*)&ctr->count == *(volatile int64_t*)&ctr->prev_count;
        if (stable) {
            if (a.levels) {
                const int32_t* src = out - n;
                for (int64_t v = thread; v < n; v += threads) {
                    const int32_t b = src[v];
                    for (int r = i; r <= a.k; ++r) a.levels[(int64_t)r * n + v] = b;
                }
            } else {
                const int32_t* src = i & 1 ? a.ping[0] : a.ping[1];
                for (int64_t v = thread; v < n; v += threads) out[v] = src[v];
            }
            return;
        }
        if (level0) {
            for (int64_t v = thread; v < n; v += threads) {
                const uint32_t l = (uint32_t)a.key0[v];
                uint32_t m = l < (uint32_t)kDenseLabels ? a.lmin[l] & kVertexMask : (uint32_t)n;
                if ((int64_t)m >= n) {  // the keys changed since they were checked
                    set_error(ctr, kErrInvalid);
                    m = (uint32_t)v;
                }
                const uint2 rw = a.rank[m >> 5];
                out[v] = (int32_t)(rw.x + __popc(rw.y & ((1u << (m & 31)) - 1u)));
                if (p.perm) p.gat[p.perm[v]] = (int32_t)m;
                p.minof[v] = m;
            }
        } else {
            assign_frozen(p, a.rank, out, p.moved, a.f.mark ? const_cast<uint32_t*>(a.f.mark) : nullptr, &sm.pass.word);
        }
        if (hubs) {  // leave the used sets and sums empty for the next round
            for (int h = blockIdx.x; h < p.n_hubs; h += gridDim.x) {
                if (!vertex_refines(p, p.hub_v[h])) continue;
                for (int64_t q = p.hub_set_off[h] + tid; q < p.hub_set_off[h + 1]; q += kFusedThreads)
                    p.hub_sets[q] = kEmptyPair;
                if (tid == 0) {
                    p.hub_acc[h] = 0ull;
                    p.hub_cnt[h] = 0u;
                }
            }
        }
        if (i == a.k) return;
        if (!grid_barrier(ctr, target, a.max_polls)) return;

        // ---- frozen blocks of the next round
        const int per_warp = (int)min((int64_t)32, max((int64_t)1, nw / warps));
        if (!level0 && few_moved(p)) {  // (the count is read after the barrier and not written before the next)
            for (int64_t w0 = my_warp * per_warp; w0 < nw; w0 += warps * per_warp)
                dirty_blocks(p, a.f.edgeless, p.moved, kMaxHubThreshold, const_cast<uint32_t*>(a.f.mark), per_warp, nullptr,
                             w0);
            if (!grid_barrier(ctr, target, a.max_polls)) return;
        }
        FreezePass f = a.f;
        f.per_warp = per_warp;
        if (level0) {  // only its singletons are frozen, as after launch_dense_level0
            f.edgeless = nullptr;
            f.mark = nullptr;
            f.moved_clear = nullptr;
            for (int64_t l = thread; l < kDenseLabels; l += threads) a.lmin[l] = kNoMember;
        }
        __syncthreads();
        if (tid < 4) sm.pass.on[tid] = 0u;
        __syncthreads();
        for (int64_t w0 = my_warp * per_warp; w0 < nw; w0 += warps * per_warp)
            freeze_clean(f, sm.pass.clean[warp], sm.pass.on, w0);
        __syncthreads();
        add_frozen(ctr, sm.pass.on);
        if (i == a.last) return;
        if (!grid_barrier(ctr, target, a.max_polls)) return;
    }
}

}  // namespace

int fused_max_ctas() {
    int device = 0, sms = 0, coop = 0, per_sm = 0;
    if (cudaGetDevice(&device) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device) != cudaSuccess || !coop ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaFuncSetAttribute(fused_rounds_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FusedSmem)) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fused_rounds_kernel, kFusedThreads, sizeof(FusedSmem)) !=
            cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms * per_sm;
}

cudaError_t launch_fused_rounds(const FusedRounds& a, int max_ctas, bool again, cudaStream_t s) {
    FusedRounds b = a;
    // a CTA per 256 vertices or 1024 edges, whichever are more: more only lengthen
    // the barriers, fewer leave vertices of high degree to a few CTAs (whole calls by
    // vertices alone / with edges: 1500 vertices of 1000 edges 1567 / 149 us, 10^4 of
    // 100 469 / 212, 300 of 500 755 / 120; Erdos-Renyi and power-law graphs of 2 x 10^4
    // to 1.7 x 10^6 edges with 3 to 12 a vertex: within 3% or up to 12% faster)
    const int64_t want = std::max((a.p.n + 255) / 256, (a.edges + 1023) / 1024);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(max_ctas, want));
    if (b.p.warp_verts <= 0) {  // a task per warp, at least a window
        const int64_t per = (a.p.n + (int64_t)grid * kFusedWarps - 1) / ((int64_t)grid * kFusedWarps);
        b.p.warp_verts = (int32_t)std::min<int64_t>(kDefaultWarpVerts, std::max<int64_t>(32, (per + 31) & ~(int64_t)31));
    }
    if (again) {
        const cudaError_t e = cudaMemsetAsync(&a.p.ctr->arrived, 0, sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
    }
    void* args[] = {&b};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(fused_rounds_kernel), dim3(grid), dim3(kFusedThreads),
                                       args, sizeof(FusedSmem), s);
}

}  // namespace kb
