// kb_refine_round_noalloc: one refinement round that allocates no device
// memory.  Its scratch (block table, slot per vertex, empty-signature minima,
// bitmap of block minima and its prefix, degree classes, counters) lives
// in one file-scope device array of fixed size, shared by every call on a
// device and kept until the process exits.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "kb_internal.cuh"

namespace {

constexpr int64_t kMaxVertices = KB_NOALLOC_MAX_VERTICES;
constexpr uint64_t kTableCap = (uint64_t)2 * kMaxVertices;  // load factor 0.5 at the limit
constexpr size_t kAlign = 256;

constexpr size_t up(size_t x) { return (x + kAlign - 1) & ~(kAlign - 1); }
constexpr int64_t kWords = (kMaxVertices >> 5) + 1;
// layout of the scratch array
constexpr size_t kOffCtr = 0;  // kb::Counters, tile counts and minima bitmap: one memset clears all three
constexpr size_t kTiles = (size_t)((kMaxVertices + 131071) / 131072);
constexpr size_t kOffTiles = kOffCtr + up(sizeof(kb::Counters));
constexpr size_t kOffBitmap = kOffTiles + up(kb::kClassLists * sizeof(uint32_t) * kTiles);
constexpr size_t kOffClasses = kOffBitmap + up(sizeof(uint32_t) * kWords);  // kb::DegreeClass
constexpr size_t kOffTable = kOffClasses + (1 + kb::kClassLists) * up(sizeof(uint32_t) * kWords);
constexpr size_t kOffSlot = kOffTable + up(sizeof(uint64_t) * kTableCap);
constexpr size_t kOffEmin = kOffSlot + up(sizeof(int32_t) * kMaxVertices);
constexpr size_t kOffPrefix = kOffEmin + up(sizeof(uint64_t) * kMaxVertices);
constexpr size_t kOffScan = kOffPrefix + up(sizeof(uint2) * (kWords + 1));  // rank words
constexpr size_t kScanWords = (size_t)((kWords + 4095) / 4096) + 1;
constexpr size_t kOffMed = kOffScan + up(sizeof(uint32_t) * kScanWords);
constexpr size_t kScratchBytes = kOffMed + up(sizeof(int32_t) * kMaxVertices);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
void* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once
// per device; the symbol's host-side name is not a device address).
kb_status scratch_address(int device, unsigned char** out) {
    if (device < 0 || device >= kMaxDevices) return KB_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[device]) {
        void* ptr = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess || !ptr) {
            cudaGetLastError();
            return KB_ERR_CUDA;
        }
        g_scratch_ptr[device] = ptr;
    }
    *out = reinterpret_cast<unsigned char*>(g_scratch_ptr[device]);
    return KB_OK;
}

// What a call starts with: two runs of zeros and one of ones, in 16-byte words
// (one launch in the place of three clears).
__global__ void __launch_bounds__(256) reset_kernel(uint4* zero_a, int64_t a, uint4* zero_b, int64_t b, uint4* ones,
                                                    int64_t c) {
    const int64_t stride = (int64_t)gridDim.x * 256;
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u), o = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (int64_t i = t; i < a; i += stride) zero_a[i] = z;
    for (int64_t i = t; i < b; i += stride) zero_b[i] = z;
    for (int64_t i = t; i < c; i += stride) ones[i] = o;
}

uint64_t next_pow2(uint64_t x) {
    uint64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

#define NA_CUDA(call)                                  \
    do {                                               \
        if ((call) != cudaSuccess) {                   \
            cudaGetLastError();                        \
            return KB_ERR_CUDA;                        \
        }                                              \
    } while (0)

}  // namespace

extern "C" kb_status kb_refine_round_noalloc(void* stream, const kb_graph* g, const kb_options* opt,
                                             const int32_t* prev, int32_t* out, int64_t* count) {
    if (!g || !opt || !count) return KB_ERR_INVALID_ARG;
    if (g->n < 0 || g->m < 0 || g->n > kMaxVertices) return KB_ERR_INVALID_ARG;
    if (opt->direction != KB_DIR_OUT) return KB_ERR_INVALID_ARG;
    if (opt->subject != KB_SUBJECT_PREVIOUS) return KB_ERR_INVALID_ARG;
    if (opt->hash_mode < 0 || opt->hash_mode > 1) return KB_ERR_INVALID_ARG;
    if (opt->hub_threshold < 0 || opt->hub_threshold > kb::kMaxHubThreshold) return KB_ERR_INVALID_ARG;
    if (opt->small_task_vertices != 0 && (opt->small_task_vertices < 32 || opt->small_task_vertices > 65536))
        return KB_ERR_INVALID_ARG;
    if (opt->medium_split < 0 || opt->medium_split > kb::kMaxMedSplit) return KB_ERR_INVALID_ARG;
    if (opt->small_max_degree < 0 || opt->small_max_degree > kb::kMidDegree) return KB_ERR_INVALID_ARG;
    if (g->n == 0) {
        *count = 0;
        return KB_OK;
    }
    if (!g->row_offsets || !prev || !out || (g->m > 0 && !g->col_indices)) return KB_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int device = 0;
    NA_CUDA(cudaGetDevice(&device));
    unsigned char* base = nullptr;
    const kb_status st = scratch_address(device, &base);
    if (st != KB_OK) return st;

    const int64_t n = g->n;
    const int32_t thr = opt->hub_threshold > 0 ? opt->hub_threshold : kb::kDefaultHubThreshold;
    const uint64_t cap = std::max<uint64_t>(1024, next_pow2((uint64_t)(2 * n)));
    kb::Counters* ctr = reinterpret_cast<kb::Counters*>(base + kOffCtr);

    kb::RoundParams p{};
    p.n = n;
    p.row = g->row_offsets;
    p.col = g->col_indices;
    p.lab = opt->use_edge_labels ? g->edge_labels : nullptr;
    p.prev = prev;
    p.hub_threshold = thr;
    p.mid_max = std::min(opt->small_max_degree > 0 ? opt->small_max_degree : kb::kMidDegree, thr);
    p.small_max = std::min(p.mid_max, kb::kSmallDegree);
    p.warp_verts = opt->small_task_vertices;
    p.hub_chunk = kb::kDefaultHubChunk;  // no hubs here
    p.med_split = opt->medium_split > 0 ? opt->medium_split : kb::kDefaultMedSplit;
    p.hash_mode = opt->hash_mode;
    p.epoch = 1;
    p.table = reinterpret_cast<uint64_t*>(base + kOffTable);
    p.mask = cap - 1;
    p.slot_of = reinterpret_cast<int32_t*>(base + kOffSlot);
    p.emin = reinterpret_cast<uint64_t*>(base + kOffEmin);
    p.ehigh = 0xfffffffeu;  // emin is reset to all ones below, so this round's entries win
    p.bitmap = reinterpret_cast<uint32_t*>(base + kOffBitmap);
    p.ctr = ctr;
    p.n_hubs = 0;

    // The array keeps the previous call's contents: reset what must start clean.
    // (every part of it is padded to 256 bytes)
    auto words = [](size_t bytes) { return (int64_t)((bytes + sizeof(uint4) - 1) / sizeof(uint4)); };
    const int64_t table_words = words(sizeof(uint64_t) * cap);
    reset_kernel<<<(unsigned)std::min<int64_t>((table_words + 255) / 256, 152 * 8), 256, 0, s>>>(
        reinterpret_cast<uint4*>(base), words(kOffBitmap + sizeof(uint32_t) * (size_t)((n >> 5) + 1)),
        reinterpret_cast<uint4*>(p.table), table_words, reinterpret_cast<uint4*>(p.emin),
        words(sizeof(uint64_t) * (size_t)n));
    // the degree classes: no vertex may lie above the hub threshold (no hub path
    // here) or have a negative degree.  Level i-1 must hold ids in [0, n) (they
    // index the empty-signature minima).
    kb::CheckIds ids;
    ids.a[0] = prev;
    ids.count[0] = n;
    if (opt->validate) {
        ids.a[1] = g->col_indices;
        ids.count[1] = g->m;
    }
    uint32_t* bits = reinterpret_cast<uint32_t*>(base + kOffClasses);
    const int64_t pitch = (int64_t)(up(sizeof(uint32_t) * kWords) / sizeof(uint32_t));
    uint32_t* tiles = reinterpret_cast<uint32_t*>(base + kOffTiles);
    const kb::ClassBounds bounds{p.small_max, p.mid_max, thr};
    kb::launch_classes(n, g->m, p.row, bounds, bits, pitch, tiles,
                       opt->validate ? kb::CheckRows::kAll : kb::CheckRows::kOrder, ids, kb::HubSink{}, ctr, s);
    NA_CUDA(cudaGetLastError());
    kb::Counters host_ctr{};
    NA_CUDA(cudaMemcpyAsync(&host_ctr, ctr, sizeof(host_ctr), cudaMemcpyDeviceToHost, s));
    NA_CUDA(cudaStreamSynchronize(s));
    if (host_ctr.err & kb::kErrInvalid) return KB_ERR_INVALID_ARG;
    if (host_ctr.n_class[2] > 0) return KB_ERR_INVALID_ARG;  // a degree above the hub threshold
    // the two lists share the array: together they hold at most n vertices
    p.n_mid = host_ctr.n_class[0];
    p.n_med = host_ctr.n_class[1];
    int32_t* lists = reinterpret_cast<int32_t*>(base + kOffMed);
    p.mid_v = lists;
    p.med_v = lists + p.n_mid;
    kb::launch_class_lists(n, p.row, bits, pitch, tiles, {kb::kMid, p.n_mid, lists, nullptr},
                           {kb::kMedium, p.n_med, lists + p.n_mid, nullptr}, s);

    kb::launch_keys(p, s);
    kb::launch_renumber(p, reinterpret_cast<uint2*>(base + kOffPrefix), reinterpret_cast<uint32_t*>(base + kOffScan),
                        out, nullptr, false, s);
    NA_CUDA(cudaGetLastError());
    NA_CUDA(cudaMemcpyAsync(&host_ctr, ctr, sizeof(host_ctr), cudaMemcpyDeviceToHost, s));
    NA_CUDA(cudaStreamSynchronize(s));
    if (host_ctr.err & kb::kErrTableFull) return KB_ERR_TABLE_FULL;
    if (host_ctr.err) return KB_ERR_DEVICE_CHECK;
    *count = host_ctr.count;
    return KB_OK;
}
