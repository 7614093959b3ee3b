// Host side of the SQuant library: validation, launch plans, the C ABI of include/squant.h.
#include "squant.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <list>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "squant_device.cuh"
#include "squant_stream.cuh"
#include "squant_wide.cuh"

namespace {

using sq::Item;
using sq::LayerDesc;

constexpr int kMaxSmemFallback = 232448;   // 227 KB: per-CTA opt-in limit of sm_100
constexpr int64_t kMaxChannelElems = 65535; // one-CTA paths: keeps the clamp-edge element out of every top-k (its
                                            // perturbation is <= one ulp of qmax); wider channels take the cluster
                                            // kernel, which checks every candidate against the clip range
constexpr int64_t kMaxKernels = (1 << sq::kIdxBits) - 1;   // kernels per channel: the select keys hold 18 index bits
constexpr size_t kMaxPlans = 64;
constexpr int kLongChannel = 8192;           // weights: longer channels are launched apart from the others
constexpr int kStreamKernels = 1184;         // 3x3 channels of at least as many kernels go to the streaming kernel (stream_eligible)
constexpr int kGroupedSmemGoal = 55 << 10;   // shared memory of a grouped CTA with which four of them share a multiprocessor
constexpr int kSmSmem = 228 << 10;           // shared memory of a multiprocessor; every thread block takes 1 KB of it for the system
constexpr int kBlockSmemReserved = 1 << 10;
constexpr int kWideSmemGoal = 112 << 10;     // the same of a cluster's thread block: two of them

std::mutex g_mutex;
std::atomic<int64_t> g_launches{0};
thread_local std::string t_cuda_error;

int cuda_fail(cudaError_t e, const char *what)
{
    t_cuda_error = std::string(what) + ": " + cudaGetErrorString(e);
    return SQUANT_ERR_CUDA;
}

#define SQ_CUDA(call)                                          \
    do {                                                       \
        cudaError_t e__ = (call);                              \
        if (e__ != cudaSuccess) return cuda_fail(e__, #call);  \
    } while (0)

inline int align16(int v) { return (v + 15) & ~15; }
inline int64_t align16_64(int64_t v) { return (v + 15) & ~static_cast<int64_t>(15); }

struct HostPlan {
    std::vector<LayerDesc> layers;
    std::vector<Item> items;
    int smem_bytes = 0;
    int qmax = 0;
    unsigned mode = 0;
};

// Threads that share one output channel, by channel length.
int group_size(int64_t nk)
{
    if (nk <= 1024) return 32;
    if (nk <= 2048) return 64;
    if (nk <= 4096) return 128;
    return 256;
}

int validate(const squant_layer *layers, int32_t n_layers, const squant_options *opt,
             bool need_pointers, squant_options &o)
{
    o.bits = 4;
    o.mode = SQUANT_MODE_EKC;
    o.flags = SQUANT_FLAG_NARROW_RANGE;
    if (opt) {
        o = *opt;
        if (o.mode == 0) o.mode = SQUANT_MODE_EKC;
    }
    if (n_layers < 0) return SQUANT_ERR_SHAPE;
    if (n_layers > 0 && !layers) return SQUANT_ERR_NULL;
    if (o.bits < 2 || o.bits > 8) return SQUANT_ERR_BITS;
    if (!(o.mode & SQUANT_MODE_E) || (o.mode & ~SQUANT_MODE_EKC)) return SQUANT_ERR_MODE;
    if (o.flags & ~(SQUANT_FLAG_NARROW_RANGE | SQUANT_FLAG_PACK_INT4)) return SQUANT_ERR_MODE;
    if ((o.flags & SQUANT_FLAG_PACK_INT4) && o.bits > 4) return SQUANT_ERR_BITS;
    for (int i = 0; i < n_layers; ++i) {
        const squant_layer &l = layers[i];
        if (l.cout <= 0 || l.cin <= 0 || l.kh <= 0 || l.kw <= 0) return SQUANT_ERR_SHAPE;
        const int64_t k = static_cast<int64_t>(l.kh) * l.kw;
        const int64_t nk = k * l.cin;
        if (k > 65535 || nk > (1ll << 30)) return SQUANT_ERR_SHAPE;
        if (static_cast<int64_t>(l.cout) * nk > (1ll << 40)) return SQUANT_ERR_SHAPE;
        if (l.cin > kMaxKernels) return SQUANT_ERR_TOO_WIDE;
        if (need_pointers) {
            if (!l.w || !l.codes || !l.scales) return SQUANT_ERR_NULL;
            if ((reinterpret_cast<uintptr_t>(l.w) & 3) || (reinterpret_cast<uintptr_t>(l.scales) & 3) ||
                (reinterpret_cast<uintptr_t>(l.kernel_err) & 3) ||
                (reinterpret_cast<uintptr_t>(l.channel_err) & 3) || (reinterpret_cast<uintptr_t>(l.dequant) & 3) ||
                (reinterpret_cast<uintptr_t>(l.scales_in) & 3) || (reinterpret_cast<uintptr_t>(l.dequant_bf16) & 1))
                return SQUANT_ERR_ALIGN;
        }
        // supplied scales: the element-wise channel step of E|C on larger kernels is not built for clipping
        if (l.scales_in && k > 1 && (o.mode & SQUANT_MODE_C) && !(o.mode & SQUANT_MODE_K)) return SQUANT_ERR_MODE;
    }
    return SQUANT_OK;
}

// Layout of a channel with staged weights and per-kernel arrays: E|C on
// larger kernels, 1x1 rows beyond the registers of one thread block.
void layout_staged(const squant_layer &l, LayerDesc &d, unsigned mode)
{
    d.g = group_size(d.NK);
    d.g_shift = 0;
    while ((1 << d.g_shift) < d.g) ++d.g_shift;
    int off = align16(4 * d.NK);              // staged weights
    d.off_codes = off; off += align16(d.NK);  // staged codes
    const bool ec_only = (mode & SQUANT_MODE_C) && !(mode & SQUANT_MODE_K);   // elements are the candidates
    if ((d.K == 1 || ec_only) && !l.scales_in) {   // perturbations overwrite the weights
        d.off_ev = 0; d.off_vv = 0; d.off_vi = 0;
    } else {
        d.off_ev = off; off += align16(4 * d.N);
        d.off_vv = off; off += align16(4 * d.N);
        d.off_vi = off; off += align16(2 * d.N);
    }
    d.off_hist = off; off += 4 * sq::kHistBins;
    d.off_red = off; off += 256;
    d.slice_bytes = off;
}

// 1x1: every row of weights, error sums and codes starts on a vector.
int regular_rows(const LayerDesc &d)
{
    return (d.N & 3) == 0 && (reinterpret_cast<uintptr_t>(d.w) & 15) == 0 && (reinterpret_cast<uintptr_t>(d.kerr) & 15) == 0 &&
           (reinterpret_cast<uintptr_t>(d.codes) & 3) == 0;
}

// Device-side descriptor of one layer: group size and the layout of a group's shared-memory
// slice.  Returns the dynamic shared memory one CTA needs for this layer.  spread_rows, spread_kernels: 1, 2 or
// 4 times the threads per channel that use them best.
int64_t layout_layer(const squant_layer &l, LayerDesc &d, unsigned mode, unsigned flags, int spread_rows = 1, int spread_kernels = 1)
{
    d.w = l.w; d.codes = l.codes; d.scales = l.scales; d.kerr = l.kernel_err; d.cerr = l.channel_err; d.deq = l.dequant;
    d.sin = l.scales_in; d.deq16 = l.dequant_bf16;
    d.M = l.cout; d.N = l.cin; d.K = l.kh * l.kw; d.NK = d.N * d.K;
    d.g = group_size(d.NK);
    d.g_shift = 0;
    while ((1 << d.g_shift) < d.g) ++d.g_shift;
    // No layout holds a channel in less than 5 B a weight; the sizes below are 32-bit numbers.
    if (5ll * d.NK > kMaxSmemFallback) return 5ll * d.NK;
    // Depthwise layers (one kernel per output channel) with plain outputs: a whole channel per thread.
    // SQuant-C is void there once SQuant-K has run; without K (E|C) the channel step is real.
    if (d.N == 1 && d.K <= 64 && !l.scales_in && !l.dequant && !l.dequant_bf16 && !(flags & SQUANT_FLAG_PACK_INT4) &&
        ((mode & SQUANT_MODE_K) || !(mode & SQUANT_MODE_C))) {
        d.g = 1;
        d.g_shift = 0;
        d.off_codes = 4 * d.K; d.off_ev = 0; d.off_vv = 0; d.off_vi = 0; d.off_hist = 0; d.off_red = 0;
        d.slice_bytes = align16(5 * d.K);
        return static_cast<int64_t>(sq::kCtaThreads) * d.slice_bytes;
    }
    if (d.K == 1) {   // a channel that fits the registers of at most one thread block: no staging
        const int first = static_cast<int>((reinterpret_cast<uintptr_t>(l.w) >> 2) & 3);
        const int vecs = (d.N & 3) ? (d.N + 6) >> 2 : (d.N + first + 3) >> 2;   // of the most misaligned row
        int g = sq::row_group(vecs);
        if (g) {
            for (int s = 1; s < spread_rows && g < sq::kCtaThreads && 2 * g <= vecs; s *= 2) g *= 2;
            d.g = g;
            d.g_shift = 0;
            while ((1 << d.g_shift) < d.g) ++d.g_shift;
            d.off_codes = 0; d.off_ev = 0; d.off_vv = 0; d.off_vi = vecs; d.off_hist = 0; d.off_red = 0;
            d.slice_bytes = align16(sq::row_bytes(g, vecs));
            return static_cast<int64_t>(sq::kCtaThreads / d.g) * d.slice_bytes;
        }
    }
    if (d.K > 1 && !((mode & SQUANT_MODE_C) && !(mode & SQUANT_MODE_K))) {   // kernels: a thread settles up to four of them (larger than 3x3: two)
        const int per = std::max((d.K <= 9 ? 4 : 2) / spread_kernels, 1);
        int g = 32;
        while (g < sq::kCtaThreads && (per * g < d.N || sq::kCtaThreads / g * sq::conv_bytes(g, d.NK, d.K) > kGroupedSmemGoal)) g *= 2;
        d.g = g;
        d.g_shift = 0;
        while ((1 << d.g_shift) < d.g) ++d.g_shift;
        d.off_codes = 0; d.off_ev = 0; d.off_vv = 0; d.off_vi = 0; d.off_hist = 0; d.off_red = 0;
        d.slice_bytes = align16(sq::conv_bytes(g, d.NK, d.K));
        return static_cast<int64_t>(sq::kCtaThreads / d.g) * d.slice_bytes;
    }
    layout_staged(l, d, mode);
    return static_cast<int64_t>(sq::kCtaThreads / d.g) * d.slice_bytes;
}

// Work list in a table (global-memory variant): CTA-sized items, heaviest first.
int build_plan(const squant_layer *layers, int32_t n_layers, const squant_options &o, int max_smem,
               HostPlan &p)
{
    p.qmax = (1 << (o.bits - 1)) - 1;
    p.mode = o.mode | ((o.flags & SQUANT_FLAG_PACK_INT4) ? sq::kModePackInt4 : 0u) |
             ((o.flags & SQUANT_FLAG_NARROW_RANGE) ? 0u : sq::kModeWideRange);
    p.layers.resize(n_layers);
    p.smem_bytes = 0;
    struct Batch { int64_t work; int layer; int ch0; };
    std::vector<Batch> batches;
    for (int i = 0; i < n_layers; ++i) {
        LayerDesc &d = p.layers[i];
        const int64_t cta_smem = layout_layer(layers[i], d, o.mode, o.flags);
        if (cta_smem > max_smem) return SQUANT_ERR_TOO_WIDE;
        const int groups = sq::kCtaThreads / d.g;
        LayerDesc staged = d;
        layout_staged(layers[i], staged, o.mode);   // (the limit: a channel staged with its per-kernel arrays)
        if (static_cast<int64_t>(sq::kCtaThreads / staged.g) * staged.slice_bytes > max_smem) return SQUANT_ERR_TOO_WIDE;
        if (cta_smem > p.smem_bytes) p.smem_bytes = static_cast<int>(cta_smem);
        for (int c = 0; c < d.M; c += groups) {
            const int nch = (d.M - c < groups) ? d.M - c : groups;
            batches.push_back({static_cast<int64_t>(nch) * d.NK, i, c});
        }
    }
    // Heaviest CTAs first, so that the tail of the launch is made of light ones.
    std::stable_sort(batches.begin(), batches.end(),
                     [](const Batch &a, const Batch &b) { return a.work > b.work; });
    p.items.resize(batches.size());
    for (size_t i = 0; i < batches.size(); ++i) p.items[i] = {batches[i].layer, batches[i].ch0};
    return SQUANT_OK;
}

// Scratch memory of the streaming kernel (what SQuant-C needs of every kernel one step later: four sets of
// 18 KB per thread block; the launch's work counters) is shared by the plan that launches with it and by every
// graph that captured such a launch, and goes with the last of them.  A graph lets go inside a CUDA callback,
// where no CUDA call is allowed: the memory is then listed here and freed by the next call that quantizes device
// or host buffers and is not being captured, or by squant_shutdown (cudaFree waits for the device, so no launch
// still uses it).
struct DeadScratch {
    std::mutex mutex;
    std::vector<void *> list;
    std::atomic<bool> any{false};
};

DeadScratch &dead_scratch()
{
    static DeadScratch *d = new DeadScratch;   // outlives graphs that are destroyed at exit
    return *d;
}

void scratch_unused(void *p)
{
    DeadScratch &d = dead_scratch();
    std::lock_guard<std::mutex> lock(d.mutex);
    try {
        d.list.push_back(p);
        d.any.store(true, std::memory_order_release);
    } catch (const std::bad_alloc &) {   // host memory is exhausted: left to the end of the process
    }
}

void free_dead_scratch()
{
    DeadScratch &d = dead_scratch();
    std::vector<void *> list;
    {
        std::lock_guard<std::mutex> lock(d.mutex);
        list.swap(d.list);
        d.any.store(false, std::memory_order_relaxed);
    }
    // captures of other streams may be under way; they do not depend on this memory
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    for (void *p : list)
        if (cudaFree(p) != cudaSuccess) {
            cudaGetLastError();   // not the caller's error: it stays listed
            scratch_unused(p);
        }
    cudaThreadExchangeStreamCaptureMode(&mode);
}

// The same unless `stream` is being captured; costs nothing where there is nothing to free.
int free_dead_scratch(cudaStream_t stream)
{
    if (!dead_scratch().any.load(std::memory_order_acquire)) return SQUANT_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    SQ_CUDA(cudaStreamIsCapturing(stream, &cap));
    if (cap == cudaStreamCaptureStatusNone) free_dead_scratch();
    return SQUANT_OK;
}

struct StreamScratch {
    unsigned char *mem;
    size_t area;   // bytes before the work counters
    int device;
    StreamScratch(unsigned char *m, size_t a, int d) : mem(m), area(a), device(d) {}
    StreamScratch(const StreamScratch &) = delete;
    StreamScratch &operator=(const StreamScratch &) = delete;
    ~StreamScratch() { scratch_unused(mem); }
    unsigned *work() const { return reinterpret_cast<unsigned *>(mem + area); }
};
using ScratchRef = std::shared_ptr<StreamScratch>;

std::vector<std::weak_ptr<StreamScratch>> g_scratch;   // every area in use; guarded by g_mutex

// A new area on the current device; its work counters are zeroed in the order of `stream`.  Leaves `out` empty
// where there is no memory.
int new_scratch(int device, int sms, cudaStream_t stream, ScratchRef &out)
{
    const size_t area = static_cast<size_t>(sms) * sq::kStreamHeldSets * sq::kStreamHeldBytes;
    void *mem = nullptr;
    if (cudaMalloc(&mem, area + sq::kStreamWorkBytes) != cudaSuccess) {
        cudaGetLastError();   // reported by the return code of the call, not left pending
        return SQUANT_OK;
    }
    ScratchRef s = std::make_shared<StreamScratch>(static_cast<unsigned char *>(mem), area, device);
    SQ_CUDA(cudaMemsetAsync(s->work(), 0, sq::kStreamWorkBytes, stream));
    g_scratch.erase(std::remove_if(g_scratch.begin(), g_scratch.end(), [](const std::weak_ptr<StreamScratch> &w) { return w.expired(); }),
                    g_scratch.end());
    g_scratch.push_back(s);
    out = std::move(s);
    return SQUANT_OK;
}

void CUDART_CB release_scratch(void *p) { delete static_cast<ScratchRef *>(p); }

// The graph that is being captured takes a share in the scratch memory that its kernel node points to.
int share_with_graph(const ScratchRef &scratch, cudaGraph_t graph)
{
    auto *share = new (std::nothrow) ScratchRef(scratch);
    if (!share) return SQUANT_ERR_NOMEM;
    cudaUserObject_t obj = nullptr;
    const cudaError_t e = cudaUserObjectCreate(&obj, share, release_scratch, 1, cudaUserObjectNoDestructorSync);
    if (e != cudaSuccess) {
        delete share;
        return cuda_fail(e, "cudaUserObjectCreate");
    }
    const cudaError_t r = cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove);
    if (r != cudaSuccess) {
        cudaUserObjectRelease(obj, 1);
        return cuda_fail(r, "cudaGraphRetainUserObject");
    }
    return SQUANT_OK;
}

// Launch tables for the parameter-space variant: layers ordered by the work of one of their
// CTAs (heaviest first, so the tail of the launch is made of light CTAs), at most
// kMaxParamLayers per launch.
struct ParamPlan {
    struct Grouped { sq::LaunchTable table; int grid, smem; sq::Scales scales; };
    std::vector<Grouped> grouped;   // grouped kernel: one CTA per item
    int qmax = 0;
    unsigned mode = 0;
    // cluster kernel (channels wider than one CTA): one launch per layer
    struct Wide { LayerDesc d; int cluster, kpc, smem; };
    std::vector<Wide> wide;
    // row kernel (1x1 rows too long for a group): one item per output channel
    enum RowForm { kRow512, kLong512, kRow256 };   // row_body with 512 threads, long_row_body with 512, row_body with 256
    struct Rows { sq::LaunchTable table; RowForm form; int grid, smem; };
    std::vector<Rows> rows;
    // streaming kernel (layers of long 3x3 channels): one item per output channel
    struct Stream {
        sq::LaunchTable table;
        int items = 0, nk_max = 0, n_max = 0;
        bool out = false;                     // packed or dequantized outputs wanted
        ScratchRef scratch;                   // allocated at the plan's first launch outside a capture
        // Layers with packed or dequantized outputs can also go to the grouped kernel, which needs no scratch:
        // where it cannot be allocated (a full device, the plan's first launch inside a stream capture).
        sq::LaunchTable grouped;
        int grouped_grid = 0, grouped_smem = 0;
    };
    mutable std::vector<Stream> streams;
};

// Layers the streaming kernel takes: 3x3 channels so long that no four CTAs of the grouped kernel fit a
// multiprocessor (kStreamKernels input channels on), input channels a multiple of four and one quad of kernels per
// quantizer thread, SQuant-K on, absmax scales, and its buffers fit the shared memory of one SM.
// Grouped / streaming kernel in us, cold and with the events' own time, at 1152, 1184, 1280, 1408 and 2048 input channels:
//   2048 output channels, plain codes   56 / 60, 58 / 60, 67 / 60, 71 / 63, 99 / 69
//                         packed codes          60 / 69, 69 / 71, 74 / 70, 106 / 79
//                         bf16 output           68 / 78, 75 / 78, 81 / 79, 118 / 89
//   512 output channels,  plain codes   25 / 28, 25 / 27, 32 / 28, 34 / 28, 40 / 32
//                         packed codes          28 / 30, 32 / 32, 33 / 31, 42 / 36
//   148 output channels   plain codes   19 / 17, 20 / 17, 20 / 17, 20 / 20, 22 / 20
// (with further outputs both kernels are even at about 1350; the line is the plain codes').
bool stream_eligible(const squant_layer &l, const LayerDesc &d, const squant_options &o, int max_smem)
{
    if (d.K != 9 || (d.N & 3) != 0 || d.N < kStreamKernels) return false;
    if (!(o.mode & SQUANT_MODE_K) || l.scales_in) return false;
    if ((reinterpret_cast<uintptr_t>(l.w) & 15) || (reinterpret_cast<uintptr_t>(l.codes) & 15)) return false;
    if (d.N > 4 * sq::kStreamQuantThreads) return false;
    return sq::stream_layout(d.NK, d.N).total <= max_smem;
}

// Launch table of n layers; work items are CTAs of the grouped kernel or single output channels.  Returns
// the number of items.
int fill_table(sq::LaunchTable &t, const std::vector<LayerDesc> &descs, const int *layers, int n, bool ctas)
{
    std::memset(&t, 0, sizeof(t));
    t.n_layers = n;
    for (int step = 1; step < n; step <<= 1) t.top_step = step;
    int items = 0;
    for (int j = 0; j < n; ++j) {
        const LayerDesc &d = descs[layers[j]];
        const int groups = ctas ? sq::kCtaThreads / d.g : 1;
        t.layers[j] = d;
        t.first_item[j] = items;
        items += (d.M + groups - 1) / groups;
    }
    for (int j = n; j <= sq::kMaxParamLayers; ++j) t.first_item[j] = items;
    return items;
}

// kernels: SQUANT_KERNEL_* of every layer, or null.
int build_param_plan(const squant_layer *layers, int32_t n_layers, const squant_options &o,
                     int max_smem, int sms, ParamPlan &p, int32_t *kernels = nullptr)
{
    p.qmax = (1 << (o.bits - 1)) - 1;
    p.mode = o.mode | ((o.flags & SQUANT_FLAG_PACK_INT4) ? sq::kModePackInt4 : 0u) |
             ((o.flags & SQUANT_FLAG_NARROW_RANGE) ? 0u : sq::kModeWideRange);
    const bool pack = (o.flags & SQUANT_FLAG_PACK_INT4) != 0;
    std::vector<LayerDesc> descs(n_layers);
    std::vector<int> order, streamed[2], rows;
    for (int i = 0; i < n_layers; ++i) {
        const int64_t cta_smem = layout_layer(layers[i], descs[i], o.mode, o.flags);
        if (cta_smem > max_smem || descs[i].NK > kMaxChannelElems) {
            // a cluster of 2, 4 or 8 CTAs per output channel, each with an even number of kernels (packed codes of a
            // run start on a byte), of 1x1 rows a multiple of four (a run starts on a vector)
            if ((o.mode & SQUANT_MODE_C) && !(o.mode & SQUANT_MODE_K) && descs[i].K > 1) return SQUANT_ERR_TOO_WIDE;   // E|C selects among elements: one CTA only
            // (the limit: what eight of them hold at 5 B a weight and 10 B a larger kernel)
            ParamPlan::Wide w{descs[i], 0, 0, 0};
            const int64_t k8 = (((descs[i].N + 7) / 8) + 1) & ~1;
            if (align16_64(4 * k8 * descs[i].K) + align16_64(k8 * descs[i].K) + (descs[i].K > 1 ? 2 * align16_64(4 * k8) + align16_64(2 * k8) : 0) + 2304 > max_smem)
                return SQUANT_ERR_TOO_WIDE;
            // two thread blocks per multiprocessor if the channel can be cut that small: while one waits for its
            // weights or for its cluster the other works.  Few 1x1 rows take clusters of four at least (46,500 weights, in
            // clusters of two / four: 16 rows 17.8 / 14.4 us on a B200, 64 18.5 / 18.0, 74 18.5 / 23.9, 200 39.9 / 47.2).
            const int least = descs[i].K == 1 && 16ll * descs[i].M <= 7ll * sms ? 4 : 2;
            for (int goal = kWideSmemGoal;; goal = max_smem) {
                for (int c = least; c <= sq::kWideMaxCluster && !w.cluster; c *= 2) {
                    const int unit = descs[i].K == 1 ? 4 : 2;
                    const int kpc = ((descs[i].N + c - 1) / c + unit - 1) / unit * unit;
                    const int64_t bytes = sq::wide_bytes(kpc, descs[i].K, pack);
                    if (bytes <= goal) { w.cluster = c; w.kpc = kpc; w.smem = static_cast<int>(bytes); }
                }
                if (w.cluster || goal == max_smem) break;
            }
            if (!w.cluster) return SQUANT_ERR_TOO_WIDE;
            w.d.off_vi = (w.kpc + 6) >> 2;
            w.d.off_ev = regular_rows(w.d);
            p.wide.push_back(w);
            if (kernels) kernels[i] = SQUANT_KERNEL_CLUSTER;
            continue;
        }
        if (stream_eligible(layers[i], descs[i], o, max_smem)) {
            const squant_layer &l = layers[i];
            streamed[l.dequant || l.dequant_bf16 || (o.flags & SQUANT_FLAG_PACK_INT4) ? 1 : 0].push_back(i);
            if (kernels) kernels[i] = SQUANT_KERNEL_STREAM;
            continue;
        }
        if (descs[i].K == 1 && descs[i].off_hist != 0 && descs[i].N <= sq::kRowBlockElems) {   // too long for a group
            rows.push_back(i);
            if (kernels) kernels[i] = SQUANT_KERNEL_ROW;
            continue;
        }
        order.push_back(i);
        if (kernels) kernels[i] = SQUANT_KERNEL_GROUPED;
    }
    // Long rows, a thread block per output channel, in one of three forms.  row_body holds 5 B of shared memory a
    // weight, long_row_body 4.  What counts is how many threads a multiprocessor holds and over how many vectors a
    // thread spreads the code that runs once.
    //   - More than two and a quarter rows a multiprocessor, so short that three thread blocks of 256 threads fit one
    //     (14.8 K weights): row_body with 256 threads.
    //   - More rows than multiprocessors of which two thread blocks fit one only in long_row_body (22 to 27 K
    //     weights), neither packed codes nor scales of their own: long_row_body with 512 threads.
    //   - All others row_body with 512 threads.
    // us a call on a B200, row_body with 256 threads / with 512 / long_row_body with 512:
    //   rows of 9000       300 12.5 / 12.3 / 14.4, 400 14.4 / 15.8 / 18.7, 4096 69.9 / 94.1 / 117
    //     packed codes     2000 40.2 / 51.2 / 69.2
    //     their own scales 1500 39.4 / 47.4 / 65.7
    //   of 12,000          100 12.9 / 10.3 / 12.8, 500 19.5 / 20.5 / 25.0, 4096 89.6 / 105 / 128
    //   of 14,100          4096 106.7 / 124.1 / 142.3
    //   of 15,001          4096 135.3 / 127.7 / 153.8
    //   of 22,100          1000 - / 49.6 / 57.1
    //   of 25,001          300 - / 30.7 / 30.8, 2000 - / 127.2 / 110.7
    //   of 30,000          300 - / 31.2 / 36.9
    const auto blocks = [&](int bytes) { return kSmSmem / (bytes + kBlockSmemReserved); };   // on a multiprocessor
    const auto small_blocks = [&](int i) {   // of 256 threads, none if the row is too long for them
        return descs[i].N > 4 * 2 * sq::kRowVecs * 256 ? 0 : std::min(4, blocks(sq::row_bytes(256, (descs[i].N + 6) >> 2, sq::kBlock)));
    };
    const auto only_long = [&](int i) {
        const int vecs = (descs[i].N + 6) >> 2;
        return !pack && !descs[i].sin && blocks(sq::row_bytes(512, vecs, sq::kBlock)) < 2 && blocks(sq::long_row_bytes(512, vecs, false, sq::kBlock)) >= 2;
    };
    int64_t small = 0, longer = 0;   // rows
    for (int i : rows) {
        if (small_blocks(i) >= 3) small += descs[i].M;
        if (only_long(i)) longer += descs[i].M;
    }
    const auto form_of = [&](int i) {
        if (small_blocks(i) >= 3 && 4 * small > 9ll * sms) return ParamPlan::kRow256;
        return only_long(i) && longer > sms ? ParamPlan::kLong512 : ParamPlan::kRow512;
    };
    // Rows of 256 threads of which four thread blocks fit a multiprocessor have a launch apart from those of which three do.
    const auto launch_of = [&](int i) { return form_of(i) == ParamPlan::kRow256 ? 8 - small_blocks(i) : static_cast<int>(form_of(i)); };
    std::stable_sort(rows.begin(), rows.end(), [&](int a, int b) {   // by form, longest first
        return launch_of(a) != launch_of(b) ? launch_of(a) < launch_of(b) : descs[a].N > descs[b].N;
    });
    for (size_t base = 0; base < rows.size();) {
        const ParamPlan::RowForm form = form_of(rows[base]);
        size_t n = 0;
        int smem = 0;
        while (base + n < rows.size() && n < sq::kMaxParamLayers && launch_of(rows[base + n]) == launch_of(rows[base])) {
            LayerDesc &d = descs[rows[base + n]];
            d.off_vi = (d.N + 6) >> 2;
            d.off_ev = regular_rows(d);
            smem = std::max(smem, form == ParamPlan::kLong512 ? sq::long_row_bytes(512, d.off_vi, false, sq::kBlock)
                                                              : sq::row_bytes(form == ParamPlan::kRow512 ? 512 : 256, d.off_vi, sq::kBlock));
            ++n;
        }
        p.rows.emplace_back();
        ParamPlan::Rows &r = p.rows.back();
        r.grid = fill_table(r.table, descs, rows.data() + base, static_cast<int>(n), false);
        r.form = form;
        r.smem = smem;
        base += n;
    }
    for (int kind = 1; kind >= 0; --kind) {
        const std::vector<int> &list = streamed[kind];
        for (size_t base = 0; base < list.size(); base += sq::kMaxParamLayers) {
            const int n = static_cast<int>(std::min<size_t>(list.size() - base, sq::kMaxParamLayers));
            p.streams.emplace_back();
            ParamPlan::Stream &st = p.streams.back();
            st.items = fill_table(st.table, descs, list.data() + base, n, false);
            st.grouped_grid = fill_table(st.grouped, descs, list.data() + base, n, true);
            for (int j = 0; j < n; ++j) {
                const LayerDesc &d = descs[list[base + j]];
                st.nk_max = std::max(st.nk_max, d.NK);
                st.n_max = std::max(st.n_max, d.N);
                st.grouped_smem = std::max(st.grouped_smem, sq::kCtaThreads / d.g * d.slice_bytes);
            }
            st.out = kind != 0;
        }
    }
    // A launch whose warps do not fill the GPU takes the time of one channel, so its channels get twice or
    // four times the threads (up to 32 warps per multiprocessor for 1x1 rows: 3531 rows of 461 weights
    // 27.0 -> 17.4 us, MobileNetV2 shapes at half width 12.3 -> 8.0; half as many for larger kernels: 256x256x3x3
    // 7.3 -> 6.4, whereas 512x512x3x3 is slower with twice the threads, 10.5 against 9.4 us).
    int64_t warps = 0;
    for (int i : order) warps += (static_cast<int64_t>(descs[i].M) * descs[i].g + 31) / 32;
    int spread[2] = {1, 1};
    for (int k = 0; k < 2; ++k)
        while (spread[k] < 4 && 2 * spread[k] * warps <= static_cast<int64_t>(sms) * (k ? 16 : 32)) spread[k] *= 2;
    if (spread[0] > 1)
        for (int i : order) layout_layer(layers[i], descs[i], o.mode, o.flags, spread[0], spread[1]);
    // The grouped kernel takes the rest, layers of long channels in launches of their own: their CTAs need
    // shared memory that would cost the others their fourth CTA per multiprocessor.
    // Estimated duration of one CTA of the layer.  Kernel sizes without a body of their own take the
    // general per-thread path, which is latency-bound and far slower per weight, so those start first.
    auto cta_work = [&](int i) {
        const LayerDesc &d = descs[i];
        const int64_t groups = sq::kCtaThreads / d.g;
        const bool own = d.K == 1 || d.K == 3 || d.K == 7 || d.K == 9;
        return (groups < d.M ? groups : d.M) * (own ? d.NK : static_cast<int64_t>(d.NK) * 64 * d.K);
    };
    auto is_long = [&](int i) { return descs[i].NK > kLongChannel; };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return is_long(a) != is_long(b) ? is_long(a) : cta_work(a) > cta_work(b);
    });
    for (size_t base = 0; base < order.size();) {
        size_t n = 1;
        while (base + n < order.size() && n < sq::kMaxParamLayers && is_long(order[base + n]) == is_long(order[base])) ++n;
        p.grouped.emplace_back();
        ParamPlan::Grouped &gl = p.grouped.back();
        gl.smem = 0;
        size_t own = 0;   // layers with scales of their own
        for (size_t j = 0; j < n; ++j) {
            const LayerDesc &d = descs[order[base + j]];
            own += d.sin ? 1 : 0;
            gl.smem = std::max(gl.smem, sq::kCtaThreads / d.g * d.slice_bytes);
        }
        gl.scales = own == 0 ? sq::kAbsmax : (own == n ? sq::kOwnScales : sq::kEither);
        gl.grid = fill_table(gl.table, descs, order.data() + base, static_cast<int>(n), true);
        base += n;
    }
    return SQUANT_OK;
}

// Launch tables are plain host data; the most recent ones are kept, keyed by the exact
// descriptors and options, so that a repeated call only enqueues its kernel(s).
struct CachedPlan {
    int device = -1;
    std::string key;
    ParamPlan plan;
};

std::list<CachedPlan> g_plans;              // most recently used first
std::vector<int> g_smem_limit_by_device;   // opt-in limit set on the kernels, per device
std::vector<int> g_sm_count_by_device;     // multiprocessors, per device

std::string plan_key(const squant_layer *layers, int32_t n_layers, const squant_options &o)
{
    std::string k(reinterpret_cast<const char *>(&o), sizeof(o));
    k.append(reinterpret_cast<const char *>(layers), sizeof(squant_layer) * static_cast<size_t>(n_layers));
    return k;
}

int device_smem_limit(int device, int &limit)
{
    if (static_cast<int>(g_smem_limit_by_device.size()) <= device)
        g_smem_limit_by_device.resize(device + 1, 0);
    if (g_smem_limit_by_device[device] == 0) {
        int v = 0;
        SQ_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
        for (auto kernel : {sq::squant_model_kernel<sq::kAbsmax>, sq::squant_model_kernel<sq::kOwnScales>, sq::squant_model_kernel<sq::kEither>})
            SQ_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        for (auto kernel : {sq::squant_table_kernel<sq::kAbsmax>, sq::squant_table_kernel<sq::kOwnScales>})
            SQ_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        SQ_CUDA(cudaFuncSetAttribute((sq::squant_row_kernel<256, false>),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        SQ_CUDA(cudaFuncSetAttribute((sq::squant_row_kernel<512, true>),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        SQ_CUDA(cudaFuncSetAttribute((sq::squant_row_kernel<512, false>),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        SQ_CUDA(cudaFuncSetAttribute(sq::squant_wide_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        SQ_CUDA(cudaFuncSetAttribute(sq::squant_stream_kernel<false>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        SQ_CUDA(cudaFuncSetAttribute(sq::squant_stream_kernel<true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, v));
        int sms = 0;
        SQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
        if (static_cast<int>(g_sm_count_by_device.size()) <= device) g_sm_count_by_device.resize(device + 1, 0);
        g_sm_count_by_device[device] = sms;
        g_smem_limit_by_device[device] = v;
    }
    limit = g_smem_limit_by_device[device];
    return SQUANT_OK;
}

int get_plan(const squant_layer *layers, int32_t n_layers, const squant_options &o, const ParamPlan *&out)
{
    int device = 0;
    SQ_CUDA(cudaGetDevice(&device));
    std::string key = plan_key(layers, n_layers, o);
    for (auto it = g_plans.begin(); it != g_plans.end(); ++it) {
        if (it->device == device && it->key == key) {
            g_plans.splice(g_plans.begin(), g_plans, it);
            out = &g_plans.front().plan;
            return SQUANT_OK;
        }
    }
    int limit = 0;
    int rc = device_smem_limit(device, limit);
    if (rc) return rc;
    CachedPlan cp;
    cp.device = device;
    cp.key = std::move(key);
    rc = build_param_plan(layers, n_layers, o, limit, std::max(g_sm_count_by_device[device], 1), cp.plan);
    if (rc) return rc;
    if (g_plans.size() >= kMaxPlans) g_plans.pop_back();
    g_plans.push_front(std::move(cp));
    out = &g_plans.front().plan;
    return SQUANT_OK;
}

// Plans of a host-buffer call, one per chunk of layers; apart from those of device calls, of which a few large models in
// host memory would leave none cached.  The chunks run one after the other and every call ends with its work done, so one
// scratch area per device serves all of them.
struct HostCall {
    int device = -1;
    std::string key;
    std::vector<ParamPlan> chunks;
};
constexpr size_t kMaxHostCalls = 8;
std::list<HostCall> g_host_calls;         // most recently used first
std::vector<ScratchRef> g_host_scratch;   // per device

int get_host_plans(const std::vector<squant_layer> &layers, const std::vector<int> &chunk_first, const squant_options &o, int device, HostCall *&out)
{
    std::string key = plan_key(layers.data(), static_cast<int32_t>(layers.size()), o);   // (the chunks follow from the sizes)
    for (auto it = g_host_calls.begin(); it != g_host_calls.end(); ++it)
        if (it->device == device && it->key == key) {
            g_host_calls.splice(g_host_calls.begin(), g_host_calls, it);
            out = &g_host_calls.front();
            return SQUANT_OK;
        }
    int limit = 0;
    int rc = device_smem_limit(device, limit);
    if (rc) return rc;
    HostCall hc;
    hc.device = device;
    hc.key = std::move(key);
    hc.chunks.resize(chunk_first.size() - 1);
    for (size_t c = 0; c < hc.chunks.size(); ++c) {
        rc = build_param_plan(layers.data() + chunk_first[c], chunk_first[c + 1] - chunk_first[c], o, limit,
                              std::max(g_sm_count_by_device[device], 1), hc.chunks[c]);
        if (rc) return rc;
    }
    if (g_host_calls.size() >= kMaxHostCalls) g_host_calls.pop_back();
    g_host_calls.push_front(std::move(hc));
    out = &g_host_calls.front();
    return SQUANT_OK;
}

int launch_plan(const ParamPlan &p, cudaStream_t stream)
{
    const int freed = free_dead_scratch(stream);   // of graphs and of plans that have left the cache
    if (freed) return freed;
    // The row and cluster kernels may start before the launch in front of them has ended (see next_launch_may_start).
    // Not the streaming kernels, which may share a scratch area, nor the grouped one (the wait at its end would cost
    // it registers), nor what a graph captures.
    const size_t plain = std::max<size_t>(p.streams.size() + p.grouped.size(), 1), launches = p.streams.size() + p.grouped.size() + p.rows.size() + p.wide.size();
    size_t j = 0;   // of this call's launches
    bool overlap = false;
    if (launches > plain) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        SQ_CUDA(cudaStreamIsCapturing(stream, &cap));
        overlap = cap == cudaStreamCaptureStatusNone;
    }
    const auto early = [&](size_t i) { return overlap && i >= plain; };
    const auto mode = [&] { return p.mode | (early(j) ? sq::kModeMayStartEarly : 0u); };
    // long 3x3 channels first: one persistent CTA per multiprocessor
    for (ParamPlan::Stream &st : p.streams) {
        int device = 0;
        SQ_CUDA(cudaGetDevice(&device));
        const int sms = std::max(g_sm_count_by_device[device], 1);
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        cudaGraph_t graph = nullptr;
        SQ_CUDA(cudaStreamGetCaptureInfo_v2(stream, &cap, nullptr, &graph, nullptr, nullptr));
        const bool capturing = cap == cudaStreamCaptureStatusActive;
        ScratchRef scratch = st.scratch;
        if (!scratch && (!st.out || !capturing)) {
            const int rc = new_scratch(device, sms, stream, scratch);
            if (rc) return rc;
            if (!scratch && !st.out) return SQUANT_ERR_NOMEM;
            if (!capturing) st.scratch = scratch;   // (of a capture: zeroed by the graph, so the graph's alone)
        }
        if (scratch && capturing) {
            const int rc = share_with_graph(scratch, graph);
            if (rc) return rc;
        }
        if (scratch) {
            const int grid = std::min(st.items, sms), smem = sq::stream_layout(st.nk_max, st.n_max).total;
            auto kernel = st.out ? sq::squant_stream_kernel<true> : sq::squant_stream_kernel<false>;
            kernel<<<grid, sq::kStreamThreads, smem, stream>>>(st.table, p.qmax, p.mode, st.items, st.nk_max, st.n_max, scratch->mem, scratch->work());
        } else {
            sq::squant_model_kernel<sq::kAbsmax><<<st.grouped_grid, sq::kCtaThreads, st.grouped_smem, stream>>>(st.grouped, p.qmax, p.mode);
        }
        SQ_CUDA(cudaGetLastError());
        g_launches.fetch_add(1, std::memory_order_relaxed);
        ++j;
    }
    const auto launch = [&](auto kernel, int grid, int threads, int smem, int cluster, const auto &...args) -> int {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(grid));
        cfg.blockDim = dim3(static_cast<unsigned>(threads));
        cfg.dynamicSmemBytes = static_cast<size_t>(smem);
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        if (cluster > 1) {
            attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
            attr[cfg.numAttrs].val.clusterDim.x = static_cast<unsigned>(cluster);
            attr[cfg.numAttrs].val.clusterDim.y = 1;
            attr[cfg.numAttrs].val.clusterDim.z = 1;
            ++cfg.numAttrs;
        }
        if (early(j)) {
            attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
            ++cfg.numAttrs;
        }
        cfg.attrs = attr;
        void *const argv[] = {const_cast<void *>(static_cast<const void *>(&args))...};   // (of the kernels' own types)
        SQ_CUDA(cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kernel), const_cast<void **>(argv)));
        g_launches.fetch_add(1, std::memory_order_relaxed);
        ++j;
        return SQUANT_OK;
    };
    for (const ParamPlan::Grouped &gl : p.grouped) {
        auto kernel = gl.scales == sq::kAbsmax ? sq::squant_model_kernel<sq::kAbsmax>
                      : gl.scales == sq::kOwnScales ? sq::squant_model_kernel<sq::kOwnScales> : sq::squant_model_kernel<sq::kEither>;
        const int rc = launch(kernel, gl.grid, sq::kCtaThreads, gl.smem, 1, gl.table, p.qmax, p.mode);
        if (rc) return rc;
    }
    for (const ParamPlan::Rows &r : p.rows) {
        auto kernel = r.form == ParamPlan::kRow512 ? sq::squant_row_kernel<512, false>
                      : r.form == ParamPlan::kLong512 ? sq::squant_row_kernel<512, true> : sq::squant_row_kernel<256, false>;
        const int rc = launch(kernel, r.grid, r.form == ParamPlan::kRow256 ? 256 : 512, r.smem, 1, r.table, p.qmax, mode());
        if (rc) return rc;
    }
    for (const ParamPlan::Wide &w : p.wide) {   // one cluster per output channel
        const int rc = launch(sq::squant_wide_kernel, w.d.M * w.cluster, sq::kBlockThreads, w.smem, w.cluster, w.d, p.qmax, mode(), w.kpc);
        if (rc) return rc;
    }
    return SQUANT_OK;
}

// Device staging of the host-buffer entry point, one arena per device, grown on demand.
struct Arena { void *ptr = nullptr; size_t bytes = 0; };
std::vector<Arena> g_arenas;

// Copy streams and events of the host-buffer entry point, one set per device, created on first
// use: uploads, kernels and downloads of consecutive chunks of layers overlap.
struct HostPipe {
    cudaStream_t in = nullptr, out = nullptr;
    cudaEvent_t start = nullptr;
    std::vector<cudaEvent_t> uploaded, computed;
};
std::vector<HostPipe> g_host_pipes;
// Weights per chunk.  A chunk's downloads can run while the next chunks' weights are on their way, so what remains
// outside the overlap is about one chunk at either end: ResNet-50 shapes (102 MB up, 87 MB down) take 3356 us, and
// 4286 us in chunks of 64 MB with every tensor copied by itself.
constexpr size_t kHostChunkBytes = 8u << 20;
constexpr size_t kHostChunks = 24;   // and no more than about these: each has a plan of its own
// Outputs of at most this many bytes come down through pinned staging memory, all of a chunk in one copy: a copy of a
// few KB costs its fixed few microseconds on the copy engine, more than the host's memcpy takes.  (Inputs don't: work
// that the caller's stream still holds may be about to write them.)
constexpr size_t kHostSmallBytes = 32u << 10;

// Pinned staging memory of the host-buffer entry point, one per device, grown on demand.
struct Staging { void *ptr = nullptr; size_t bytes = 0; };
std::vector<Staging> g_stagings;

int host_pipe(int device, size_t chunks, HostPipe *&out)
{
    if (static_cast<int>(g_host_pipes.size()) <= device) g_host_pipes.resize(device + 1);
    HostPipe &hp = g_host_pipes[device];
    if (!hp.in) {
        SQ_CUDA(cudaStreamCreateWithFlags(&hp.in, cudaStreamNonBlocking));
        SQ_CUDA(cudaStreamCreateWithFlags(&hp.out, cudaStreamNonBlocking));
        SQ_CUDA(cudaEventCreateWithFlags(&hp.start, cudaEventDisableTiming));
    }
    while (hp.uploaded.size() < chunks) {
        cudaEvent_t a = nullptr, b = nullptr;
        SQ_CUDA(cudaEventCreateWithFlags(&a, cudaEventDisableTiming));
        SQ_CUDA(cudaEventCreateWithFlags(&b, cudaEventDisableTiming));
        hp.uploaded.push_back(a);
        hp.computed.push_back(b);
    }
    out = &hp;
    return SQUANT_OK;
}

inline size_t align256(size_t v) { return (v + 255) & ~static_cast<size_t>(255); }

// ---- launch table of squant_quantize_layer_noalloc: part of the library image, never allocated.
// Layout: one LayerDesc in the first 256 bytes, then up to SQUANT_NOALLOC_MAX_CTAS Items.
// In host code the name below is only a handle of the symbol; the address a kernel can use comes
// from cudaGetSymbolAddress, taken once per device with that device current.
static_assert(sizeof(LayerDesc) <= 256, "layer descriptor must fit the table header");
static_assert(sizeof(Item) == 8, "table size in squant.h assumes 8-byte entries");
static __device__ __align__(256) unsigned char g_noalloc_table[SQUANT_NOALLOC_TABLE_BYTES];
unsigned char g_noalloc_host[SQUANT_NOALLOC_TABLE_BYTES];   // host image, guarded by g_mutex
std::vector<void *> g_noalloc_dev;                          // per device: address of the table

int noalloc_table_address(int device, void *&ptr)
{
    if (static_cast<int>(g_noalloc_dev.size()) <= device) g_noalloc_dev.resize(device + 1, nullptr);
    if (!g_noalloc_dev[device]) {
        void *p = nullptr;
        SQ_CUDA(cudaGetSymbolAddress(&p, g_noalloc_table));   // current device is `device`
        g_noalloc_dev[device] = p;
    }
    ptr = g_noalloc_dev[device];
    return SQUANT_OK;
}

}  // namespace

extern "C" {

int squant_quantize_model(const squant_layer *layers, int32_t n_layers, const squant_options *opt,
                          void *cuda_stream)
{
    squant_options o;
    int rc = validate(layers, n_layers, opt, true, o);
    if (rc) return rc;
    if (n_layers == 0) return SQUANT_OK;
    std::lock_guard<std::mutex> lock(g_mutex);
    const ParamPlan *pp = nullptr;
    rc = get_plan(layers, n_layers, o, pp);
    if (rc) return rc;
    return launch_plan(*pp, static_cast<cudaStream_t>(cuda_stream));
}

int squant_quantize_layer(const squant_layer *layer, const squant_options *opt, void *cuda_stream)
{
    if (!layer) return SQUANT_ERR_NULL;
    return squant_quantize_model(layer, 1, opt, cuda_stream);
}

int squant_quantize_model_host(const squant_layer *layers, int32_t n_layers,
                               const squant_options *opt, void *cuda_stream)
{
    squant_options o;
    int rc = validate(layers, n_layers, opt, true, o);
    if (rc) return rc;
    if (n_layers == 0) return SQUANT_OK;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    std::lock_guard<std::mutex> lock(g_mutex);
    int device = 0;
    SQ_CUDA(cudaGetDevice(&device));
    // Chunks of consecutive layers.  Uploads run on one
    // copy stream, each chunk's launches on the caller's stream once its upload is done, its
    // downloads on a second copy stream once its launches are done: the two copy directions and
    // the kernels overlap.
    std::vector<int> chunk_first(1, 0);
    {
        size_t acc = 0, all = 0;
        const auto weight_bytes = [&](int i) { return static_cast<size_t>(layers[i].cin) * layers[i].kh * layers[i].kw * layers[i].cout * 4; };
        for (int i = 0; i < n_layers; ++i) all += weight_bytes(i);
        const size_t goal = std::max(kHostChunkBytes, all / kHostChunks);
        for (int i = 0; i < n_layers; ++i) {
            acc += weight_bytes(i);
            if (acc >= goal && i + 1 < n_layers) { chunk_first.push_back(i + 1); acc = 0; }
        }
        chunk_first.push_back(n_layers);
    }
    const size_t chunks = chunk_first.size() - 1;
    // every tensor of the call, in the order of squant_layer's inputs and outputs
    struct Tensor { void *host; size_t bytes, off; bool small; };
    constexpr int kInputs = 2, kTensors = 8;   // weights, supplied scales | codes, scales, sums (kernels, channels), dequantized (fp32, bf16)
    std::vector<Tensor> tensors(static_cast<size_t>(n_layers) * kTensors);
    for (int i = 0; i < n_layers; ++i) {
        const squant_layer &l = layers[i];
        const size_t m = static_cast<size_t>(l.cout), nk = static_cast<size_t>(l.cin) * l.kh * l.kw, n = m * nk;
        const size_t code_bytes = (o.flags & SQUANT_FLAG_PACK_INT4) ? m * ((nk + 1) / 2) : n;
        Tensor *t = &tensors[static_cast<size_t>(i) * kTensors];
        const auto put = [&](int k, const void *p, size_t bytes) {
            t[k] = {const_cast<void *>(p), p ? bytes : 0, 0, k >= kInputs && bytes <= kHostSmallBytes};
        };
        put(0, l.w, n * 4);
        put(1, l.scales_in, m * 4);
        put(2, l.codes, code_bytes);
        put(3, l.scales, m * 4);
        put(4, l.kernel_err, m * l.cin * 4);
        put(5, l.channel_err, m * 4);
        put(6, l.dequant, n * 4);
        put(7, l.dequant_bf16, n * 2);
    }
    // One device arena; a chunk's small outputs lie together in it.
    struct Run { size_t off, bytes, at; };   // in the arena; its place in the staging memory
    std::vector<Run> small(chunks);
    size_t total = 0, staged = 0;
    for (size_t c = 0; c < chunks; ++c)
        for (int pass = 0; pass < 2; ++pass) {   // the small ones first
            if (pass == 0) small[c] = {total, 0, staged};
            for (int i = chunk_first[c]; i < chunk_first[c + 1]; ++i)
                for (int k = 0; k < kTensors; ++k) {
                    Tensor &t = tensors[static_cast<size_t>(i) * kTensors + k];
                    if (!t.host || t.small != (pass == 0)) continue;
                    t.off = total;
                    total += align256(t.bytes);
                }
            if (pass == 0) {
                small[c].bytes = total - small[c].off;
                staged += small[c].bytes;
            }
        }
    if (static_cast<int>(g_arenas.size()) <= device) g_arenas.resize(device + 1);
    Arena &a = g_arenas[device];
    if (a.bytes < total) {
        if (a.ptr) { SQ_CUDA(cudaDeviceSynchronize()); SQ_CUDA(cudaFree(a.ptr)); a.ptr = nullptr; a.bytes = 0; }
        cudaError_t e = cudaMalloc(&a.ptr, total);
        if (e != cudaSuccess) { a.ptr = nullptr; return e == cudaErrorMemoryAllocation ? SQUANT_ERR_NOMEM : cuda_fail(e, "cudaMalloc"); }
        a.bytes = total;
    }
    if (static_cast<int>(g_stagings.size()) <= device) g_stagings.resize(device + 1);
    Staging &stg = g_stagings[device];
    if (stg.bytes < staged) {   // (no call is under way: each ends with its copies done)
        if (stg.ptr) { SQ_CUDA(cudaFreeHost(stg.ptr)); stg.ptr = nullptr; stg.bytes = 0; }
        if (cudaHostAlloc(&stg.ptr, staged, cudaHostAllocDefault) == cudaSuccess) {
            stg.bytes = staged;
        } else {   // no pinned memory to be had: every tensor is copied by itself
            cudaGetLastError();
            stg.ptr = nullptr;
        }
    }
    unsigned char *base = static_cast<unsigned char *>(a.ptr), *pinned = static_cast<unsigned char *>(stg.ptr);
    std::vector<squant_layer> dev(layers, layers + n_layers);
    for (int i = 0; i < n_layers; ++i) {
        const Tensor *t = &tensors[static_cast<size_t>(i) * kTensors];
        const auto at = [&](int k) -> void * { return t[k].host ? base + t[k].off : nullptr; };
        dev[i].w = static_cast<const float *>(at(0));
        dev[i].scales_in = static_cast<const float *>(at(1));
        dev[i].codes = static_cast<int8_t *>(at(2));
        dev[i].scales = static_cast<float *>(at(3));
        dev[i].kernel_err = static_cast<float *>(at(4));
        dev[i].channel_err = static_cast<float *>(at(5));
        dev[i].dequant = static_cast<float *>(at(6));
        dev[i].dequant_bf16 = static_cast<uint16_t *>(at(7));
    }
    // every chunk's plan first: a call that is refused has copied and launched nothing
    HostCall *plans = nullptr;
    rc = get_host_plans(dev, chunk_first, o, device, plans);
    if (rc) return rc;
    if (static_cast<int>(g_host_scratch.size()) <= device) g_host_scratch.resize(device + 1);
    for (const ParamPlan &plan : plans->chunks)
        for (ParamPlan::Stream &st : plan.streams) {
            ScratchRef &shared = g_host_scratch[device];
            if (!shared) rc = new_scratch(device, std::max(g_sm_count_by_device[device], 1), stream, shared);   // (none to be had: launch_plan's to settle)
            if (rc) return rc;
            st.scratch = shared;
        }
    HostPipe *hp = nullptr;
    rc = host_pipe(device, chunks, hp);
    if (rc) return rc;
    const auto each = [&](size_t c, bool outputs, auto fn) -> int {   // a chunk's tensors
        for (int i = chunk_first[c]; i < chunk_first[c + 1]; ++i)
            for (int k = outputs ? kInputs : 0; k < (outputs ? kTensors : kInputs); ++k) {
                const Tensor &t = tensors[static_cast<size_t>(i) * kTensors + k];
                if (!t.host) continue;
                const int e = fn(t);
                if (e) return e;
            }
        return SQUANT_OK;
    };
    // whatever ends the call, its copies have ended then too
    struct Drain {
        cudaStream_t a, b, c;
        bool armed;
        ~Drain()
        {
            if (!armed) return;
            cudaStreamSynchronize(a);
            cudaStreamSynchronize(b);
            cudaStreamSynchronize(c);
        }
    };
    Drain drain{hp->in, stream, hp->out, true};
    SQ_CUDA(cudaEventRecord(hp->start, stream));          // uploads follow what the caller's stream holds so far
    SQ_CUDA(cudaStreamWaitEvent(hp->in, hp->start, 0));
    for (size_t c = 0; c < chunks; ++c) {
        rc = each(c, false, [&](const Tensor &t) -> int {
            SQ_CUDA(cudaMemcpyAsync(base + t.off, t.host, t.bytes, cudaMemcpyHostToDevice, hp->in));
            return SQUANT_OK;
        });
        if (rc) return rc;
        SQ_CUDA(cudaEventRecord(hp->uploaded[c], hp->in));
    }
    for (size_t c = 0; c < chunks; ++c) {
        SQ_CUDA(cudaStreamWaitEvent(stream, hp->uploaded[c], 0));
        rc = launch_plan(plans->chunks[c], stream);
        if (rc) return rc;
        SQ_CUDA(cudaEventRecord(hp->computed[c], stream));
        SQ_CUDA(cudaStreamWaitEvent(hp->out, hp->computed[c], 0));
        const Run &run = small[c];
        rc = each(c, true, [&](const Tensor &t) -> int {
            if (!pinned || !t.small) SQ_CUDA(cudaMemcpyAsync(t.host, base + t.off, t.bytes, cudaMemcpyDeviceToHost, hp->out));
            return SQUANT_OK;
        });
        if (rc) return rc;
        if (pinned && run.bytes) SQ_CUDA(cudaMemcpyAsync(pinned + run.at, base + run.off, run.bytes, cudaMemcpyDeviceToHost, hp->out));
    }
    drain.armed = false;
    SQ_CUDA(cudaStreamSynchronize(hp->out));
    SQ_CUDA(cudaStreamSynchronize(stream));
    if (pinned)
        for (size_t c = 0; c < chunks; ++c)
            each(c, true, [&](const Tensor &t) -> int {
                if (t.small) std::memcpy(t.host, pinned + small[c].at + (t.off - small[c].off), t.bytes);
                return SQUANT_OK;
            });
    return SQUANT_OK;
}

int squant_quantize_layer_noalloc(const squant_layer *layer, const squant_options *opt,
                                  void *cuda_stream)
{
    if (!layer) return SQUANT_ERR_NULL;
    squant_options o;
    int rc = validate(layer, 1, opt, true, o);
    if (rc) return rc;
    HostPlan hp;   // host-side bookkeeping only; nothing below allocates device memory
    rc = build_plan(layer, 1, o, kMaxSmemFallback, hp);
    if (rc) return rc;
    if (hp.items.size() > static_cast<size_t>(SQUANT_NOALLOC_MAX_CTAS)) return SQUANT_ERR_LIMIT;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    std::lock_guard<std::mutex> lock(g_mutex);
    {   // the table upload below reads a host image that the next call rewrites: not for a captured stream
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        SQ_CUDA(cudaStreamIsCapturing(stream, &cap));
        if (cap != cudaStreamCaptureStatusNone) return SQUANT_ERR_CAPTURE;
    }
    int device = 0;
    SQ_CUDA(cudaGetDevice(&device));
    int limit = 0;
    rc = device_smem_limit(device, limit);
    if (rc) return rc;
    if (hp.smem_bytes > limit) return SQUANT_ERR_TOO_WIDE;
    void *table = nullptr;
    rc = noalloc_table_address(device, table);
    if (rc) return rc;
    const size_t ibytes = sizeof(Item) * hp.items.size();
    std::memcpy(g_noalloc_host, hp.layers.data(), sizeof(LayerDesc));
    std::memcpy(g_noalloc_host + 256, hp.items.data(), ibytes);
    // Pageable source: the runtime has taken its copy of the bytes when this returns, so the host
    // image may be rewritten by the next call; the device-side copy is ordered on `stream`.
    SQ_CUDA(cudaMemcpyAsync(table, g_noalloc_host, 256 + ibytes, cudaMemcpyHostToDevice, stream));
    const LayerDesc *dl = static_cast<const LayerDesc *>(table);
    const Item *di = reinterpret_cast<const Item *>(static_cast<const unsigned char *>(table) + 256);
    auto kernel = hp.layers[0].sin ? sq::squant_table_kernel<sq::kOwnScales> : sq::squant_table_kernel<sq::kAbsmax>;
    kernel<<<static_cast<unsigned>(hp.items.size()), sq::kCtaThreads, hp.smem_bytes, stream>>>(dl, di, hp.qmax, hp.mode);
    SQ_CUDA(cudaGetLastError());
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return SQUANT_OK;
}

int squant_plan_info(const squant_layer *layers, int32_t n_layers, const squant_options *opt,
                     int32_t *grid_ctas, int32_t *cta_threads, int32_t *dynamic_smem_bytes)
{
    squant_options o;
    int rc = validate(layers, n_layers, opt, false, o);
    if (rc) return rc;
    HostPlan hp;
    rc = build_plan(layers, n_layers, o, kMaxSmemFallback, hp);
    if (rc) return rc;
    if (grid_ctas) *grid_ctas = static_cast<int32_t>(hp.items.size());
    if (cta_threads) *cta_threads = sq::kCtaThreads;
    if (dynamic_smem_bytes) *dynamic_smem_bytes = hp.smem_bytes;
    return SQUANT_OK;
}

int squant_plan_kernels(const squant_layer *layers, int32_t n_layers, const squant_options *opt, int32_t *kernels)
{
    squant_options o;
    int rc = validate(layers, n_layers, opt, false, o);
    if (rc) return rc;
    if (n_layers > 0 && !kernels) return SQUANT_ERR_NULL;
    ParamPlan plan;
    return build_param_plan(layers, n_layers, o, kMaxSmemFallback, 148, plan, kernels);
}

int squant_selfcheck_division(const float *scales, int32_t n, int32_t bits, uint64_t *mismatches,
                              void *cuda_stream)
{
    if (!scales || !mismatches) return SQUANT_ERR_NULL;
    if (n <= 0 || n > 65535) return SQUANT_ERR_SHAPE;
    if (bits < 2 || bits > 8) return SQUANT_ERR_BITS;
    for (int i = 0; i < n; ++i)
        if (!(scales[i] >= 0x1p-60f && scales[i] <= 0x1p60f)) return SQUANT_ERR_SHAPE;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    float *d_s = nullptr;
    unsigned long long *d_m = nullptr;
    SQ_CUDA(cudaMalloc(&d_s, sizeof(float) * n));
    cudaError_t e = cudaMalloc(&d_m, sizeof(unsigned long long) * n);
    if (e != cudaSuccess) { cudaFree(d_s); return cuda_fail(e, "cudaMalloc"); }
    e = cudaMemcpyAsync(d_s, scales, sizeof(float) * n, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_m, 0, sizeof(unsigned long long) * n, stream);
    if (e == cudaSuccess) {
        sq::selfcheck_division_kernel<<<dim3(1184, n), 256, 0, stream>>>(d_s, n, (1 << (bits - 1)) - 1, d_m);
        e = cudaGetLastError();
        g_launches.fetch_add(1, std::memory_order_relaxed);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(mismatches, d_m, sizeof(unsigned long long) * n, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    cudaFree(d_s);
    cudaFree(d_m);
    if (e != cudaSuccess) return cuda_fail(e, "squant_selfcheck_division");
    return SQUANT_OK;
}

int squant_device_status(void)
{
    std::lock_guard<std::mutex> lock(g_mutex);
    SQ_CUDA(cudaDeviceSynchronize());
    int st = 0;
    SQ_CUDA(cudaMemcpyFromSymbol(&st, sq::g_device_status, sizeof(int)));
    if (st == 0) return SQUANT_OK;
    const int zero = 0;
    SQ_CUDA(cudaMemcpyToSymbol(sq::g_device_status, &zero, sizeof(int)));
    // a launch that gave up may have left its work counters half drawn: all start clean again
    int device = 0;
    SQ_CUDA(cudaGetDevice(&device));
    for (const std::weak_ptr<StreamScratch> &w : g_scratch)
        if (const ScratchRef s = w.lock())
            if (s->device == device) SQ_CUDA(cudaMemset(s->work(), 0, sq::kStreamWorkBytes));
    return SQUANT_ERR_TIMEOUT;
}

int squant_debug_violations(int32_t *count, int32_t *first_site)
{
    std::lock_guard<std::mutex> lock(g_mutex);
    SQ_CUDA(cudaDeviceSynchronize());
    unsigned n = 0;
    int site = 0;
    SQ_CUDA(cudaMemcpyFromSymbol(&n, sq::g_debug_violations, sizeof(n)));
    SQ_CUDA(cudaMemcpyFromSymbol(&site, sq::g_debug_site, sizeof(site)));
    if (count) *count = static_cast<int32_t>(n);
    if (first_site) *first_site = site;
    const unsigned zero = 0;
    SQ_CUDA(cudaMemcpyToSymbol(sq::g_debug_violations, &zero, sizeof(zero)));
    SQ_CUDA(cudaMemcpyToSymbol(sq::g_debug_site, &zero, sizeof(int)));
#ifdef SQUANT_DEBUG_BOUNDS
    return 1;   // this library was built with the checks
#else
    return SQUANT_OK;
#endif
}

int64_t squant_debug_sums_checked(void)
{
    std::lock_guard<std::mutex> lock(g_mutex);
    SQ_CUDA(cudaDeviceSynchronize());
    unsigned n = 0;
    SQ_CUDA(cudaMemcpyFromSymbol(&n, sq::g_debug_sums, sizeof(n)));
    const unsigned zero = 0;
    SQ_CUDA(cudaMemcpyToSymbol(sq::g_debug_sums, &zero, sizeof(zero)));
    return static_cast<int64_t>(n);
}

int squant_debug_set_status(int value)
{
    std::lock_guard<std::mutex> lock(g_mutex);
    SQ_CUDA(cudaMemcpyToSymbol(sq::g_device_status, &value, sizeof(int)));
    return SQUANT_OK;
}

int squant_debug_wait_expires(int32_t max_polls, void *cuda_stream)
{
    if (max_polls < 1 || max_polls > 4096) return SQUANT_ERR_SHAPE;
    sq::debug_wait_kernel<<<1, 32, 0, static_cast<cudaStream_t>(cuda_stream)>>>(max_polls);
    SQ_CUDA(cudaGetLastError());
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return SQUANT_OK;
}

int64_t squant_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char *squant_strerror(int code)
{
    switch (code) {
        case SQUANT_OK: return "success";
        case SQUANT_ERR_NULL: return "a required pointer is NULL";
        case SQUANT_ERR_SHAPE: return "a layer dimension is not positive or the element count overflows";
        case SQUANT_ERR_BITS: return "bits must be in 2..8 (2..4 with SQUANT_FLAG_PACK_INT4)";
        case SQUANT_ERR_MODE: return "mode mask must contain E (E, E|K, E|C or E|K|C); unknown mode or flag bits are rejected";
        case SQUANT_ERR_ALIGN: return "float pointers must be 4-byte aligned";
        case SQUANT_ERR_TOO_WIDE: return "an output channel (cin*kh*kw) does not fit the on-chip path, not even spread over a cluster of 8 thread blocks";
        case SQUANT_ERR_CUDA: return "a CUDA runtime call failed (see squant_last_cuda_error)";
        case SQUANT_ERR_NOMEM: return "out of host or device memory";
        case SQUANT_ERR_TIMEOUT: return "a kernel gave up a bounded wait on an asynchronous copy; outputs of that launch are incomplete";
        case SQUANT_ERR_CAPTURE: return "squant_quantize_layer_noalloc was called on a stream that is being captured; it uploads its launch table from a host image that the next call rewrites";
        case SQUANT_ERR_LIMIT: return "the layer needs more thread blocks than the fixed launch table of squant_quantize_layer_noalloc holds (SQUANT_NOALLOC_MAX_CTAS); split it by output-channel range";
        default: return "unknown squant error code";
    }
}

const char *squant_last_cuda_error(void) { return t_cuda_error.c_str(); }

int squant_shutdown(void)
{
    std::lock_guard<std::mutex> lock(g_mutex);
    int cur = 0;
    const bool have = cudaGetDevice(&cur) == cudaSuccess;
    g_plans.clear();
    g_host_calls.clear();
    g_host_scratch.clear();
    free_dead_scratch();   // (areas that a graph still holds go with the graph)
    for (size_t d = 0; d < g_arenas.size(); ++d) {
        if (g_arenas[d].ptr) { cudaSetDevice(static_cast<int>(d)); cudaDeviceSynchronize(); cudaFree(g_arenas[d].ptr); }
    }
    g_arenas.clear();
    for (Staging &stg : g_stagings)
        if (stg.ptr) cudaFreeHost(stg.ptr);
    g_stagings.clear();
    for (size_t d = 0; d < g_host_pipes.size(); ++d) {
        HostPipe &hp = g_host_pipes[d];
        if (!hp.in) continue;
        cudaSetDevice(static_cast<int>(d));
        for (cudaEvent_t e : hp.uploaded) cudaEventDestroy(e);
        for (cudaEvent_t e : hp.computed) cudaEventDestroy(e);
        cudaEventDestroy(hp.start);
        cudaStreamDestroy(hp.in);
        cudaStreamDestroy(hp.out);
    }
    g_host_pipes.clear();
    if (have) cudaSetDevice(cur);
    return SQUANT_OK;
}

}  // extern "C"
