// C-ABI of the qlinear library: handle life cycle, stage-aware dispatch (paper Section 3.7) and the
// launchers of the decode and prefill kernels.  Single translation unit for all device code.
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>

#include "../../include/qlinear.h"
#include "layout.h"

namespace ql {
// Set by a kernel that gave up a bounded wait: [0] = non-zero code identifying the wait, [1] = count.
__device__ unsigned int g_device_flag[2];
// Device-side alias of one word of pinned host memory (null until the first handle on the device exists): the
// same code, readable by the host without synchronising.
__device__ unsigned int* g_status_host;
}  // namespace ql

#include "dequant.cuh"
#include "embed.cuh"
#include "gemv.cuh"
#include "gemv_cols.cuh"
#include "gemv_rows.cuh"
#include "gemv_stream.cuh"
#include "gemv_a8.cuh"
#include "kv.cuh"
#include "gemm.cuh"
#include "gemm_mid.cuh"
#include "gemm_rows.cuh"
#include "gemm_pair.cuh"
#include "gemm_pair_ta.cuh"
#include "gemm_narrow.cuh"
#include "norm.cuh"
#include "rope.cuh"

using namespace ql;

namespace {

int env_int(const char* name, int dflt)
{
    const char* v = std::getenv(name);
    return (v && *v) ? std::atoi(v) : dflt;
}

// Every QLINEAR_* switch, read from the environment ONCE per process (at the first call that needs one).
struct Config {
    int gemv_max_m;          // QLINEAR_GEMV_MAX_M: largest M served by the decode kernels (1..8)
    bool pdl;                // QLINEAR_PDL: programmatic dependent launch attribute on every kernel
    int warps_per_sm;        // QLINEAR_GEMV_WARPS_PER_SM: residency target of the cluster decode kernel
    bool oversubscribe;      // QLINEAR_GEMV_OVERSUBSCRIBE=0: the group-scaled int4 decode kernel never takes more CTAs than fit at once
    int force_ks;            // QLINEAR_GEMV_KS: forced K split of the cluster decode kernel (0 = planned)
    int mid_max_m;           // QLINEAR_MID_MAX_M: largest M up to 64 that the kernels for a batch of tokens may serve (0: none); see takes_mid, narrow_can
    int narrow;              // QLINEAR_GEMM_NARROW: 0 gemm_narrow.cuh serves no call, 1 by the rules (default), 2 every call that it can serve
    bool xdirect;            // QLINEAR_GEMV_XDIRECT: x fragments straight from global memory
    int kernel;              // QLINEAR_GEMV_KERNEL: 0 / 1 cluster kernel (default), 2 streaming kernel
    int stream_ctas_per_sm, stream_stages;
    GemmConfig gemm;
    unsigned generation;     // bumped by qlinear_debug_reload_config (tests)
};
Config g_cfg;
std::once_flag g_cfg_once;
std::atomic<unsigned> g_getenv_reads{0};

void load_config()
{
    Config c{};
    c.gemv_max_m = std::max(1, std::min(8, env_int("QLINEAR_GEMV_MAX_M", 8)));
    c.pdl = env_int("QLINEAR_PDL", 1) != 0;
    c.warps_per_sm = env_int("QLINEAR_GEMV_WARPS_PER_SM", 32);
    c.oversubscribe = env_int("QLINEAR_GEMV_OVERSUBSCRIBE", 1) != 0;
    c.force_ks = env_int("QLINEAR_GEMV_KS", 0);
    c.mid_max_m = env_int("QLINEAR_MID_MAX_M", 64);
    c.narrow = env_int("QLINEAR_GEMM_NARROW", 1);
    c.xdirect = env_int("QLINEAR_GEMV_XDIRECT", 1) != 0;
    const char* kc = std::getenv("QLINEAR_GEMV_KERNEL");
    c.kernel = !kc ? 0 : !std::strcmp(kc, "cluster") ? 1 : !std::strcmp(kc, "stream") ? 2 : 0;
    c.stream_ctas_per_sm = std::max(1, std::min(4, env_int("QLINEAR_STREAM_CTAS_PER_SM", 3)));
    c.stream_stages = env_int("QLINEAR_STREAM_STAGES", kStreamMaxStages);
    c.gemm.force_bn = env_int("QLINEAR_GEMM_BN", 0);
    c.gemm.force_split = env_int("QLINEAR_GEMM_SPLIT", 0);
    c.gemm.force_tb = env_int("QLINEAR_GEMM_TB", 0);
    c.gemm.pair = env_int("QLINEAR_GEMM_PAIR", 1) != 0;
    c.gemm.ta = env_int("QLINEAR_GEMM_TA", 1) != 0;
    c.generation = g_cfg.generation + 1;
    g_cfg = c;
    g_getenv_reads.fetch_add(1);
}
const Config& config()
{
    std::call_once(g_cfg_once, load_config);
    return g_cfg;
}

}  // namespace

namespace ql {
GemmConfig& gemm_config() { return const_cast<Config&>(config()).gemm; }
}  // namespace ql

namespace {

struct GemvPlan {
    int32_t ks_cta, cl, cps, x_stride, x_bytes, smem_bytes, grid;
    double max_over_mean;    // chunks of the busiest SM over the mean, as the hardware would place the grid
};

// Device memory the library owns, ONE set per device, created with the first handle on that device and shared by
// every handle there (kernels that use it run in stream order: see include/qlinear.h).
struct DeviceState {
    bool ready = false;
    int sms = 0;
    int handles = 0;
    unsigned int* status_host = nullptr;     // pinned, mapped: the code of the last expired wait (0 = none)
    float* gemm_scratch = nullptr;           // CTA-pair prefill kernel, K-split of single-round layers
    unsigned int* gemm_counters = nullptr;
    float* stream_scratch = nullptr;         // streaming decode kernel (only when QLINEAR_GEMV_KERNEL=stream)
    unsigned int* stream_counters = nullptr;
};
constexpr int kMaxDevices = 64;
constexpr int kStreamMaxRsb = 4096;          // row super-blocks the shared streaming-kernel counters cover
DeviceState g_dev[kMaxDevices];
std::mutex g_dev_mutex;

}  // namespace

struct qlinear_s {
    // Immutable after qlinear_create (but for `cache`).
    Layout L;
    const uint8_t* blob;
    int device;
    int num_sms;
    int gemv_max_m;
    bool pdl;
    int n_rb;                  // row-blocks holding at least one real row
    GemvPlan gemv[9];          // cluster decode kernel, index = M (1..8)
    bool use_stream;
    int stream_P, stream_stages;
    CUtensorMap wmap;          // the packed body as rows of 64 bytes (prefill kernel with the weights in tensor memory)
    CUtensorMap wmap_wide;     // the same with a box of 128 k per step (the integer form, gemm_narrow.cuh)
    bool wmap_ok, wmap_wide_ok;
    DeviceState* dev;
    // Set by the first append: the blob is a KV cache, and the kernel before a reader in the stream may be writing it.  Its readers
    // then touch it only after griddepcontrol.wait (`late` in their parameters; the decode readers of a cache: only the tokens that held_tokens
    // names), or are launched without the programmatic edge (early(): int8 activations, the streaming kernel).  (Written under no lock: a caller that enqueues a reader behind an append has ordered the two calls.)
    std::atomic<bool> cache{false};
    // The last append that was launched: its tokens [first, end) and where it was enqueued.  Guarded by g_append_mutex[device].
    struct Append {
        int32_t first = 0, end = 0;
        cudaStream_t stream = nullptr;
        unsigned long long capture = 0;      // id of the stream capture that recorded it, 0: none
        bool alone = false;                  // every append to this cache in that capture was enqueued on this stream
    } append;
    bool early() const { return pdl && !cache.load(std::memory_order_relaxed); }
};

namespace {

bool any_cache(const qlinear_s* const* hs, int n)
{
    for (int i = 0; i < n; ++i)
        if (hs[i]->cache.load(std::memory_order_relaxed)) return true;
    return false;
}

// Held while an append is launched and recorded, so that appends to one cache are recorded in the order in which they were enqueued.
std::mutex g_append_mutex[kMaxDevices];

// The capture that a launch on `st` would be recorded in (0: none); false where that cannot be told, or where the handle does not name one
// stream (cudaStreamPerThread).
bool capture_of(cudaStream_t st, unsigned long long* id)
{
    *id = 0;
    if (st == cudaStreamPerThread) return false;
    cudaStreamCaptureStatus status;
    if (cudaStreamGetCaptureInfo(st, &status, id) != cudaSuccess) { cudaGetLastError(); return false; }
    if (status == cudaStreamCaptureStatusNone) *id = 0;
    return status != cudaStreamCaptureStatusInvalidated;
}

// The tokens [first, end) that appends may still be writing in the caches of a decode launch on `st` while it runs ahead of its
// griddepcontrol.wait; empty for layers that are no cache.  Those of the last append, where that append was enqueued on the same stream and
// in the same capture: an append releases its dependents only past its own wait, when every kernel before it in the stream is
// complete, and what other streams hold is behind an event, a full dependency.  Everything where the last append was enqueued elsewhere (an
// append before it may then be the one in flight: a capture between append and reader, a second stream), and where a capture
// has appends on several streams (the edges that join them may all be programmatic).
constexpr int32_t kHoldAll = 0x7fffffe0;                                 // (a multiple of 32)
void held_tokens(const qlinear_s* const* hs, int n, cudaStream_t st, int32_t* first, int32_t* end)
{
    *first = *end = 0;
    if (!any_cache(hs, n)) return;
    unsigned long long capture;
    const bool known = capture_of(st, &capture);
    std::lock_guard<std::mutex> lock(g_append_mutex[hs[0]->device]);
    for (int i = 0; i < n; ++i) {
        if (!hs[i]->cache.load(std::memory_order_relaxed)) continue;
        const qlinear_s::Append& a = hs[i]->append;
        if (!known || !a.alone || a.stream != st || a.capture != capture) { *first = 0; *end = kHoldAll; return; }
        *first = *end == 0 ? a.first : std::min(*first, a.first);
        *end = std::max(*end, a.end);
    }
}

// The same for a launch over caches of up to `tokens`: true, and an empty range, where all of them are held.
bool hold_range(const qlinear_s* const* hs, int n, cudaStream_t st, int32_t tokens, int32_t* first, int32_t* end)
{
    held_tokens(hs, n, st, first, end);
    const bool all = *first == 0 && *end >= tokens;
    if (all) *end = 0;
    return all;
}

constexpr int kGemvMaxSmem = 96 * 1024;
constexpr int kSmSharedBytes = 228 * 1024;   // shared memory of one SM

// n_rb: row-blocks of the launch (one layer, or all layers of a group that shares x).
// gated: the launch needs both branches of a channel in one CTA: an even number of row-blocks per CTA, no cluster.
// a8: the int8-activation kernel keeps the quantised x of the CTA's K range, and its per-group sums, in shared memory.
GemvPlan plan_gemv(const Layout& L, int n_rb, int M, int num_sms, bool gated = false, bool a8 = false)
{
    const Config& cfg = config();
    const double target = (double)num_sms * cfg.warps_per_sm;
    GemvPlan best{};
    double best_score = -1e30;
    for (int ks_cta = 1; ks_cta <= 8; ks_cta *= 2)
        for (int cl = 1; cl <= (ks_cta == 8 ? 8 : 1); ++cl) {
            if (gated && (ks_cta > 4 || cl > 1)) continue;
            const int ks = ks_cta * cl;
            const int cps = (L.n_kc + ks - 1) / ks;
            if ((ks - 1) * cps >= L.n_kc && ks > 1) continue;               // would leave a slice empty
            const int span = std::min(ks_cta * cps, L.n_kc) * L.chunk_k;
            const int x_stride = span + (((span * 2) % 128) == 0 ? 32 : 0);
            // x fragments straight from global memory need K to be a whole number of chunks (no bounds checks
            // in the kernel); otherwise x is staged in shared memory with zeros beyond K
            const bool direct = cfg.xdirect && (L.K % L.chunk_k) == 0;
            const int a8_span = ks_cta * cps * L.chunk_k;
            const int x_bytes = a8 ? ((M * (a8_span + 32) + 15) / 16) * 16 + a8_span
                                   : direct ? 0 : ((M * x_stride * 2 + 127) / 128) * 128;
            const int smem = x_bytes + kGemvWarps * (kGemvRing * 512 + (L.grouped ? 1024 : 0));
            if (smem > kGemvMaxSmem) continue;
            const double warps = (double)n_rb * ks;
            const double eff = (double)L.n_kc / ((double)ks * cps);
            // slices of fewer than 4 chunks never reach a steady state (measured: 2-chunk slices lose to 4-chunk
            // slices on half as many warps)
            double score = -std::fabs(std::log2(warps / target)) + 2.0 * std::log2(eff) - (cps < 4 ? 1.25 : 0.0) - (cps < 2 ? 1.0 : 0.0);
            // More CTAs than fit at once mean a second wave -- except, for the group-scaled int4 kernel (bound by its
            // instruction stream, not by the memory system) at one token, up to about one and a half waves of CTAs without
            // clusters whose slices stay long: the partial second wave fills in as the first one drains, and the finer
            // units even out the end (Llama gate + up: 17.8 us with 0.76 of a wave, 17.2 us with 1.5 waves).  Measured limits
            // of the rule: the int8 and per-channel forms of the same launch lose 2 to 7 % that way, and with 2 to 8 tokens
            // the launch itself still gains but the step that contains it loses 1 to 3 % (the next launch gets its SMs later).
            if (warps > target) score += (cfg.oversubscribe && M == 1 && L.grouped && cl == 1 && warps <= 1.55 * target && cps >= 16) ? 0.25 : -2.0;
            // a cluster launch and its two cluster-wide barriers cost a microsecond or two (the CTAs of a cluster start
            // together and leave together): more than a launch of a few MB gains from the extra warps (one 2304 x 2304 int8 layer:
            // 4.0 us with a cluster, 3.7 without).
            // Larger launches keep their clusters: timed alone they look better without (Llama o, 16.8 MB: 5.9 / 4.6 us),
            // but inside the step the under-filled grid costs the launches around it more than it saves.
            if (cl > 1 && (double)n_rb * L.n_kc * 512.0 < 6.0e6) score -= 0.75;
            if (a8 && cl > 1) {
                // Every CTA of the int8-activation kernel reads all of x for the row maxima, so doubling the CTAs gives less
                // here once every SM has one: a cluster then has to fill the chip almost as well again (0.9 of a doubling).
                // And its quantised x lies in shared memory, which leaves room for fewer than kGemvA8MaxResident CTAs per SM
                // when M or the range is large: the CTAs that don't fit run as a second wave, with a whole quantisation
                // before it.  For three and more CTAs the last 5 % of the slots count as taken: a cluster needs its slots within one GPC.
                // Seven launches of a block, before -> with both lines: Llama 3.1 8B 844 3 tokens 69.4 -> 62.4 us, 844g32 2 tokens
                // 64.7 -> 59.9; Gemma 2 2B q8 1 token 39.0 -> 36.8, 6 tokens 72.0 -> 67.3, 844g32 8 tokens 80.0 -> 73.1;
                // Llama q8 and 844 at 1 and 4 tokens within 1 %, none slower.  Without the condition on one CTA per SM the
                // Llama cases at 1 to 3 tokens lose 1 to 5 % of it again (k and v, 1024 x 4096, are left with 64 CTAs).
                const int resident = std::min(kGemvA8MaxResident, kSmSharedBytes / (smem + kGemvA8OtherSmem));
                const int ctas = ((n_rb + kGemvWarps / ks_cta - 1) / (kGemvWarps / ks_cta)) * cl;
                if (ctas > (cl > 2 ? 0.95 : 1.0) * num_sms * resident) score -= 2.0;
                if (ctas > num_sms) score -= 0.9 * std::log2((double)cl);
            }
            if (cfg.force_ks && !gated) score = (ks == cfg.force_ks) ? 0.0 : -1e29;
            if (score > best_score) {
                best_score = score;
                const int rb_per_cta = kGemvWarps / ks_cta;
                const int grid = ((n_rb + rb_per_cta - 1) / rb_per_cta) * cl;
                // CTAs spread over the SMs one by one: the busiest SM holds ceil(grid / SMs) of them
                const double per_sm = (double)grid / num_sms;
                best = GemvPlan{ks_cta, cl, cps, x_stride, x_bytes, smem, grid,
                                grid <= 4 * num_sms ? std::ceil(per_sm) / per_sm / eff : 2.0};
            }
        }
    return best;
}

template <typename Kern, typename Params>
cudaError_t launch(Kern kern, const Params& prm, dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, bool pdl)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attrs[2];
    int na = 0;
    if (cluster > 1) {
        attrs[na].id = cudaLaunchAttributeClusterDimension;
        attrs[na].val.clusterDim.x = cluster;
        attrs[na].val.clusterDim.y = 1;
        attrs[na].val.clusterDim.z = 1;
        ++na;
    }
    if (pdl) {
        attrs[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attrs;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, kern, prm);
}

// cudaFuncSetAttribute once per (kernel instantiation, device); `flags` is that instantiation's table.
template <typename Kern>
cudaError_t ensure_smem_attr(Kern kern, std::atomic<bool>* flags, int device, int bytes)
{
    if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
    if (flags[device].load(std::memory_order_acquire)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) flags[device].store(true, std::memory_order_release);
    return e;
}

template <int BITS, bool GROUPED, bool XDIRECT, bool GATED = false, int NG = kGemvMaxGroup, bool ONE = false>
cudaError_t launch_gemv_x(const qlinear_s* h, const GemvParamsT<NG>& prm, const GemvPlan& pl, cudaStream_t st)
{
    if constexpr (GROUPED && !ONE) {
        if (prm.M == 1) return launch_gemv_x<BITS, GROUPED, XDIRECT, GATED, NG, true>(h, prm, pl, st);
    }
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemv_kernel<BITS, GROUPED, XDIRECT, GATED, NG, ONE>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, kGemvMaxSmem);
    if (e != cudaSuccess) return e;
    return launch(kern, prm, dim3(pl.grid), dim3(kGemvThreads), pl.smem_bytes, st, pl.cl, h->pdl);
}

template <int BITS, bool GROUPED>
cudaError_t launch_gemv(const qlinear_s* h, const GemvParams& prm, const GemvPlan& pl, cudaStream_t st, bool gated = false)
{
    if (gated) return launch_gemv_x<BITS, GROUPED, true, true>(h, prm, pl, st);     // (planned only with direct x)
    return prm.x_bytes == 0 ? launch_gemv_x<BITS, GROUPED, true>(h, prm, pl, st)
                            : launch_gemv_x<BITS, GROUPED, false>(h, prm, pl, st);
}
// The wide form (5 to 8 layers, each with its own input read straight from global memory): int8 layers, the KV heads of
// an attention layer.
cudaError_t launch_gemv_wide(const qlinear_s* h, const GemvParamsT<kGemvMaxBatch>& prm, const GemvPlan& pl, cudaStream_t st)
{
    return launch_gemv_x<8, false, true, false, kGemvMaxBatch>(h, prm, pl, st);
}

template <int NG>
void fill_gemv_params(GemvParamsT<NG>& prm, qlinear_s* const* hs, int n, const void* x, void* const* ys, int M, int n_rb, const GemvPlan& pl,
                      int act, const void* const* xs)
{
    const Layout& L = hs[0]->L;
    const bool gated = act >= 0;
    int acc = 0;
    for (int i = 0; i < n; ++i) {
        const Layout& Li = hs[i]->L;
        prm.body[i] = hs[i]->blob + Li.body_offset;
        prm.chan_scales[i] = Li.grouped ? nullptr : reinterpret_cast<const __half*>(hs[i]->blob + Li.chan_scale_offset);
        prm.y[i] = static_cast<__half*>(ys[gated ? 0 : i]);
        prm.N[i] = Li.N;
        acc += hs[i]->n_rb;
        prm.rb_end[i] = acc;
    }
    prm.n_layers = n;
    prm.act = gated ? act : 0;
    prm.late = any_cache(hs, n);
    prm.x = static_cast<const __half*>(xs ? xs[0] : x);
    for (int i = 0; i < NG; ++i) prm.xl[i] = static_cast<const __half*>(xs ? xs[i < n ? i : 0] : x);
    prm.M = M; prm.K = L.K;
    prm.n_rb = n_rb;
    prm.n_kc = L.n_kc;
    prm.block_bytes = L.block_bytes;
    prm.ks_cta = pl.ks_cta; prm.ks_cta_log2 = pl.ks_cta == 8 ? 3 : pl.ks_cta == 4 ? 2 : pl.ks_cta == 2 ? 1 : 0; prm.cl = pl.cl; prm.cps = pl.cps; prm.x_stride = pl.x_stride; prm.x_bytes = pl.x_bytes;
}

// The persistent form for int8 layers with many rows and a short K (gemv_rows.cuh): every layer with its own input.
template <int NKC>
cudaError_t launch_gemv_rows(const qlinear_s* h, const GemvRowsParams& prm, cudaStream_t st)
{
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemv_rows_kernel<NKC>;
    const int smem = kGemvWarps * 2 * NKC * 512;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::min(prm.n_rsb, h->num_sms * (NKC <= 4 ? 4 : 3));
    return launch(kern, prm, dim3(grid), dim3(kGemvThreads), smem, st, 1, h->pdl);
}

// Clusters of `cl` CTAs of the value product's kernel (one CTA per SM) that run at once on `device`: a cluster lies inside one GPC, so
// fewer fit than the SMs alone would hold (148 SMs: 33 of 4, 15 of 8).
int cols_clusters_at_once(int device, int cl)
{
    static std::atomic<int> known[kMaxDevices][4];
    std::atomic<int>& k = known[device][cl == 8 ? 3 : cl == 4 ? 2 : cl == 2 ? 1 : 0];
    int n = k.load(std::memory_order_relaxed);
    if (n) return n;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = cl;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(kColsThreads);
    cfg.dynamicSmemBytes = kColsSmem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, gemv_cols_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    k.store(n, std::memory_order_relaxed);
    return n;
}

// K parts of the value product (CTAs per cluster) for n_rb row-blocks of all its layers: a K of more than 64 chunks is split as far as all
// clusters run at once and every warp keeps 4 chunks, or 2 where the clusters fill no more than half of the GPU (the kernel before
// still holds SMs when these start).  Measured, us undivided / 2 / 4 / 8 parts: 8 row-blocks (a head of 128) at 2048 positions 2.5 / 2.8 /
// 2.7 / 2.8, at 4096 3.5 / 3.2 / 2.8 / 2.8, at 8192 5.0 / 4.4 / 3.2 / 3.0, at 32768 13.9 / 8.8 / 5.9 / 4.4; 16 row-blocks at 32768 14.1 / 8.9 / 5.9 /
// 8.3, 64 of them 14.7 / 10.0 / 12.9 / 21.9 (a second wave of clusters costs more than the split gains); 32 row-blocks at 4096, alone
// 3.5 / 3.2 / 3.1 / 7.4, behind append and scores 6.7 us as 2 parts and 7.3 as 4.
int cols_split(int device, int n_rb, int n_kc)
{
    int cl = 1;
    while (cl < 8 && n_kc > 64) {
        const int at_once = cols_clusters_at_once(device, cl * 2);
        if (n_rb > at_once || n_kc < kColsWarps * cl * 2 * (n_rb * 2 <= at_once ? 2 : 4)) break;
        cl *= 2;
    }
    return cl;
}

// The value product over a KV cache (gemv_cols.cuh): int8 layers of equal shape, every layer with its own input and input scales.
ql_status forward_gemv_cols(qlinear_s* const* hs, int n, const void* const* xs, const void* const* xscales, void* const* ys, int M, cudaStream_t st)
{
    const qlinear_s* h = hs[0];
    const Layout& L = h->L;
    GemvColsParams p{};
    for (int i = 0; i < n; ++i) {
        p.body[i] = hs[i]->blob + L.body_offset;
        p.chan_scales[i] = reinterpret_cast<const __half*>(hs[i]->blob + L.chan_scale_offset);
        p.x[i] = static_cast<const __half*>(xs[i]);
        p.xscale[i] = static_cast<const __half*>(xscales[i]);
        p.y[i] = static_cast<__half*>(ys[i]);
    }
    p.n_layers = n; p.M = M; p.N = L.N; p.K = L.K; p.n_rb = h->n_rb; p.n_kc = L.n_kc;
    p.late = hold_range(hs, n, st, L.K, &p.hold0, &p.hold1);
    p.hold0 /= 32;
    p.hold1 = (p.hold1 + 31) / 32;
    static std::atomic<bool> attr_set[kMaxDevices];
    cudaError_t e = ensure_smem_attr(gemv_cols_kernel, attr_set, h->device, kColsSmem);
    if (e != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
    p.cl = cols_split(h->device, n * h->n_rb, L.n_kc);
    p.cps = (L.n_kc + kColsWarps * p.cl - 1) / (kColsWarps * p.cl);
    e = launch(gemv_cols_kernel, p, dim3(n * h->n_rb * p.cl), dim3(kColsThreads), kColsSmem, st, p.cl, h->pdl);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

// The layers that gemv_rows.cuh (decode) and gemm_rows.cuh (more tokens) take: int8, K of 64, 128 or 256 (the head dimensions of a K
// cache), any number of rows.
bool takes_rows(const Layout& L) { return L.bits == 8 && (L.n_kc == 2 || L.n_kc == 4 || L.n_kc == 8) && L.K == 32 * L.n_kc; }

// One launch for n layers that read the same x (n == 1: the plain forward).  The plan of a group is made per
// call (integer arithmetic only); nothing is written to a handle.
// act >= 0: the gated form (n == 2: gate, up; ys[0] the output; the row-blocks of the two layers alternate).
// xs != nullptr: the batched form, layer i reads xs[i] (x is then ignored); needs the kernel form that reads x straight
// from global memory; int8 layers may come up to kGemvMaxBatch at a time.
ql_status forward_gemv(qlinear_s* const* hs, int n, const void* x, void* const* ys, int M, cudaStream_t st, int act = -1,
                       const void* const* xs = nullptr)
{
    const qlinear_s* h = hs[0];
    const Layout& L = h->L;
    int n_rb = 0;
    for (int i = 0; i < n; ++i) n_rb += hs[i]->n_rb;
    const bool gated = act >= 0;
    if (gated) n_rb = 2 * hs[0]->n_rb;
    // Short K (the score product over a KV cache): the persistent form, whatever the number of rows.  With at most one wave of
    // row super-blocks it wins as well, having no ring to fill, no sums across warps and no barrier (8 heads of 128 at 1280
    // positions 4.1 -> 1.8 us, at 8192 6.7 -> 3.1 us; 2 heads of 64 at 1024 3.3 -> 1.5 us).  One layer as well, a cache or not
    // (a head of 128, 4 rows, 4096 positions 3.7 -> 1.8 us; 32768 x 256 weights, 8 tokens 3.8 -> 3.5 us).
    if (xs && !gated && n <= kGemvMaxBatch && takes_rows(L)) {
        GemvRowsParams rp{};
        int n_rsb = 0;
        for (int i = 0; i < n; ++i) {
            const Layout& Li = hs[i]->L;
            rp.body[i] = hs[i]->blob + Li.body_offset;
            rp.chan_scales[i] = reinterpret_cast<const __half*>(hs[i]->blob + Li.chan_scale_offset);
            rp.y[i] = static_cast<__half*>(ys[i]);
            rp.xl[i] = static_cast<const __half*>(xs[i]);
            rp.N[i] = Li.N;
            n_rsb += Li.n_rsb;
            rp.rsb_end[i] = n_rsb;
        }
        int32_t longest = 0;
        for (int i = 0; i < n; ++i) longest = std::max(longest, hs[i]->L.N);
        rp.late = hold_range(hs, n, st, longest, &rp.hold0, &rp.hold1);
        rp.n_layers = n; rp.M = M; rp.K = L.K; rp.n_rsb = n_rsb; rp.block_bytes = L.block_bytes;
        const cudaError_t e = L.n_kc == 2 ? launch_gemv_rows<2>(h, rp, st) : L.n_kc == 4 ? launch_gemv_rows<4>(h, rp, st) : launch_gemv_rows<8>(h, rp, st);
        return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
    }
    const GemvPlan pl = gated ? plan_gemv(L, n_rb, M, h->num_sms, true) : n == 1 ? h->gemv[M] : plan_gemv(L, n_rb, M, h->num_sms);
    if ((gated || xs) && (pl.grid <= 0 || pl.x_bytes != 0)) return QL_ERR_UNSUPPORTED;
    if (n > kGemvMaxGroup && (n > kGemvMaxBatch || !xs || L.bits != 8)) return QL_ERR_UNSUPPORTED;
    cudaError_t e;
    if (pl.grid <= 0) return QL_ERR_UNSUPPORTED;
    if (n > kGemvMaxGroup) {
        GemvParamsT<kGemvMaxBatch> wide{};
        fill_gemv_params(wide, hs, n, x, ys, M, n_rb, pl, act, xs);
        return launch_gemv_wide(h, wide, pl, st) == cudaSuccess ? QL_OK : QL_ERR_CUDA;
    }
    GemvParams prm{};
    fill_gemv_params(prm, hs, n, x, ys, M, n_rb, pl, act, xs);
    if (L.bits == 8) e = launch_gemv<8, false>(h, prm, pl, st, gated);
    else if (L.grouped) e = launch_gemv<4, true>(h, prm, pl, st, gated);
    else e = launch_gemv<4, false>(h, prm, pl, st, gated);
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

template <int BITS, bool GROUPED, bool GATED, int G>
cudaError_t launch_narrow_g(const qlinear_s* h, const NarrowMaps& maps, const NarrowParams& prm, int grid, cudaStream_t st)
{
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemm_narrow_kernel<BITS, GROUPED, GATED, G>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, kNarrowSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(narrow_threads(G));
    cfg.dynamicSmemBytes = kNarrowSmem;
    cfg.stream = st;
    cudaLaunchAttribute attrs[2];
    int na = 0;
    if (prm.cl > 1) {
        attrs[na].id = cudaLaunchAttributeClusterDimension;
        attrs[na].val.clusterDim.x = prm.cl;
        attrs[na].val.clusterDim.y = attrs[na].val.clusterDim.z = 1;
        ++na;
    }
    if (h->pdl) {
        attrs[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attrs;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, kern, maps, prm);
}

template <int BITS, bool GROUPED, bool GATED>
cudaError_t launch_narrow(const qlinear_s* h, const NarrowMaps& maps, const NarrowParams& prm, int grid, cudaStream_t st)
{
    // three groups where the accumulators leave tensor memory for their slots; int8 unpacks faster and has 16 KB stages: two
    if constexpr (BITS == 4)
        if (prm.bn <= 32) return launch_narrow_g<BITS, GROUPED, GATED, 3>(h, maps, prm, grid, st);
    return launch_narrow_g<BITS, GROUPED, GATED, 2>(h, maps, prm, grid, st);
}

// (The rules below run on every call: whole-number arithmetic in place of calls into the mathematics library, whose code is cold then.)
inline double round_up(double x) { const int64_t i = (int64_t)x; return (double)(i + ((double)i < x)); }       // x >= 0
inline int log2_of(int parts) { return parts == 8 ? 3 : parts >> 1; }                                           // 1, 2, 4 or 8

// Token blocks and K parts of a launch of gemm_narrow.cuh over `rows` row super-blocks: the parts by the cost of the busiest SM.  (Costs for
// comparing the parts with each other only; narrow_us estimates a launch.)  A CTA alone on its SM takes 0.5 per weight tile of 128 k, two
// take 0.62 each; clusters of 4 and 8 lie inside a GPC, so fewer fit than the SMs alone would hold.
struct NarrowPlan { int n_tb, bn, cl; };
NarrowPlan plan_narrow(const Layout& L, int rows, bool gated, int M, int num_sms)
{
    NarrowPlan pl{};
    pl.n_tb = (M + 63) / 64;
    pl.bn = ((M + pl.n_tb - 1) / pl.n_tb + 15) / 16 * 16;
    const int64_t tiles = (int64_t)rows * pl.n_tb;
    const int n_steps = (L.K + kNarrowKStep - 1) / kNarrowKStep;
    double best = 1e30;
    for (int i = 0; i < 4 && (1 << i) <= n_steps; ++i) {
        static const double ramp[4] = {3.5, 3.8, 4.0, 4.3}, fit1[4] = {1.0, 1.0, 0.89, 0.81}, fit2[4] = {1.0, 1.0, 0.92, 0.87};
        const int cl = 1 << i, n = (n_steps * (gated ? 2 : 1) + cl - 1) / cl;
        const double alone = fit1[i] * num_sms / cl, pair = 2 * fit2[i] * num_sms / cl;
        const double us = tiles <= alone ? ramp[i] + 0.5 * n : round_up(tiles / pair) * (ramp[i] + 1.3 + 0.62 * n);
        if (us < best) { best = us; pl.cl = cl; }
    }
    return pl;
}

// n layers that share x, K and scheme; act >= 0: the gated form (n == 2, equal shapes, ys[0] the output).
ql_status forward_narrow(const qlinear_s* const* hs, int n, const void* x, void* const* ys, int M, cudaStream_t st, int act = -1)
{
    const qlinear_s* h = hs[0];
    const Layout& L = h->L;
    const bool gated = act >= 0;
    NarrowMaps maps;
    NarrowParams prm{};
    int units = 0;
    for (int i = 0; i < kGemmMaxGroup; ++i) maps.w[i] = hs[i < n ? i : 0]->wmap_wide;
    for (int i = 0; i < n; ++i) {
        const Layout& Li = hs[i]->L;
        prm.chan_scales[i] = Li.grouped ? nullptr : reinterpret_cast<const __half*>(hs[i]->blob + Li.chan_scale_offset);
        prm.y[i] = static_cast<__half*>(ys[gated ? 0 : i]);
        prm.N[i] = Li.N;
        units += Li.n_rsb;
        prm.unit_end[i] = units;
    }
    if (gated) units = L.n_rsb;
    const NarrowPlan pl = plan_narrow(L, units, gated, M, h->num_sms);
    prm.n_tb = pl.n_tb; prm.bn = pl.bn; prm.cl = pl.cl;
    prm.n_layers = n; prm.M = M; prm.K = L.K; prm.n_kc = L.n_kc; prm.w_rows = L.block_bytes / 64; prm.act = gated ? act : 0;
    prm.n_steps = (L.K + kNarrowKStep - 1) / kNarrowKStep;
    prm.late = any_cache(hs, n);
    // Ring lengths: weight stages a multiple of the groups; x stages even where every stage feeds one issuer (see the kernel).
    prm.nw = L.bits == 4 && prm.bn <= 48 ? 6 : 4;
    prm.nx = std::min(kNarrowMaxX, (kNarrowRing - prm.nw * (L.bits == 4 ? 2 : 4) * L.block_bytes) / (prm.bn * 256));
    if (!gated) prm.nx &= ~1;
    prm.a_col = (2 * prm.bn + 31) / 32 * 32;
    if (!x_tensor_map(x, L.K, M, prm.bn, &maps.x)) return QL_ERR_CUDA;
    const int grid = units * prm.n_tb * prm.cl;
    cudaError_t e;
    if (gated) e = L.bits == 8 ? launch_narrow<8, false, true>(h, maps, prm, grid, st) : L.grouped ? launch_narrow<4, true, true>(h, maps, prm, grid, st) : launch_narrow<4, false, true>(h, maps, prm, grid, st);
    else e = L.bits == 8 ? launch_narrow<8, false, false>(h, maps, prm, grid, st) : L.grouped ? launch_narrow<4, true, false>(h, maps, prm, grid, st) : launch_narrow<4, false, false>(h, maps, prm, grid, st);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

// K parts per tile of gemm_mid.cuh: what the busiest SM has to do, in stages (two CTAs per SM at once, and about 4 stages' time for the
// ramp at the start of a CTA and the sums at its end).  Powers of two: clusters of 3, 5, 6 or 7 CTAs do not fill a GPC, so
// fewer run at once than the slots counted here (Llama q + k + v at 16 tokens, 48 tiles: 12.1 us as 6 parts, 8.3 as 4).
int mid_parts(int tiles, int n_steps, int num_sms)
{
    const int slots = 2 * num_sms;
    double best = 1e30;
    int parts = 1;
    for (int cl = 1; cl <= 8 && cl <= n_steps; cl *= 2) {
        const double cost = (double)((tiles * cl + slots - 1) / slots) * ((double)n_steps / cl + 4.0 + (cl > 1 ? 1.0 : 0.0));
        if (cost < best) { best = cost; parts = cl; }
    }
    return parts;
}

template <int BITS, bool GROUPED, int NT, bool GATED, bool KSCALE>
cudaError_t launch_mid_nt(const qlinear_s* h, MidParams& prm, int units, bool pdl, cudaStream_t st)
{
    using S = MidSmem<BITS, GROUPED, NT>;
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemm_mid_kernel<BITS, GROUPED, NT, GATED, KSCALE>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, S::kTotal);
    if (e != cudaSuccess) return e;
    prm.n_tb = (prm.M + S::kTokens - 1) / S::kTokens;
    prm.n_steps = (prm.n_kc + 1) / 2;
    const int tiles = units * prm.n_tb;
    prm.cl = mid_parts(tiles, prm.n_steps, h->num_sms);
    return launch(kern, prm, dim3((unsigned)(tiles * prm.cl)), dim3(kMidThreads), S::kTotal, st, prm.cl, pdl);
}

// Which launches are the batch stage's: up to 32 tokens all of them, up to 48 those with at most 48 million weights, up to 64 those with at
// most 30 million (int8: 24) or, gated, 48 million; the others are the prefill stage's.  gemm_narrow.cuh takes calls of both stages
// (gemm_route); the line is where gemm_mid.cuh and the prefill kernel are even (21 M weights at 64 tokens 20.9 / 21.4, 34 M 17.5 / 15.9, 59 M at 48 tokens 24.3 / 25.8, 14336 x 4096 26.3 / 22.1).
// QLINEAR_MID_MAX_M lowers the number of tokens up to which this holds (0: never).
bool takes_mid(const qlinear_s* const* hs, int n, int M, bool gated = false)
{
    if (M > 64 || M > config().mid_max_m) return false;
    if (M <= 32) return true;
    int64_t weights = 0;
    for (int i = 0; i < n; ++i) weights += (int64_t)hs[i]->L.N * hs[i]->L.K;
    return weights <= (M <= 48 || gated ? 48000000 : hs[0]->L.bits == 4 ? 30000000 : 24000000);
}

// Tokens per tile of the value product, in eights: 2, 3, 4 or 8, what an estimate of the launch says is fastest (us, consecutive launches over caches
// in L2; 1350 measurements of 16 to 4096 rows, 256 to 16384 positions, heads of 64 to 256 with tiles of 16 to 64: 0.89 to 1.10 times this, 5th and
// 95th percentile).  A step costs a CTA 0.22 us and 0.048 for every 8 tokens, so few rows want narrow tiles; beyond one CTA for 0.735 of
// the SMs (14 clusters of 8 leave room for the next launch's) a launch slows down, and narrow tiles have more CTAs.  Against tiles of 64 to 64 rows, then of 32 while those
// of 64 would leave an SM with one CTA, us before / now: 4096 positions, 48 rows 7.4 / 5.1, 64 8.4 / 5.1, 128 6.4 / 5.3, 256 6.5 / 5.8, 512 9.0 / 7.3, 1024
// 9.7 / 9.5, 2048 14.6 / 13.8; 64 rows of 16384 positions 23.6 / 12.7; 13 % over all of them, the worst 0.95.
int value_tokens(int units, int M, int n_steps, int num_sms)
{
    static const int widths[4] = {2, 3, 4, 8};
    double best_us = 1e30;
    int best = 2;
    for (const int nt : widths) {
        if (nt > 2 && M <= 8 * (nt == 8 ? 4 : nt - 1)) break;            // (a narrower one holds all rows as well)
        const int tiles = units * ((M + 8 * nt - 1) / (8 * nt)), cl = mid_parts(tiles, n_steps, num_sms), ctas = tiles * cl;
        if (ctas > 2 * num_sms && nt != 8) continue;                     // (more rounds than the estimate was made for)
        const double u = ctas / (0.735 * num_sms);
        const double load = 1.0 + 0.47 * std::min(1.0, std::max(0.0, (u - 1.0) / 0.12)) + 0.158 * std::max(0.0, u - 1.12);
        const int steps = (n_steps + cl - 1) / cl, lg = log2_of(cl);
        const double us = 0.88 + 0.137 * lg + load * (0.81 + nt * (0.142 + 0.0153 * lg) + steps * (0.221 + 0.0483 * nt));
        if (us < best_us) { best_us = us; best = nt; }
    }
    return best;
}

template <int BITS, bool GROUPED, bool GATED, bool KSCALE = false>
cudaError_t launch_mid(const qlinear_s* h, MidParams& prm, int units, bool pdl, cudaStream_t st)
{
    if constexpr (KSCALE) {
        switch (value_tokens(units, prm.M, (prm.n_kc + 1) / 2, h->num_sms)) {
            case 2: return launch_mid_nt<BITS, GROUPED, 2, GATED, KSCALE>(h, prm, units, pdl, st);
            case 3: return launch_mid_nt<BITS, GROUPED, 3, GATED, KSCALE>(h, prm, units, pdl, st);
            case 4: return launch_mid_nt<BITS, GROUPED, 4, GATED, KSCALE>(h, prm, units, pdl, st);
            default: return launch_mid_nt<BITS, GROUPED, 8, GATED, KSCALE>(h, prm, units, pdl, st);
        }
    } else {
        if (prm.M <= 16) return launch_mid_nt<BITS, GROUPED, 2, GATED, KSCALE>(h, prm, units, pdl, st);
        if (prm.M <= 24) return launch_mid_nt<BITS, GROUPED, 3, GATED, KSCALE>(h, prm, units, pdl, st);
        if (prm.M <= 32) return launch_mid_nt<BITS, GROUPED, 4, GATED, KSCALE>(h, prm, units, pdl, st);
        if (prm.M <= 48) return launch_mid_nt<BITS, GROUPED, 6, GATED, KSCALE>(h, prm, units, pdl, st);
        return launch_mid_nt<BITS, GROUPED, 8, GATED, KSCALE>(h, prm, units, pdl, st);
    }
}

// n layers that share K and scheme, layer i on xs[i]; act >= 0: the gated form (n == 2, equal shapes, ys[0] the output);
// kscales != nullptr (int8 layers): layer i's input is multiplied by kscales[i][0 .. K).
ql_status forward_mid(const qlinear_s* const* hs, int n, const void* const* xs, void* const* ys, int M, cudaStream_t st, int act = -1,
                      const void* const* kscales = nullptr)
{
    const qlinear_s* h = hs[0];
    const Layout& L = h->L;
    MidParams prm{};
    int units = 0;
    for (int i = 0; i < n; ++i) {
        const Layout& Li = hs[i]->L;
        prm.body[i] = hs[i]->blob + Li.body_offset;
        prm.chan_scales[i] = Li.grouped ? nullptr : reinterpret_cast<const __half*>(hs[i]->blob + Li.chan_scale_offset);
        prm.x[i] = static_cast<const __half*>(xs[i]);
        prm.kscale[i] = static_cast<const __half*>(kscales ? kscales[i] : nullptr);
        prm.y[i] = static_cast<__half*>(ys[act >= 0 ? 0 : i]);
        prm.N[i] = Li.N;
        units += Li.n_rsb;
        prm.unit_end[i] = units;
    }
    if (act >= 0) units = (L.N + 63) / 64;                               // half super-blocks of one layer
    prm.n_layers = n; prm.M = M; prm.K = L.K; prm.n_kc = L.n_kc; prm.act = act >= 0 ? act : 0;
    prm.late = any_cache(hs, n);
    const bool pdl = h->pdl;
    cudaError_t e;
    if (kscales) e = launch_mid<8, false, false, true>(h, prm, units, pdl, st);
    else if (act >= 0) e = L.bits == 8 ? launch_mid<8, false, true>(h, prm, units, pdl, st) : L.grouped ? launch_mid<4, true, true>(h, prm, units, pdl, st) : launch_mid<4, false, true>(h, prm, units, pdl, st);
    else e = L.bits == 8 ? launch_mid<8, false, false>(h, prm, units, pdl, st) : L.grouped ? launch_mid<4, true, false>(h, prm, units, pdl, st) : launch_mid<4, false, false>(h, prm, units, pdl, st);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

template <int NKC, int NT>
cudaError_t launch_gemm_rows_nt(const qlinear_s* h, GemmRowsParams& prm, int n_rsb, bool pdl, cudaStream_t st)
{
    using S = GemmRowsSmem<NKC, NT>;
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemm_rows_kernel<NKC, NT>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, S::kTotal);
    if (e != cudaSuccess) return e;
    prm.n_tb = (prm.M + S::kTokens - 1) / S::kTokens;
    prm.n_tiles = n_rsb * prm.n_tb;
    return launch(kern, prm, dim3(std::min(prm.n_tiles, 2 * h->num_sms)), dim3(256), S::kTotal, st, 1, pdl);
}
template <int NKC>
cudaError_t launch_gemm_rows(const qlinear_s* h, GemmRowsParams& prm, int n_rsb, bool pdl, cudaStream_t st)
{
    if (prm.M <= 16) return launch_gemm_rows_nt<NKC, 2>(h, prm, n_rsb, pdl, st);
    if (prm.M <= 32) return launch_gemm_rows_nt<NKC, 4>(h, prm, n_rsb, pdl, st);
    return launch_gemm_rows_nt<NKC, 8>(h, prm, n_rsb, pdl, st);
}
template <int NKC>
cudaError_t launch_gemm_rows_tc(const qlinear_s* h, const GemmRowsMaps& maps, GemmRowsParams& prm, int n_rsb, cudaStream_t st)
{
    using S = GemmRowsTcSmem<NKC>;
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemm_rows_tc_kernel<NKC>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, S::kTotal);
    if (e != cudaSuccess) return e;
    prm.n_tb = (prm.M + kRowsTcTokens - 1) / kRowsTcTokens;
    prm.n_tiles = n_rsb * prm.n_tb;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(std::min(prm.n_tiles, 2 * h->num_sms));
    cfg.blockDim = dim3(kRowsTcThreads);
    cfg.dynamicSmemBytes = S::kTotal;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = h->pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, maps, prm);
}

// Which of the two kernels for short K a layer takes, the smallest of those in one launch: the tensor-core form has the longer ramp and the
// faster tiles, converts each super-block's weights once for all of its token blocks, and has another order of sums inside an MMA.  The rule
// looks at one layer, so that a head gets the same bits alone and among others: from the tiles of 128 x 64 on at which one layer alone is about
// even, and at d_h = 128 from 3 token blocks on.  Measured, time of gemm_rows_tc_kernel / gemm_rows_kernel, of one layer and of eight:
//   d_h = 64, 1024 tiles (cache 32768, 8192, 2048) 0.99, 0.98, 0.94 and 0.91, 0.85, 0.84; 768 tiles 1.05, 1.04, 1.02 and 0.93, 0.87, 0.85
//   d_h = 128, 512 tiles (16384, 8192, 4096) 1.06, 1.04, 1.00 and 0.89, 0.76, 0.68; 1024 0.86, 0.85, 0.78 and 0.78, 0.69, 0.64
//   d_h = 128, 2 token blocks of 32768 positions 1.06 and 1.07 (40.4 / 43.2 us), 3 0.95 and 0.96
//   d_h = 256, 512 tiles (32768, 16384, 8192, 4096) 0.99, 1.16, 0.97, 0.94 and 0.77, 0.63, 0.53, 0.48
bool rows_take_tc(int layer_rsb, int n_kc, int M, int num_sms)
{
    const int n_tb = (M + kRowsTcTokens - 1) / kRowsTcTokens;
    return (int64_t)layer_rsb * n_tb * 20 >= num_sms * (n_kc == 2 ? 138 : n_kc == 4 ? 69 : 60) && (n_kc != 4 || n_tb >= 3);
}

ql_status forward_gemm_rows(const qlinear_s* const* hs, int n, const void* const* xs, void* const* ys, int M, cudaStream_t st)
{
    const qlinear_s* h = hs[0];
    GemmRowsParams prm{};
    int n_rsb = 0;
    for (int i = 0; i < n; ++i) {
        const Layout& Li = hs[i]->L;
        prm.body[i] = hs[i]->blob + Li.body_offset;
        prm.chan_scales[i] = reinterpret_cast<const __half*>(hs[i]->blob + Li.chan_scale_offset);
        prm.x[i] = static_cast<const __half*>(xs[i]);
        prm.y[i] = static_cast<__half*>(ys[i]);
        prm.N[i] = Li.N;
        n_rsb += Li.n_rsb;
        prm.rsb_end[i] = n_rsb;
    }
    prm.n_layers = n; prm.M = M;
    const bool pdl = h->pdl;                                             // (every byte is read after griddepcontrol.wait)
    const int n_kc = h->L.n_kc;
    int layer_rsb = h->L.n_rsb;
    for (int i = 1; i < n; ++i) layer_rsb = std::min(layer_rsb, hs[i]->L.n_rsb);
    if (rows_take_tc(layer_rsb, n_kc, M, h->num_sms)) {
        GemmRowsMaps maps;
        for (int i = 0; i < kRowsMaxLayers; ++i)
            if (!x_tensor_map(xs[i < n ? i : 0], h->L.K, M, kRowsTcTokens, &maps.x[i])) return QL_ERR_CUDA;
        const cudaError_t e = n_kc == 2 ? launch_gemm_rows_tc<2>(h, maps, prm, n_rsb, st) : n_kc == 4 ? launch_gemm_rows_tc<4>(h, maps, prm, n_rsb, st) : launch_gemm_rows_tc<8>(h, maps, prm, n_rsb, st);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
    }
    const cudaError_t e = n_kc == 2 ? launch_gemm_rows<2>(h, prm, n_rsb, pdl, st) : n_kc == 4 ? launch_gemm_rows<4>(h, prm, n_rsb, pdl, st) : launch_gemm_rows<8>(h, prm, n_rsb, pdl, st);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

GemmPairLayers pair_layers(const qlinear_s* const* hs, int n, void* const* ys)
{
    GemmPairLayers set{};
    set.n = n;
    set.late = any_cache(hs, n);
    for (int i = 0; i < n; ++i) {
        set.L[i] = &hs[i]->L; set.blob[i] = hs[i]->blob; set.y[i] = ys ? ys[i] : nullptr;
        set.wmap[i] = hs[i]->wmap_ok ? &hs[i]->wmap : nullptr;
    }
    return set;
}

// The unfused gating route's two projections fit the device's scratch.
bool gate_fits_scratch(int N, int M, int num_sms) { return (size_t)M * N * 2 * sizeof(__half) <= gemm_pair_scratch_bytes(num_sms); }

// Estimates of a launch, us, as consecutive launches with the weights out of HBM take it: what lies between gemm_narrow.cuh and the kernels
// that served its calls before.  Fitted to 9217 calls of random shapes (8 to 32768 channels, K 32 to 16384, at most 80 million weights, 9 to 2048
// tokens, plain and gated, the three schemes), each on both routes; long calls and the shapes of the two models weigh more.  Measured /
// estimate, 5th and 95th percentile (1st and 99th): narrow_us 0.90 and 1.11 (0.84, 1.17), mid_us 0.90 and 1.11 (0.85, 1.16), prefill_us on the
// CTA-pair kernel's plans of the fewest blocks 0.83 and 1.19 (0.81, 1.70: gated pairs of K up to 128, far from the line; those it searches, of 700 later
// calls: 0.88 and 1.12), on the single-CTA kernel 0.86 and 1.07 (0.79, 1.17), unfused 0.86 and 1.05 (0.81, 1.13).  The fused gated forms of more
// than 128 tokens have estimates of their own (narrow_gated_us, gemm_pair_ta_us, gemm_pair_gated_us).
// What a CTA's time is multiplied by for the others of the launch, `ctas` in all in clusters of cl, two to an SM: up to one per SM they slow it
// down by `first`, the second ones by `second` more; beyond two per SM further rounds, of which the last one costs `last` at least.
// (Clusters of 4 and 8 lie inside a GPC: fewer fit.)
double sm_load(double ctas, int cl, int num_sms, double first, double second, double last)
{
    const double u = ctas / (num_sms * (cl == 8 ? 0.87 : cl == 4 ? 0.97 : 1.0));
    if (u <= 2.0) return 1.0 + first * std::min(u, 1.0) + second * std::max(u - 1.0, 0.0);
    return (1.0 + first + second) * std::min(round_up(u / 2.0), u / 2.0 + last);
}

int total_rsb(const qlinear_s* const* hs, int n) { int t = 0; for (int i = 0; i < n; ++i) t += hs[i]->L.n_rsb; return t; }
double out_mb(const qlinear_s* const* hs, int n, int M) { double t = 0; for (int i = 0; i < n; ++i) t += 2e-6 * M * hs[i]->L.N; return t; }

// Gated pairs that the kernels of CTA pairs can serve as well, which was a corner of the calls that the estimate below was made with: fitted to 1675
// such pairs of 129 to 4096 tokens, measured / estimate 0.93 and 1.10 (the other one: 0.82 and 1.18).
double narrow_gated_us(const qlinear_s* const* hs, int M)
{
    const Layout& L = hs[0]->L;
    const NarrowPlan pl = plan_narrow(L, L.n_rsb, true, M, hs[0]->num_sms);
    const int steps = ((L.K + kNarrowKStep - 1) / kNarrowKStep + pl.cl - 1) / pl.cl * 2;
    const double cta = steps * (L.bits == 4 ? 0.304 : 0.289) + 0.63 + 0.0342 * pl.bn;
    return 0.92 + 0.77 * log2_of(pl.cl) + sm_load((double)L.n_rsb * pl.n_tb * pl.cl, pl.cl, hs[0]->num_sms, 0.672, 0.205, 0.408) * cta;
}

double narrow_us(const qlinear_s* const* hs, int n, int M, bool gated)
{
    const Layout& L = hs[0]->L;
    if (gated && gemm_pair_applicable(L, M)) return narrow_gated_us(hs, M);
    const int rows = gated ? L.n_rsb : total_rsb(hs, n);
    const NarrowPlan pl = plan_narrow(L, rows, gated, M, hs[0]->num_sms);
    const int steps = ((L.K + kNarrowKStep - 1) / kNarrowKStep + pl.cl - 1) / pl.cl * (gated ? 2 : 1);
    const double cta = steps * (L.bits == 4 ? 0.350 : 0.391) + 1.44 + pl.bn * (0.0204 + (pl.cl == 1 ? 0.0 : gated ? 0.0197 : 0.0067));
    return 0.47 + 0.087 * log2_of(pl.cl) + sm_load((double)rows * pl.n_tb * pl.cl, pl.cl, hs[0]->num_sms, 0.489, 0.259, 0.37) * cta;
}

double mid_us(const qlinear_s* const* hs, int n, int M, bool gated)      // up to 64 tokens
{
    const Layout& L = hs[0]->L;
    const int nt = M <= 16 ? 2 : M <= 24 ? 3 : M <= 32 ? 4 : M <= 48 ? 6 : 8, units = gated ? (L.N + 63) / 64 : total_rsb(hs, n);
    const int n_steps = (L.n_kc + 1) / 2, cl = mid_parts(units, n_steps, hs[0]->num_sms);
    const double step = L.bits == 8 ? 0.113 + 0.0511 * nt : 0.174 + 0.0886 * nt;
    const double cta = (n_steps + cl - 1) / cl * step + 0.313 + nt * (0.127 + (cl > 1 ? 0.054 : 0.0));
    return 0.96 + 0.093 * log2_of(cl) + sm_load((double)units * cl, cl, hs[0]->num_sms, 0.772, 0.252, 0.46) * cta;
}

double pair_ta_fewest_us(int bn, int rounds, int steps, int split, double mb)   // plans of the fewest blocks
{
    return 2.66 + 0.0058 * bn + rounds * (((steps + split - 1) / split) * (0.236 + 0.0003 * bn)) + (split > 1 ? 6.2 + 0.0162 * bn : 0.0) + 0.34 * mb;
}

double pair_ta_us(const Layout& L, int pairs, int M, bool split, double mb, int num_sms)
{
    const int steps = (L.K + kGemmKStep - 1) / kGemmKStep, clusters = num_sms / 2;
    const TaPlan pl = gemm_pair_ta_plan(pairs, M, steps, 1, false, num_sms, split);
    if (gemm_pair_ta_searches(pairs, M, steps, false)) return gemm_pair_ta_us(pairs, pl.n_mblk, pl.bn, pl.split, steps, 1, false, false, num_sms) + 0.286 * mb;
    return pair_ta_fewest_us(pl.bn, (pairs * pl.n_mblk * pl.split + clusters - 1) / clusters, steps, pl.split, mb);
}

double pair_ta_gated_us(const Layout& L, int M, double mb, int num_sms)
{
    const bool both = gemm_pair_ta_both(L, M, num_sms);
    const TaPlan pl = gemm_pair_ta_gated_plan(L, M, num_sms);            // (what the launch takes)
    return gemm_pair_ta_us(L.n_rsb / 2, pl.n_mblk, pl.bn, 1, (L.K + kGemmKStep - 1) / kGemmKStep, 2, both, false, num_sms) + (both ? 0.56 : 0.53) * mb;
}

double single_us(const Layout& L, int M, double mb, int num_sms)
{
    const int bn = gemm_pick_bn(L, M, num_sms), steps = (L.K + kGemmKStep - 1) / kGemmKStep;
    const double w = (double)L.n_rsb * ((M + bn - 1) / bn) / num_sms;
    return 4.5 + 0.0038 * bn + std::max(1.0, std::min(round_up(w), w + 0.76)) * (0.0175 * bn + steps * (0.203 + 0.0011 * bn)) + 0.28 * mb;
}

// `kernel`: what prefill_kernel says of the call.
double prefill_us(ql_kernel kernel, const qlinear_s* const* hs, int n, int M, bool gated)
{
    const Layout& L = hs[0]->L;
    const int sms = hs[0]->num_sms;
    const double mb = out_mb(hs, gated ? 1 : n, M);
    if (kernel == QL_KERNEL_SINGLE) return single_us(L, M, mb, sms);
    if (kernel == QL_KERNEL_SEPARATE) {
        if (gated && L.n_rsb % 2 == 0) return 4.2 + pair_ta_us(L, L.n_rsb, M, false, 2 * mb, sms) + 0.92 * mb;
        double us = gated ? 1.7 + 0.92 * mb : 0.0;
        for (int i = 0; i < n; ++i) {
            const Layout& Li = hs[i]->L;
            const double m = out_mb(hs + i, 1, M);
            us += Li.n_rsb % 2 ? single_us(Li, M, m, sms) : pair_ta_us(Li, Li.n_rsb / 2, M, true, m, sms);
        }
        return us;
    }
    if (gated && kernel == QL_KERNEL_PAIR) return gemm_pair_gated_us(L, M, mb, sms);
    return gated ? pair_ta_gated_us(L, M, mb, sms) : pair_ta_us(L, total_rsb(hs, n) / 2, M, true, mb, sms);
}

ql_kernel prefill_kernel(const qlinear_s* const* hs, int n, int M, bool gated)
{
    const Layout& L = hs[0]->L;
    const int sms = hs[0]->num_sms;
    const GemmPairLayers set = pair_layers(hs, n, nullptr);
    if (gated && !gemm_pair_applicable(L, M)) return QL_KERNEL_SEPARATE;
    if (gemm_pair_ta_applicable(set, M, sms, gated)) return QL_KERNEL_PAIR_TA;
    for (int i = 0; i < n; ++i)
        if (!gemm_pair_applicable(hs[i]->L, M)) return n > 1 ? QL_KERNEL_SEPARATE : QL_KERNEL_SINGLE;
    return QL_KERNEL_PAIR;
}

// Whether gemm_narrow.cuh can serve the call at all.  (QLINEAR_MID_MAX_M < M <= 64: the prefill kernels, whatever the estimate.  A pair whose
// unfused product does not fit the scratch has only ever been served by the fused kernels of the prefill stage.)
bool narrow_can(const qlinear_s* const* hs, int n, int M, bool gated, bool batch)
{
    if (config().narrow == 0 || (M <= 64 && M > config().mid_max_m)) return false;
    for (int i = 0; i < n; ++i)
        if (!hs[i]->wmap_wide_ok) return false;
    return batch || !gated || gate_fits_scratch(hs[0]->L.N, M, hs[0]->num_sms) || gemm_pair_applicable(hs[0]->L, M);
}

// The kernel of a call beyond the decode stage: one layer, n > 1 layers that share x, or (gated) a pair.  gemm_narrow.cuh where its
// estimate is below that of gemm_mid.cuh, the CTA-pair kernel or the three other forms (single CTA, shared-memory gating, unfused gating).  No line is always right with these errors.  Of the calls above and 3110 others, 63 run more than 3 %
// slower this way than on the other route: 54 of 4821 against gemm_mid.cuh (two of them by 46 and 26 %, the others by 24 % at most), 9
// of 5488 against the other forms (9 %).  Against the CTA-pair kernel with its plans searched, 700 calls take 0.3 % more than on the faster route each,
// the worst 21 %.  1676 gated pairs of 129 to 4096 tokens, timed on every form and width: 1.3 % more than on the fastest, the worst 26 %.  Measured, us, the route otherwise / gemm_narrow.cuh:
//   weights                        16 tokens     24           32           48           64
//     0.3 M (512 x 512)             2.8 /  3.7   3.0 /  3.8   3.3 /  4.0   3.8 /  4.2   4.1 /  4.5
//     1 M (1024 x 1024, int8)       3.2 /  4.3   3.5 /  4.5   4.0 /  4.6   4.6 /  5.0   5.2 /  5.3
//     5 M (gated 2688 x 1024)       4.1 /  5.1   4.7 /  5.5   5.5 /  5.8   7.1 /  6.8   8.5 /  7.6
//     9 M (Gemma2-2B q + k + v)     5.0 /  5.8   5.8 /  6.3   6.9 /  6.4   8.9 /  7.3  10.5 /  7.9
//    21 M (its down)                8.9 /  8.9  11.2 /  9.3  12.8 /  9.6  16.7 / 10.2  20.9 / 11.5
//    25 M (Llama q + k + v)         8.8 /  9.1  10.8 /  9.4  12.3 /  9.6  16.7 / 11.4
//    42 M (Gemma2-2B gate + up)     9.4 / 12.4  11.6 / 12.7  13.2 / 13.6  16.6 / 14.6  19.7 / 14.8
//    59 M (Llama down)             13.8 / 13.5  16.6 / 14.0  18.9 / 14.3               27.9 / 15.8
//   117 M (Llama gate + up)        26.0 / 22.7  31.9 / 23.2  37.0 / 23.6               43.8 / 26.0
ql_kernel gemm_route(const qlinear_s* const* hs, int n, int M, bool gated)
{
    const Layout& L = hs[0]->L;
    if (n == 1 && takes_rows(L)) return rows_take_tc(L.n_rsb, L.n_kc, M, hs[0]->num_sms) ? QL_KERNEL_ROWS_TC : QL_KERNEL_ROWS;
    const bool batch = takes_mid(hs, n, M, gated);
    const ql_kernel other = batch ? QL_KERNEL_MID : prefill_kernel(hs, n, M, gated);
    if (!narrow_can(hs, n, M, gated, batch)) return other;
    if (config().narrow == 2) return QL_KERNEL_NARROW;
    // (Pairs that the kernels of CTA pairs can serve: up to 4 % above.  With one accumulator they round act(gate) to fp16, which this one doesn't.)
    const double lean = gated && gemm_pair_applicable(L, M) ? 1.04 : 1.0;
    return narrow_us(hs, n, M, gated) < (batch ? mid_us(hs, n, M, gated) : lean * prefill_us(other, hs, n, M, gated)) ? QL_KERNEL_NARROW : other;
}

// y = act(g) * u, element-wise (the unfused form of the gating, for shapes the fused kernels do not take).
__global__ void __launch_bounds__(256) gate_mul_kernel(const __half* g, const __half* u, __half* y, int64_t n, int act)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        y[i] = __float2half_rn(gate_activation(__half2float(g[i]), act) * __half2float(u[i]));
}

template <int BITS, bool GROUPED, int NS>
cudaError_t launch_stream_ns(const qlinear_s* h, const StreamParams& prm, cudaStream_t st)
{
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemv_stream_kernel<BITS, GROUPED, NS>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, NS * StreamStage<BITS>::kBytes);
    if (e != cudaSuccess) return e;
    return launch(kern, prm, dim3(prm.P), dim3(kStreamThreads), (size_t)NS * StreamStage<BITS>::kBytes, st, 1, h->early());
}

template <int BITS, bool GROUPED>
cudaError_t launch_stream(const qlinear_s* h, const StreamParams& prm, cudaStream_t st)
{
    switch (prm.stages) {
        case 6: return launch_stream_ns<BITS, GROUPED, 6>(h, prm, st);
        case 8: return launch_stream_ns<BITS, GROUPED, 8>(h, prm, st);
        case 12: return launch_stream_ns<BITS, GROUPED, 12>(h, prm, st);
        case 16: return launch_stream_ns<BITS, GROUPED, 16>(h, prm, st);
    }
    return cudaErrorInvalidValue;
}

ql_status forward_gemv_stream(const qlinear_s* h, const void* x, void* y, int M, cudaStream_t st)
{
    const Layout& L = h->L;
    StreamParams prm{};
    prm.body = h->blob + L.body_offset;
    prm.chan_scales = L.grouped ? nullptr : reinterpret_cast<const __half*>(h->blob + L.chan_scale_offset);
    prm.x = static_cast<const __half*>(x);
    prm.y = static_cast<__half*>(y);
    prm.scratch = h->dev->stream_scratch;
    prm.counters = h->dev->stream_counters;
    prm.M = M; prm.N = L.N; prm.K = L.K;
    prm.n_rsb = L.n_rsb; prm.n_kc = L.n_kc; prm.block_bytes = L.block_bytes;
    prm.P = h->stream_P;
    prm.stages = h->stream_stages;
    cudaError_t e;
    if (L.bits == 8) e = launch_stream<8, false>(h, prm, st);
    else if (L.grouped) e = launch_stream<4, true>(h, prm, st);
    else e = launch_stream<4, false>(h, prm, st);
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

// The CTA-pair prefill kernels: `kernel` says which (QL_KERNEL_PAIR_TA, QL_KERNEL_PAIR); act >= 0: both accumulators for a gated pair.
ql_status forward_pair(const qlinear_s* const* hs, int n, ql_kernel kernel, const void* x, void* const* ys, int M, cudaStream_t st, int act = -1)
{
    const qlinear_s* h = hs[0];
    const GemmPairLayers set = pair_layers(hs, n, ys);
    if (act >= 0) return kernel == QL_KERNEL_PAIR_TA ? gemm_pair_ta_forward_gated(set, x, M, act, st, h->device, h->pdl, h->num_sms)
                                                     : gemm_pair_forward_gated(set, x, M, act, st, h->device, h->pdl, h->num_sms);
    return kernel == QL_KERNEL_PAIR_TA ? gemm_pair_ta_forward(set, x, M, st, h->device, h->pdl, h->num_sms, h->dev->gemm_scratch, h->dev->gemm_counters)
                                       : gemm_pair_forward(set, x, M, st, h->device, h->pdl, h->num_sms, h->dev->gemm_scratch, h->dev->gemm_counters);
}

// ---- debug: the integers as the device unpack routines see them
template <int BITS>
__global__ void __launch_bounds__(256) debug_unpack_kernel(const uint8_t* body, int8_t* q_out, int N, int K,
                                                           int n_kc, int block_bytes)
{
    const int rsb = blockIdx.y, kc = blockIdx.x;
    const int rb = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    const uint8_t* blk = body + ((int64_t)rsb * n_kc + kc) * block_bytes;
    const uint4 w = *reinterpret_cast<const uint4*>(blk + rb * 512 + lane * 16);
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
    const int row0 = rsb * kRsbRows + rb * kRbRows + g;
    constexpr int NMMA = BITS == 4 ? 4 : 2;
#pragma unroll
    for (int i = 0; i < NMMA; ++i) {
        uint32_t a[4];
        if (BITS == 4) unpack_int4_word(ww[i], a);
        else unpack_int8_words(ww[2 * i], ww[2 * i + 1], a);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const __half2 hv = *reinterpret_cast<const __half2*>(&a[r]);
            const int row = row0 + 8 * (r & 1);
            const int j = 2 * (r >> 1);
            const int kbase = BITS == 4 ? kc * 64 + int4_k_in_chunk(c, i, j) : kc * 32 + 8 * c + 4 * i + j;
            if (row < N && kbase < K) {
                q_out[(int64_t)row * K + kbase] = (int8_t)__half2int_rn(__low2half(hv));
                q_out[(int64_t)row * K + kbase + 1] = (int8_t)__half2int_rn(__high2half(hv));
            }
        }
    }
}

// Test aid: the bounded wait of the kernels on a barrier that nothing completes.
__global__ void __launch_bounds__(32) expire_wait_kernel()
{
    __shared__ __align__(8) unsigned long long bar;
    __shared__ volatile uint32_t abort_word[3];                          // [0] abort, [2] "dependency resolved"
    if (threadIdx.x == 0) {
        abort_word[0] = 0;
        abort_word[1] = 0;
        abort_word[2] = 1;
        mbar_init(smem_u32(&bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait<true>(smem_u32(&bar), 0, abort_word, 0x9A0);   // gives up, records the code
}

struct DeviceGuard {
    int prev = -1;
    bool ok = true;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
        if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
        if (prev == dev) prev = -1;
    }
    ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

}  // namespace

namespace {

// Creates the device's shared state on first use (the device must be current).  Called under g_dev_mutex.
ql_status device_state_init(int device, int sms, DeviceState* d)
{
    if (d->ready) return QL_OK;
    const Config& cfg = config();
    d->sms = sms;
    const size_t cb = gemm_pair_counter_count(sms) * sizeof(unsigned int);
    bool ok = cudaHostAlloc(reinterpret_cast<void**>(&d->status_host), 64, cudaHostAllocMapped | cudaHostAllocPortable) == cudaSuccess;
    unsigned int* status_dev = nullptr;
    if (ok) {
        d->status_host[0] = 0;
        ok = cudaHostGetDevicePointer(reinterpret_cast<void**>(&status_dev), d->status_host, 0) == cudaSuccess &&
             cudaMemcpyToSymbol(g_status_host, &status_dev, sizeof(status_dev)) == cudaSuccess;
    }
    ok = ok && cudaMalloc(&d->gemm_scratch, gemm_pair_scratch_bytes(sms)) == cudaSuccess &&
         cudaMalloc(&d->gemm_counters, cb) == cudaSuccess && cudaMemset(d->gemm_counters, 0, cb) == cudaSuccess;
    if (ok && cfg.kernel == 2) {
        const size_t sbytes = (size_t)sms * 4 * 2 * kStreamPartialFloats * sizeof(float);
        const size_t cbytes = (size_t)kStreamMaxRsb * 8 * sizeof(unsigned int);
        ok = cudaMalloc(&d->stream_scratch, sbytes) == cudaSuccess && cudaMalloc(&d->stream_counters, cbytes) == cudaSuccess &&
             cudaMemset(d->stream_counters, 0, cbytes) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        unsigned int* null_ptr = nullptr;
        cudaMemcpyToSymbol(g_status_host, &null_ptr, sizeof(null_ptr));
        cudaFreeHost(d->status_host); cudaFree(d->gemm_scratch); cudaFree(d->gemm_counters);
        cudaFree(d->stream_scratch); cudaFree(d->stream_counters);
        cudaGetLastError();
        *d = DeviceState{};
        return QL_ERR_CUDA;
    }
    d->ready = true;
    return QL_OK;
}

// An earlier kernel on this device gave up a bounded wait: the host sees the code without synchronising.
inline bool device_timed_out(const qlinear_s* h)
{
    return *reinterpret_cast<volatile unsigned int*>(h->dev->status_host) != 0;
}

}  // namespace

extern "C" ql_status qlinear_create(const qlinear_desc* d, const void* packed_dev, int device, qlinear_t* out)
{
    if (!d || !packed_dev || !out) return QL_ERR_INVALID_ARG;
    *out = nullptr;
    Layout L;
    if (!make_layout(d->N, d->K, d->bits, d->group, &L)) return QL_ERR_UNSUPPORTED;
    if (reinterpret_cast<uintptr_t>(packed_dev) % 256) return QL_ERR_INVALID_ARG;
    int n_dev = 0;
    if (cudaGetDeviceCount(&n_dev) != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
    if (device < 0 || device >= n_dev || device >= kMaxDevices) return QL_ERR_INVALID_ARG;
    int major = 0, sms = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return QL_ERR_CUDA;
    if (major != 10) return QL_ERR_ARCH;
    const Config& cfg = config();
    qlinear_s* h = new (std::nothrow) qlinear_s();
    if (!h) return QL_ERR_ALLOC;
    h->L = L;
    h->blob = static_cast<const uint8_t*>(packed_dev);
    h->device = device;
    h->num_sms = sms;
    h->gemv_max_m = cfg.gemv_max_m;
    h->pdl = cfg.pdl;
    h->n_rb = (L.N + kRbRows - 1) / kRbRows;
    h->wmap_ok = w_tensor_map(L, h->blob, &h->wmap);
    h->wmap_wide_ok = w_tensor_map(L, h->blob, &h->wmap_wide, true);
    for (int M = 1; M <= 8; ++M) {
        h->gemv[M] = plan_gemv(L, h->n_rb, M, sms);
        if (h->gemv[M].grid <= 0 && M <= h->gemv_max_m) { delete h; return QL_ERR_UNSUPPORTED; }   // no decode plan fits this shape
    }
    {
        // streaming decode kernel (QLINEAR_GEMV_KERNEL=stream): persistent grid and ring depth
        const int stage_bytes = L.bits == 4 ? StreamStage<4>::kBytes : StreamStage<8>::kBytes;
        const int max_stages = std::min(cfg.stream_stages, (220 * 1024 / cfg.stream_ctas_per_sm - 1536) / stage_bytes);
        h->stream_stages = max_stages >= 16 ? 16 : max_stages >= 12 ? 12 : max_stages >= 8 ? 8 : 6;   // instantiated ring depths
        const int64_t B = (int64_t)L.n_rsb * L.n_kc;
        h->stream_P = (int)std::min<int64_t>(B, (int64_t)sms * cfg.stream_ctas_per_sm);
        // the streaming kernel reads whole 64-k slices of x and shares counters sized for kStreamMaxRsb row super-blocks
        h->use_stream = cfg.kernel == 2 && !(L.bits == 4 && (L.K % 64)) && L.n_rsb <= kStreamMaxRsb;
    }
    {
        DeviceGuard guard(device);
        std::lock_guard<std::mutex> lock(g_dev_mutex);
        ql_status st = guard.ok ? device_state_init(device, sms, &g_dev[device]) : QL_ERR_CUDA;
        if (st != QL_OK) { cudaGetLastError(); delete h; return st; }
        h->dev = &g_dev[device];
        ++h->dev->handles;
    }
    *out = h;
    return QL_OK;
}

extern "C" int32_t qlinear_path_for(qlinear_t h, int32_t M)
{
    if (!h || M < 1) return 0;
    return M <= h->gemv_max_m ? QL_PATH_GEMV : QL_PATH_GEMM;
}

extern "C" ql_status qlinear_forward(qlinear_t h, const void* x, void* y, int32_t M, void* stream)
{
    if (!h || !x || !y || M < 1) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) return QL_ERR_INVALID_ARG;
    if ((int64_t)M * h->L.K > INT32_MAX || (int64_t)M * h->L.N > INT32_MAX) return QL_ERR_INVALID_ARG;
    if (device_timed_out(h)) return QL_ERR_DEVICE_TIMEOUT;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (M <= h->gemv_max_m) {
        if (h->use_stream) return forward_gemv_stream(h, x, y, M, st);
        return forward_gemv(&h, 1, x, &y, M, st, -1, takes_rows(h->L) ? &x : nullptr);   // (short K: the persistent form, see there)
    }
    const ql_kernel kernel = gemm_route(&h, 1, M, false);
    switch (kernel) {
        case QL_KERNEL_ROWS:
        case QL_KERNEL_ROWS_TC: return forward_gemm_rows(&h, 1, &x, &y, M, st);
        case QL_KERNEL_MID: return forward_mid(&h, 1, &x, &y, M, st);
        case QL_KERNEL_NARROW: return forward_narrow(&h, 1, x, &y, M, st);
        case QL_KERNEL_PAIR_TA:
        case QL_KERNEL_PAIR: return forward_pair(&h, 1, kernel, x, &y, M, st);
        default: return gemm_forward(h->L, h->blob, x, y, M, st, h->device, h->pdl, h->num_sms, any_cache(&h, 1));
    }
}

extern "C" ql_status qlinear_forward_group(const qlinear_t* hs, int32_t n, const void* x, void* const* ys, int32_t M, void* stream)
{
    if (!hs || !ys || !x || n < 1 || n > kGemvMaxGroup || M < 1) return QL_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i) {
        if (!hs[i] || !ys[i] || (reinterpret_cast<uintptr_t>(ys[i]) & 15)) return QL_ERR_INVALID_ARG;
        const Layout &a = hs[0]->L, &b = hs[i]->L;
        if (hs[i]->device != hs[0]->device || a.K != b.K || a.bits != b.bits || a.group != b.group) return QL_ERR_INVALID_ARG;
        if ((int64_t)M * b.N > INT32_MAX) return QL_ERR_INVALID_ARG;
    }
    if ((reinterpret_cast<uintptr_t>(x) & 15) || (int64_t)M * hs[0]->L.K > INT32_MAX) return QL_ERR_INVALID_ARG;
    if (device_timed_out(hs[0])) return QL_ERR_DEVICE_TIMEOUT;
    // One kernel where the decode kernel serves the call; otherwise the layers run one after the other.
    if (n > 1 && M <= hs[0]->gemv_max_m && !hs[0]->use_stream) {
        DeviceGuard guard(hs[0]->device);
        if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
        return forward_gemv(const_cast<qlinear_s* const*>(hs), n, x, ys, M, static_cast<cudaStream_t>(stream));
    }
    if (n > 1 && M > hs[0]->gemv_max_m) {
        const ql_kernel kernel = gemm_route(hs, n, M, false);
        if (kernel != QL_KERNEL_SEPARATE) {
            DeviceGuard guard(hs[0]->device);
            if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
            const void* xs[kGemvMaxGroup];
            for (int i = 0; i < n; ++i) xs[i] = x;
            if (kernel == QL_KERNEL_MID) return forward_mid(hs, n, xs, ys, M, static_cast<cudaStream_t>(stream));
            if (kernel == QL_KERNEL_NARROW) return forward_narrow(hs, n, x, ys, M, static_cast<cudaStream_t>(stream));
            return forward_pair(hs, n, kernel, x, ys, M, static_cast<cudaStream_t>(stream));
        }
    }
    for (int i = 0; i < n; ++i) {
        ql_status s = qlinear_forward(hs[i], x, ys[i], M, stream);
        if (s != QL_OK) return s;
    }
    return QL_OK;
}

extern "C" ql_status qlinear_forward_batch(const qlinear_t* hs, int32_t n, const void* const* xs, void* const* ys, int32_t M, void* stream)
{
    if (!hs || !xs || !ys || n < 1 || n > kGemvMaxBatch || M < 1) return QL_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i) {
        if (!hs[i] || !xs[i] || !ys[i] || ((reinterpret_cast<uintptr_t>(xs[i]) | reinterpret_cast<uintptr_t>(ys[i])) & 15)) return QL_ERR_INVALID_ARG;
        const Layout &a = hs[0]->L, &b = hs[i]->L;
        if (hs[i]->device != hs[0]->device || a.K != b.K || a.bits != b.bits || a.group != b.group) return QL_ERR_INVALID_ARG;
        if ((int64_t)M * b.N > INT32_MAX || (int64_t)M * b.K > INT32_MAX) return QL_ERR_INVALID_ARG;
    }
    if (device_timed_out(hs[0])) return QL_ERR_DEVICE_TIMEOUT;
    if (n > 1 && M <= hs[0]->gemv_max_m && !hs[0]->use_stream) {         // one decode launch for all of them
        DeviceGuard guard(hs[0]->device);
        if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
        const ql_status s = forward_gemv(const_cast<qlinear_s* const*>(hs), n, nullptr, ys, M, static_cast<cudaStream_t>(stream), -1, xs);
        if (s != QL_ERR_UNSUPPORTED) return s;
    }
    if (n > 1 && M > hs[0]->gemv_max_m && takes_rows(hs[0]->L)) {   // (the K caches of a prompt's attention)
        DeviceGuard guard(hs[0]->device);
        if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
        return forward_gemm_rows(hs, n, xs, ys, M, static_cast<cudaStream_t>(stream));
    }
    for (int i = 0; i < n; ++i) {                                        // anything else: one call per layer
        const ql_status s = qlinear_forward(hs[i], xs[i], ys[i], M, stream);
        if (s != QL_OK) return s;
    }
    return QL_OK;
}

extern "C" ql_status qlinear_forward_gated(qlinear_t hg, qlinear_t hu, const void* x, void* y, int32_t M, int32_t act, void* stream)
{
    if (!hg || !hu || !x || !y || M < 1) return QL_ERR_INVALID_ARG;
    if (act != QL_ACT_IDENTITY && act != QL_ACT_SILU && act != QL_ACT_GELU_TANH) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) return QL_ERR_INVALID_ARG;
    const Layout &a = hg->L, &b = hu->L;
    if (hg->device != hu->device || a.N != b.N || a.K != b.K || a.bits != b.bits || a.group != b.group) return QL_ERR_INVALID_ARG;
    if ((int64_t)M * a.K > INT32_MAX || (int64_t)M * a.N > INT32_MAX) return QL_ERR_INVALID_ARG;
    if (device_timed_out(hg)) return QL_ERR_DEVICE_TIMEOUT;
    DeviceGuard guard(hg->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    qlinear_s* hs[2] = {hg, hu};
    if (M <= hg->gemv_max_m && !hg->use_stream) {                        // decode: both branches in one launch
        void* ys[2] = {y, y};
        const ql_status s = forward_gemv(hs, 2, x, ys, M, st, act);
        if (s != QL_ERR_UNSUPPORTED) return s;
    } else if (M > hg->gemv_max_m) {
        const ql_kernel kernel = gemm_route(hs, 2, M, true);
        const void* xs[2] = {x, x};
        void* ys[2] = {y, y};
        if (kernel == QL_KERNEL_MID) return forward_mid(hs, 2, xs, &y, M, st, act);
        if (kernel == QL_KERNEL_NARROW) return forward_narrow(hs, 2, x, ys, M, st, act);
        if (kernel != QL_KERNEL_SEPARATE) return forward_pair(hs, 2, kernel, x, ys, M, st, act);
    }
    // Unfused: the two projections into the device's shared scratch, then the element-wise product.
    if (!gate_fits_scratch(a.N, M, hg->num_sms)) return QL_ERR_UNSUPPORTED;
    const int64_t n = (int64_t)M * a.N;
    __half* g = reinterpret_cast<__half*>(hg->dev->gemm_scratch);
    __half* u = g + ((n + 7) & ~(int64_t)7);
    void* ys[2] = {g, u};
    ql_status s = qlinear_forward_group(hs, 2, x, ys, M, stream);
    if (s != QL_OK) return s;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)hg->num_sms * 8);
    gate_mul_kernel<<<blocks, 256, 0, st>>>(g, u, static_cast<__half*>(y), n, act);
    return cudaGetLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

namespace {
template <int BITS, bool GROUPED, int T>
cudaError_t launch_a8_t(const qlinear_s* h, const GemvA8Params& prm, const GemvPlan& pl, cudaStream_t st)
{
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemv_a8_kernel<BITS, GROUPED, T>;
    cudaError_t e = ensure_smem_attr(kern, attr_set, h->device, kGemvMaxSmem);
    if (e != cudaSuccess) return e;
    return launch(kern, prm, dim3(pl.grid), dim3(kGemvThreads), pl.smem_bytes, st, pl.cl, h->early());
}
template <int BITS, bool GROUPED>
cudaError_t launch_a8(const qlinear_s* h, const GemvA8Params& prm, const GemvPlan& pl, cudaStream_t st)
{
    if (prm.M == 1) return launch_a8_t<BITS, GROUPED, 1>(h, prm, pl, st);
    if (prm.M == 2) return launch_a8_t<BITS, GROUPED, 2>(h, prm, pl, st);
    if (prm.M <= 4) return launch_a8_t<BITS, GROUPED, 4>(h, prm, pl, st);
    return launch_a8_t<BITS, GROUPED, 8>(h, prm, pl, st);
}
}  // namespace

namespace {
cudaError_t launch_quantize(const __half* x, signed char* xq, float* scale, int32_t* rowsum, int M, int K, cudaStream_t st, bool pdl)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(M);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, quantize_activations_kernel, x, xq, scale, rowsum, M, K);
}
}  // namespace

// Bytes of the device's scratch that a prompt with int8 activations uses: the quantised rows, the per-token arrays behind them (padded to
// whole 256-token tiles) and, where the scratch holds them as well, the K parts of launches of few tiles.
namespace {
struct A8Scratch {
    size_t xq, arr;
    bool fits, parts;
};
A8Scratch a8_scratch(int M, int K, int num_sms)
{
    A8Scratch s;
    s.xq = (((size_t)M * K + 255) / 256) * 256;
    s.arr = (size_t)((M + 255) / 256) * 256 * 4;
    const size_t used = s.xq + 2 * s.arr, all = gemm_pair_scratch_bytes(num_sms);
    s.fits = used <= all;
    s.parts = used + (size_t)(num_sms / 2) * 2 * 256 * 128 * sizeof(float) <= all;
    return s;
}
}  // namespace

extern "C" ql_status qlinear_forward_a8(qlinear_t h, const void* x, void* y, int32_t M, void* stream)
{
    if (!h || !x || !y || M < 1) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) return QL_ERR_INVALID_ARG;
    if (device_timed_out(h)) return QL_ERR_DEVICE_TIMEOUT;
    const Layout& L = h->L;
    if (M > h->gemv_max_m) {
        // Prefill stage (Section 3.7): the quantisation kernel, then the integer matmul with output dequantisation.
        // Built for the per-channel schemes on the CTA-pair kernel; the quantised activations live in the device's
        // shared scratch (calls must be ordered against other users of it).
        if (L.grouped || (L.K % 128) || !gemm_pair_applicable(L, M)) return QL_ERR_UNSUPPORTED;
        const A8Scratch sc = a8_scratch(M, L.K, h->num_sms);
        if (!sc.fits) return QL_ERR_UNSUPPORTED;
        DeviceGuard guard(h->device);
        if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
        cudaStream_t st = static_cast<cudaStream_t>(stream);
        unsigned char* base = reinterpret_cast<unsigned char*>(h->dev->gemm_scratch);
        signed char* xq = reinterpret_cast<signed char*>(base);
        float* sx = reinterpret_cast<float*>(base + sc.xq);
        int32_t* rs = reinterpret_cast<int32_t*>(base + sc.xq + sc.arr);
        if (launch_quantize(static_cast<const __half*>(x), xq, sx, rs, M, L.K, st, h->pdl) != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
        GemmPairLayers set{};
        set.n = 1; set.L[0] = &h->L; set.blob[0] = h->blob; set.y[0] = y; set.wmap[0] = h->wmap_wide_ok ? &h->wmap_wide : nullptr;
        if (gemm_pair_ta_i8_applicable(set, M)) {
            float* scratch = sc.parts ? reinterpret_cast<float*>(base + sc.xq + 2 * sc.arr) : nullptr;
            return gemm_pair_ta_forward_i8(set, xq, sx, rs, M, st, h->device, h->early(), h->num_sms, scratch, h->dev->gemm_counters);
        }
        return gemm_pair_forward_i8(set, xq, sx, rs, M, st, h->device, h->num_sms);
    }
    const GemvPlan pl = plan_gemv(L, h->n_rb, M, h->num_sms, false, true);
    if (pl.grid <= 0) return QL_ERR_UNSUPPORTED;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    GemvA8Params prm{};
    prm.body = h->blob + L.body_offset;
    prm.chan_scales = L.grouped ? nullptr : reinterpret_cast<const __half*>(h->blob + L.chan_scale_offset);
    prm.x = static_cast<const __half*>(x);
    prm.y = static_cast<__half*>(y);
    prm.M = M; prm.N = L.N; prm.K = L.K;
    prm.n_rb = h->n_rb; prm.n_kc = L.n_kc; prm.block_bytes = L.block_bytes;
    prm.ks_cta = pl.ks_cta; prm.ks_cta_log2 = pl.ks_cta == 8 ? 3 : pl.ks_cta == 4 ? 2 : pl.ks_cta == 2 ? 1 : 0; prm.cl = pl.cl; prm.cps = pl.cps;
    const int span = pl.ks_cta * pl.cps * L.chunk_k;
    prm.xq_stride = span + 32;
    prm.xq_bytes = ((M * prm.xq_stride + 15) / 16) * 16;
    prm.sg_bytes = span;                                                 // 32 bytes per 32-k group
    cudaError_t e;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (L.bits == 8) e = launch_a8<8, false>(h, prm, pl, st);
    else if (L.grouped) e = launch_a8<4, true>(h, prm, pl, st);
    else e = launch_a8<4, false>(h, prm, pl, st);
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_quantize_activations(const void* x, int8_t* xq, float* scale, int32_t M, int32_t K, int device, void* stream)
{
    if (!x || !xq || !scale || M < 1 || K < 32 || (K % 32)) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(xq)) & 15) return QL_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(scale) & 3) return QL_ERR_INVALID_ARG;
    if (device < 0 || device >= kMaxDevices) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    quantize_activations_kernel<<<M, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const __half*>(x),
                                                                                reinterpret_cast<signed char*>(xq), scale, nullptr, M, K);
    return cudaGetLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_kv_append_heads(const qlinear_t* hk, const qlinear_t* hv, int32_t n_heads, const void* k_new, const void* v_new,
                                             int64_t head_stride, int64_t token_stride, void* const* v_scales, int32_t pos, int32_t n_new,
                                             void* stream)
{
    if (!hk || !hv || !v_scales || n_heads < 1 || n_heads > kKvMaxHeads || !k_new || !v_new || pos < 0 || n_new < 0) return QL_ERR_INVALID_ARG;
    if (head_stride < 0 || token_stride < 0 || ((head_stride | token_stride) & 7)) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(k_new) | reinterpret_cast<uintptr_t>(v_new)) & 15) return QL_ERR_INVALID_ARG;
    for (int i = 0; i < n_heads; ++i) {
        if (!hk[i] || !hv[i] || !v_scales[i] || (reinterpret_cast<uintptr_t>(v_scales[i]) & 15)) return QL_ERR_INVALID_ARG;
        const Layout &K = hk[i]->L, &V = hv[i]->L;
        if (hk[i]->device != hk[0]->device || hv[i]->device != hk[0]->device) return QL_ERR_INVALID_ARG;
        if (K.bits != 8 || V.bits != 8 || K.N != V.K || K.K != V.N || K.N != hk[0]->L.N || K.K != hk[0]->L.K) return QL_ERR_INVALID_ARG;
    }
    const Layout &K = hk[0]->L, &V = hv[0]->L;
    if ((int64_t)pos + n_new > K.N || K.K > 1024) return QL_ERR_INVALID_ARG;
    if (n_new == 0) return QL_OK;
    DeviceGuard guard(hk[0]->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    KvAppendParams prm{};
    for (int i = 0; i < n_heads; ++i) {
        uint8_t* kb = const_cast<uint8_t*>(hk[i]->blob);                 // the caches are the one kind of blob the library writes
        uint8_t* vb = const_cast<uint8_t*>(hv[i]->blob);
        prm.k_body[i] = kb + K.body_offset;
        prm.k_scales[i] = reinterpret_cast<__half*>(kb + K.chan_scale_offset);
        prm.v_body[i] = vb + V.body_offset;
        prm.v_scale[i] = static_cast<__half*>(v_scales[i]);
    }
    prm.k_new = static_cast<const __half*>(k_new);
    prm.v_new = static_cast<const __half*>(v_new);
    prm.head_stride = head_stride; prm.token_stride = token_stride;
    prm.d_h = K.K; prm.cache_size = K.N; prm.pos = pos; prm.n_new = n_new;
    prm.k_n_kc = K.n_kc; prm.v_n_kc = V.n_kc;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned long long capture;
    const bool known = capture_of(st, &capture);
    std::lock_guard<std::mutex> lock(g_append_mutex[hk[0]->device]);
    // Two dimensions per lane where the chain of latencies is the bound, four where the stores of many wide vectors are (half the warps then
    // read each vector).  Measured, us 2 / 4 per lane: one token of 8 heads of 128 1.62 / 1.78, of 1024 2.32 / 2.38; 512 vectors of 256 2.50 / 2.66,
    // 2048 4.62 / 4.38; 512 of 512 3.36 / 3.32, 2048 7.84 / 6.73; 128 of 1024 2.73 / 2.65, 2048 17.5 / 11.4.  The value bytes spread from 32768 values on:
    // in a row / spread, one token of a head of 32 1.38 / 1.85, of 128 1.36 / 1.46; 128 vectors of 128 1.79 / 1.78, 512 2.47 / 2.13, 2048 3.84 / 3.40.
    const int64_t values = (int64_t)n_new * n_heads * K.K;
    const bool wide = K.K > 128 && values * K.K >= (int64_t)1 << 27;
    const auto kern = wide ? kv_append_kernel<4, true> : values >= 32768 ? kv_append_kernel<2, true> : kv_append_kernel<2, false>;
    const int per_warp = wide ? 128 : 64;
    if (launch(kern, prm, dim3(n_new, n_heads), dim3(64 * ((K.K + per_warp - 1) / per_warp)), 0, st, 1, hk[0]->pdl) != cudaSuccess) {
        cudaGetLastError();                                              // nothing is in flight: the append before it stays the last one
        return QL_ERR_CUDA;
    }
    for (int i = 0; i < n_heads; ++i)
        for (qlinear_s* h : {hk[i], hv[i]}) {
            const bool joined = capture && h->append.capture == capture && (h->append.stream != st || !h->append.alone);
            h->append = {pos, pos + n_new, st, capture, known && !joined};
            h->cache.store(true, std::memory_order_relaxed);
        }
    return QL_OK;
}

extern "C" ql_status qlinear_kv_append(qlinear_t hk, qlinear_t hv, const void* k_new, const void* v_new, void* v_scale,
                                       int32_t pos, int32_t n_new, void* stream)
{
    if (!hk || !hv) return QL_ERR_INVALID_ARG;
    return qlinear_kv_append_heads(&hk, &hv, 1, k_new, v_new, 0, hk->L.K, &v_scale, pos, n_new, stream);
}

extern "C" ql_status qlinear_kv_scores(qlinear_t hk, const void* q_rows, void* scores, int32_t R, void* stream)
{
    if (!hk || hk->L.bits != 8) return QL_ERR_INVALID_ARG;
    return qlinear_forward(hk, q_rows, scores, R, stream);
}

extern "C" ql_status qlinear_kv_scores_heads(const qlinear_t* hk, int32_t n_heads, const void* q_rows, void* scores, int32_t R, void* stream)
{
    if (!hk || n_heads < 1 || n_heads > kKvMaxHeads || !q_rows || !scores || R < 1) return QL_ERR_INVALID_ARG;
    for (int i = 0; i < n_heads; ++i)
        if (!hk[i] || hk[i]->L.bits != 8 || hk[i]->L.N != hk[0]->L.N || hk[i]->L.K != hk[0]->L.K) return QL_ERR_INVALID_ARG;
    const int64_t xs_stride = (int64_t)R * hk[0]->L.K, ys_stride = (int64_t)R * hk[0]->L.N;
    if ((xs_stride | ys_stride) & 7) return QL_ERR_INVALID_ARG;          // every head's rows start on a 16-byte boundary
    for (int h0 = 0; h0 < n_heads; h0 += kGemvMaxBatch) {
        const int n = std::min(kGemvMaxBatch, n_heads - h0);
        const void* xs[kGemvMaxBatch];
        void* ys[kGemvMaxBatch];
        for (int i = 0; i < n; ++i) {
            xs[i] = static_cast<const __half*>(q_rows) + (h0 + i) * xs_stride;
            ys[i] = static_cast<__half*>(scores) + (h0 + i) * ys_stride;
        }
        const ql_status s = qlinear_forward_batch(hk + h0, n, xs, ys, R, stream);
        if (s != QL_OK) return s;
    }
    return QL_OK;
}

extern "C" ql_status qlinear_kv_output_heads(const qlinear_t* hv, int32_t n_heads, const void* prob, const void* const* v_scales, void* out,
                                             int32_t R, void* stream)
{
    if (!hv || !v_scales || n_heads < 1 || n_heads > kKvMaxHeads || !prob || !out || R < 1) return QL_ERR_INVALID_ARG;
    for (int i = 0; i < n_heads; ++i) {
        if (!hv[i] || !v_scales[i] || (reinterpret_cast<uintptr_t>(v_scales[i]) & 15)) return QL_ERR_INVALID_ARG;
        if (hv[i]->L.bits != 8 || hv[i]->L.N != hv[0]->L.N || hv[i]->L.K != hv[0]->L.K || hv[i]->device != hv[0]->device) return QL_ERR_INVALID_ARG;
    }
    const Layout& V = hv[0]->L;
    const int64_t xs_stride = (int64_t)R * V.K, ys_stride = (int64_t)R * V.N;
    if ((xs_stride | ys_stride) & 7) return QL_ERR_INVALID_ARG;
    if (((reinterpret_cast<uintptr_t>(prob) | reinterpret_cast<uintptr_t>(out)) & 15) || xs_stride > INT32_MAX) return QL_ERR_INVALID_ARG;
    if (R > hv[0]->gemv_max_m || hv[0]->use_stream) return QL_ERR_UNSUPPORTED;          // the fused form exists in the decode kernel
    if (device_timed_out(hv[0])) return QL_ERR_DEVICE_TIMEOUT;
    DeviceGuard guard(hv[0]->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    for (int h0 = 0; h0 < n_heads; h0 += kGemvMaxBatch) {
        const int n = std::min(kGemvMaxBatch, n_heads - h0);
        const void* xs[kGemvMaxBatch];
        void* ys[kGemvMaxBatch];
        for (int i = 0; i < n; ++i) {
            xs[i] = static_cast<const __half*>(prob) + (h0 + i) * xs_stride;
            ys[i] = static_cast<__half*>(out) + (h0 + i) * ys_stride;
        }
        const ql_status s = forward_gemv_cols(const_cast<qlinear_s* const*>(hv + h0), n, xs, v_scales + h0, ys, R, static_cast<cudaStream_t>(stream));
        if (s != QL_OK) return s;
    }
    return QL_OK;
}

namespace {
// Value products of many rows for which the scales as a pass of their own and the prefill kernel win: heads of more than 256 (whose
// layers the CTA-pair kernel takes), from a size on at which the batch kernel's warp-level MMAs cost more than that pass.  Measured,
// us batch kernel / pass and prefill kernel: 512 channels, 4096 positions, 1024 rows 23 / 32, 2048 rows 41 / 41, 4096 rows 76 / 61; 1024
// channels, 4096 positions, 512 rows 23 / 29, 1024 rows 41 / 34, 4096 rows 148 / 61; 1024 positions, 2048 rows 22 / 25, 4096 rows 42 / 23;
// 256 positions, 2048 rows 9 / 12, 4096 rows 16 / 13.  256 channels, 4096 positions, 4096 rows 41 / 58.
bool value_product_is_large(const Layout& V, int R)
{
    return V.n_rsb % 2 == 0 && V.N > 256 && (int64_t)R * (V.N - 256) * (V.K + 1024) > 3350000000ll;
}
}  // namespace

extern "C" int32_t qlinear_kv_output_uses_tmp(qlinear_t hv, const void* prob, const void* v_scale, int32_t R)
{
    if (!hv || ((reinterpret_cast<uintptr_t>(prob) | reinterpret_cast<uintptr_t>(v_scale)) & 15)) return 1;
    return R <= hv->gemv_max_m ? hv->use_stream : value_product_is_large(hv->L, R);
}

extern "C" ql_status qlinear_kv_output(qlinear_t hv, const void* prob, const void* v_scale, void* tmp, void* out, int32_t R, void* stream)
{
    if (!hv || !prob || !v_scale || !tmp || !out || R < 1 || hv->L.bits != 8) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(tmp) | reinterpret_cast<uintptr_t>(out)) & 15) return QL_ERR_INVALID_ARG;
    const int T = hv->L.K;
    if ((int64_t)R * T > INT32_MAX) return QL_ERR_INVALID_ARG;
    // decode-sized products whose cache length is a whole number of chunks: the scales are applied inside the kernel
    if (!qlinear_kv_output_uses_tmp(hv, prob, v_scale, R)) {
        if (R <= hv->gemv_max_m) return qlinear_kv_output_heads(&hv, 1, prob, &v_scale, out, R, stream);
        // more rows: the kernel that takes any number of tokens against few channels, with the scales folded in on the way
        if ((int64_t)R * hv->L.N > INT32_MAX) return QL_ERR_INVALID_ARG;   // (the limit of qlinear_forward)
        if (device_timed_out(hv)) return QL_ERR_DEVICE_TIMEOUT;
        DeviceGuard guard(hv->device);
        if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
        const qlinear_s* h = hv;
        return forward_mid(&h, 1, &prob, &out, R, static_cast<cudaStream_t>(stream), -1, &v_scale);
    }
    {
        DeviceGuard guard(hv->device);
        if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
        const int64_t n = (int64_t)R * T;
        const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)hv->num_sms * 8);
        kv_scale_probs_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const __half*>(prob),
                                                                                     static_cast<const __half*>(v_scale), static_cast<__half*>(tmp), n, T);
        if (cudaGetLastError() != cudaSuccess) return QL_ERR_CUDA;
    }
    return qlinear_forward(hv, tmp, out, R, stream);
}

extern "C" ql_status qlinear_embed(qlinear_t h, const int32_t* ids, int32_t n, void* y, void* stream)
{
    if (!h || n < 0) return QL_ERR_INVALID_ARG;
    if (n == 0) return QL_OK;                                            // nothing to do: the pointers may be null
    if (!ids || !y) return QL_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(y) & 15) || (reinterpret_cast<uintptr_t>(ids) & 3)) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    const Layout& L = h->L;
    EmbedParams prm{};
    prm.body = h->blob + L.body_offset;
    prm.chan_scales = L.grouped ? nullptr : reinterpret_cast<const __half*>(h->blob + L.chan_scale_offset);
    prm.ids = ids;
    prm.y = static_cast<__half*>(y);
    prm.n = n; prm.N = L.N; prm.K = L.K; prm.n_kc = L.n_kc; prm.block_bytes = L.block_bytes;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // short rows: several tokens to a CTA where that leaves several CTAs per SM (a CTA costs more than what four threads of it do)
    while (L.n_kc * 4 <= 64 >> prm.log2_tokens && n >> (prm.log2_tokens + 1) >= 4 * h->num_sms) ++prm.log2_tokens;
    auto kern = L.bits == 8 ? embed_kernel<8, false, false> : L.grouped ? embed_kernel<4, true, false> : embed_kernel<4, false, false>;
    if (L.n_kc * 4 > 128) kern = L.bits == 8 ? embed_kernel<8, false, false, 2> : L.grouped ? embed_kernel<4, true, false, 2> : embed_kernel<4, false, false, 2>;
    if (prm.log2_tokens) kern = L.bits == 8 ? embed_kernel<8, false, true> : L.grouped ? embed_kernel<4, true, true> : embed_kernel<4, false, true>;
    const cudaError_t e = launch(kern, prm, dim3(((n - 1) >> prm.log2_tokens) + 1), dim3(128), 0, st, 1, h->pdl);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_residual_rmsnorm(const void* x, const void* residual, const void* gamma, float eps, float gamma_offset,
                                              void* h_out, void* y_out, int32_t M, int32_t K, int32_t device, void* stream)
{
    if (!x || !gamma || !y_out || M < 0 || K < 8 || (K % 8) || device < 0) return QL_ERR_INVALID_ARG;
    if (!(eps >= 0.f) || y_out == h_out) return QL_ERR_INVALID_ARG;
    const uintptr_t all = reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(residual) | reinterpret_cast<uintptr_t>(gamma) |
                          reinterpret_cast<uintptr_t>(h_out) | reinterpret_cast<uintptr_t>(y_out);
    if (all & 15) return QL_ERR_INVALID_ARG;
    if (M == 0) return QL_OK;
    int n_dev = 0;
    if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device >= n_dev) { cudaGetLastError(); return QL_ERR_INVALID_ARG; }
    DeviceGuard guard(device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    NormParams prm{};
    prm.x = static_cast<const __half*>(x);
    prm.r = static_cast<const __half*>(residual);
    prm.g = static_cast<const __half*>(gamma);
    prm.h_out = static_cast<__half*>(h_out);
    prm.y_out = static_cast<__half*>(y_out);
    prm.eps = eps; prm.offset = gamma_offset; prm.M = M; prm.K = K;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int vpt = (K / 8 + kNormThreads - 1) / kNormThreads;           // 8-value vectors per thread
    const bool pdl = config().pdl;
    cudaError_t e;
    if (vpt <= 1) e = launch(residual_rmsnorm_kernel<1>, prm, dim3(M), dim3(kNormThreads), 0, st, 1, pdl);
    else if (vpt <= 2) e = launch(residual_rmsnorm_kernel<2>, prm, dim3(M), dim3(kNormThreads), 0, st, 1, pdl);
    else if (vpt <= 4) e = launch(residual_rmsnorm_kernel<4>, prm, dim3(M), dim3(kNormThreads), 0, st, 1, pdl);
    else if (vpt <= 8) e = launch(residual_rmsnorm_kernel<8>, prm, dim3(M), dim3(kNormThreads), 0, st, 1, pdl);
    else e = launch(residual_rmsnorm_kernel<0>, prm, dim3(M), dim3(kNormThreads), 0, st, 1, pdl);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_rope_qkv(const void* q, const void* k, const void* v, const int32_t* pos, const float* cos_t, const float* sin_t,
                                      int32_t n_pos, void* q_out, void* k_out, void* v_out, int32_t B, int32_t S, int32_t h_q, int32_t h_kv,
                                      int32_t d_h, int32_t device, void* stream)
{
    if (!q || !k || !v || !pos || !cos_t || !sin_t || !q_out || !k_out || !v_out) return QL_ERR_INVALID_ARG;
    if (B < 0 || S < 0 || h_q < 1 || h_kv < 1 || (h_q % h_kv) || d_h < 16 || (d_h % 16) || n_pos < 1 || device < 0) return QL_ERR_INVALID_ARG;
    if ((int64_t)B * S > INT32_MAX || (int64_t)B * S * h_q * d_h > ((int64_t)1 << 40)) return QL_ERR_INVALID_ARG;
    const uintptr_t all = reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(cos_t) |
                          reinterpret_cast<uintptr_t>(sin_t) | reinterpret_cast<uintptr_t>(q_out) | reinterpret_cast<uintptr_t>(k_out) | reinterpret_cast<uintptr_t>(v_out);
    if ((all & 15) || (reinterpret_cast<uintptr_t>(pos) & 3)) return QL_ERR_INVALID_ARG;
    if (q_out == q || k_out == k || v_out == v) return QL_ERR_INVALID_ARG;   // the layout changes: not in place
    if ((int64_t)B * S == 0) return QL_OK;
    int n_dev = 0;
    if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device >= n_dev) { cudaGetLastError(); return QL_ERR_INVALID_ARG; }
    DeviceGuard guard(device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    RopeParams prm{};
    prm.q = static_cast<const __half*>(q); prm.k = static_cast<const __half*>(k); prm.v = static_cast<const __half*>(v);
    prm.pos = pos; prm.cos_t = cos_t; prm.sin_t = sin_t;
    prm.q_out = static_cast<__half*>(q_out); prm.k_out = static_cast<__half*>(k_out); prm.v_out = static_cast<__half*>(v_out);
    prm.B = B; prm.S = S; prm.h_q = h_q; prm.h_kv = h_kv; prm.d_h = d_h; prm.n_pos = n_pos;
    // threads: the work items of a token (8-element vectors of half a head) spread evenly over the fewest passes, which are CTAs
    // of their own where the tokens leave SMs idle
    const int items = (h_q + h_kv) * (d_h / 16) + h_kv * (d_h / 8);
    const int passes = (items + kRopeThreads - 1) / kRopeThreads;
    const int threads = std::min(kRopeThreads, (((items + passes - 1) / passes) + 31) / 32 * 32);
    const cudaError_t e = launch(rope_qkv_kernel, prm, dim3(B * S, B * S <= 64 ? passes : 1), dim3(threads), 0, static_cast<cudaStream_t>(stream), 1, config().pdl);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_debug_unpack_device(qlinear_t h, int8_t* q_out, void* stream)
{
    if (!h || !q_out) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    const Layout& L = h->L;
    dim3 grid(L.n_kc, L.n_rsb);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (L.bits == 4)
        debug_unpack_kernel<4><<<grid, 256, 0, st>>>(h->blob + L.body_offset, q_out, L.N, L.K, L.n_kc, L.block_bytes);
    else
        debug_unpack_kernel<8><<<grid, 256, 0, st>>>(h->blob + L.body_offset, q_out, L.N, L.K, L.n_kc, L.block_bytes);
    return cudaGetLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}


// ---------------------------------------------------------------------------------------------------
// qlinear_decode_static: the streaming decode kernel for callers that cannot allocate device memory
// (see include/qlinear.h).  Its partial-sum slots and counters live in one file-scope device array.
namespace {

constexpr int kStaticMaxCtas = 320;                 // CTAs of the persistent grid (2 per SM on a 148-SM part)
constexpr int kStaticMaxRsb = 4096;                 // row super-blocks, i.e. N <= 524288
constexpr size_t kStaticPartialBytes = (size_t)kStaticMaxCtas * 2 * kStreamPartialFloats * sizeof(float);   // 2.5 MiB
constexpr size_t kStaticCounterBytes = (size_t)kStaticMaxRsb * 8 * sizeof(unsigned int);                    // 128 KiB
constexpr int kStaticStages = 8;

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticPartialBytes + kStaticCounterBytes];

struct StaticDevice {
    bool ready = false;
    unsigned char* base = nullptr;                  // device address of g_static_scratch on this device
    int sms = 0;
};
StaticDevice g_static_dev[64];
std::mutex g_static_mutex;

// Once per device, with that device current: the array's name is only a host-side stand-in, the address a
// kernel may use comes from cudaGetSymbolAddress.
ql_status static_setup(int device, StaticDevice** out)
{
    if (device < 0 || device >= 64) return QL_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticDevice& d = g_static_dev[device];
    if (!d.ready) {
        int major = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
            cudaGetLastError();
            return QL_ERR_CUDA;
        }
        if (major != 10) return QL_ERR_ARCH;
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return QL_ERR_CUDA;
        }
        d.base = static_cast<unsigned char*>(ptr);
        d.ready = true;
    }
    *out = &d;
    return QL_OK;
}

template <int BITS, bool GROUPED>
cudaError_t launch_stream_static(const StreamParams& prm, cudaStream_t st, int device)
{
    static std::atomic<bool> attr_set[kMaxDevices];
    auto kern = gemv_stream_kernel<BITS, GROUPED, kStaticStages>;
    const size_t smem = (size_t)kStaticStages * StreamStage<BITS>::kBytes;
    cudaError_t e = ensure_smem_attr(kern, attr_set, device, (int)smem);
    if (e != cudaSuccess) return e;
    return launch(kern, prm, dim3(prm.P), dim3(kStreamThreads), smem, st, 1, false);
}

}  // namespace

extern "C" ql_status qlinear_decode_static(const qlinear_desc* d, const void* packed_dev, const void* x, void* y, int32_t M,
                                           int device, void* stream)
{
    if (!d || !packed_dev || !x || !y) return QL_ERR_INVALID_ARG;
    if (M < 1 || M > 8) return QL_ERR_INVALID_ARG;                       // decode kernel only
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) return QL_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(packed_dev) % 256) return QL_ERR_INVALID_ARG;
    Layout L;
    if (!make_layout(d->N, d->K, d->bits, d->group, &L)) return QL_ERR_UNSUPPORTED;
    if (L.n_rsb > kStaticMaxRsb) return QL_ERR_UNSUPPORTED;              // beyond the static counters
    if (L.bits == 4 && (L.K % 64)) return QL_ERR_UNSUPPORTED;            // the streaming kernel reads whole 64-k slices
    if (device < 0 || device >= kMaxDevices) return QL_ERR_INVALID_ARG;
    {
        int n_dev = 0;
        if (cudaGetDeviceCount(&n_dev) != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
        if (device >= n_dev) return QL_ERR_INVALID_ARG;
    }
    DeviceGuard guard(device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    StaticDevice* dev = nullptr;
    ql_status sst = static_setup(device, &dev);
    if (sst != QL_OK) return sst;

    const uint8_t* blob = static_cast<const uint8_t*>(packed_dev);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    StreamParams prm{};
    prm.body = blob + L.body_offset;
    prm.chan_scales = L.grouped ? nullptr : reinterpret_cast<const __half*>(blob + L.chan_scale_offset);
    prm.x = static_cast<const __half*>(x);
    prm.y = static_cast<__half*>(y);
    prm.scratch = reinterpret_cast<float*>(dev->base);
    prm.counters = reinterpret_cast<unsigned int*>(dev->base + kStaticPartialBytes);
    prm.M = M; prm.N = L.N; prm.K = L.K;
    prm.n_rsb = L.n_rsb; prm.n_kc = L.n_kc; prm.block_bytes = L.block_bytes;
    const int64_t B = (int64_t)L.n_rsb * L.n_kc;
    prm.P = (int)std::min<int64_t>(B, std::min(kStaticMaxCtas, 2 * dev->sms));
    prm.stages = kStaticStages;
    // The array keeps whatever the last call left: the counters must start at zero (they do after a call
    // that ran to completion; this also covers one that did not).
    if (cudaMemsetAsync(prm.counters, 0, (size_t)L.n_rsb * 8 * sizeof(unsigned int), st) != cudaSuccess) {
        cudaGetLastError();
        return QL_ERR_CUDA;
    }
    cudaError_t e;
    if (L.bits == 8) e = launch_stream_static<8, false>(prm, st, device);
    else if (L.grouped) e = launch_stream_static<4, true>(prm, st, device);
    else e = launch_stream_static<4, false>(prm, st, device);
    if (e != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
    return QL_OK;
}

// A kernel that does nothing but take part in programmatic dependent launch: what a launch costs on this machine.
__global__ void null_kernel(unsigned int* sink)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (sink && threadIdx.x == 0 && blockIdx.x == 0x7fffffff) *sink = 1;   // (never true: keeps the kernel from being empty code)
}

extern "C" ql_status qlinear_debug_null_launch(qlinear_t h, int32_t grid, int32_t block, void* stream)
{
    if (!h || grid < 1 || block < 1 || block > 1024) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    const cudaError_t e = launch(null_kernel, static_cast<unsigned int*>(nullptr), dim3(grid), dim3(block), 0, static_cast<cudaStream_t>(stream), 1, h->pdl);
    return e == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_debug_expire_wait(qlinear_t h, void* stream)
{
    if (!h) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    expire_wait_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>();
    return cudaGetLastError() == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

extern "C" ql_status qlinear_device_status(qlinear_t h, uint32_t* detail)
{
    if (!h) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(h->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    unsigned int flag[2] = {0, 0};
    if (cudaDeviceSynchronize() != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
    if (cudaMemcpyFromSymbol(flag, g_device_flag, sizeof(flag)) != cudaSuccess) { cudaGetLastError(); return QL_ERR_CUDA; }
    if (detail) *detail = flag[0];
    if (flag[0] == 0) return QL_OK;
    // Clear the condition, and with it whatever an abandoned launch left in the shared arrival counters.
    const unsigned int zero[2] = {0, 0};
    cudaMemcpyToSymbol(g_device_flag, zero, sizeof(zero));
    h->dev->status_host[0] = 0;
    cudaMemset(h->dev->gemm_counters, 0, gemm_pair_counter_count(h->dev->sms) * sizeof(unsigned int));
    if (h->dev->stream_counters) cudaMemset(h->dev->stream_counters, 0, (size_t)kStreamMaxRsb * 8 * sizeof(unsigned int));
    cudaDeviceSynchronize();
    return QL_ERR_DEVICE_TIMEOUT;
}

extern "C" ql_status qlinear_destroy(qlinear_t h)
{
    if (!h) return QL_OK;
    {
        std::lock_guard<std::mutex> lock(g_dev_mutex);
        --h->dev->handles;                   // the device's shared state stays for the next handle (a few tens of MB)
    }
    delete h;
    return QL_OK;
}

extern "C" int32_t qlinear_debug_plan(qlinear_t h, int32_t M, int32_t* out, int32_t n_out)
{
    if (!h || M < 1 || M > 8 || !out) return 0;
    const int32_t v[8] = {h->use_stream ? 3 : 1, h->gemv[M].grid, h->gemv[M].cl, h->gemv[M].ks_cta, h->gemv[M].cps,
                          (int32_t)(1000 * h->gemv[M].max_over_mean), h->n_rb, h->L.n_kc};
    int n = n_out < 8 ? n_out : 8;
    for (int i = 0; i < n; ++i) out[i] = v[i];
    return n;
}

extern "C" int32_t qlinear_debug_plan_kv_output(qlinear_t h, int32_t n_heads, int32_t* out, int32_t n_out)
{
    if (!h || h->L.bits != 8 || n_heads < 1 || n_heads > kKvMaxHeads || !out) return 0;
    DeviceGuard guard(h->device);
    if (!guard.ok || cudaFuncSetAttribute(gemv_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kColsSmem) != cudaSuccess) { cudaGetLastError(); return 0; }
    const int heads = std::min(n_heads, (int32_t)kGemvMaxBatch), cl = cols_split(h->device, heads * h->n_rb, h->L.n_kc);
    const int32_t v[4] = {cl, (h->L.n_kc + kColsWarps * cl - 1) / (kColsWarps * cl), heads * h->n_rb, cl > 1 ? cols_clusters_at_once(h->device, cl) : h->num_sms};
    const int n = n_out < 4 ? n_out : 4;
    for (int i = 0; i < n; ++i) out[i] = v[i];
    return n;
}

extern "C" int32_t qlinear_debug_route(const qlinear_desc* ds, int32_t n, int32_t M, int32_t gated, int32_t num_sms, int32_t* out, int32_t n_out)
{
    if (!ds || n < 1 || n > kGemvMaxGroup || M < 1 || num_sms < 2 || !out || (gated && n != 2)) return 0;
    qlinear_s layers[kGemvMaxGroup];                                     // (host state only; nothing reads their device pointers)
    const qlinear_s* hs[kGemvMaxGroup];
    int rows = 0;
    for (int i = 0; i < n; ++i) {
        qlinear_s& h = layers[i];
        if (!make_layout(ds[i].N, ds[i].K, ds[i].bits, ds[i].group, &h.L)) return 0;
        if (h.L.K != layers[0].L.K || h.L.bits != layers[0].L.bits || h.L.group != layers[0].L.group || (gated && h.L.N != layers[0].L.N)) return 0;
        h.num_sms = num_sms;
        h.wmap_ok = w_map_fits(h.L, false);
        h.wmap_wide_ok = w_map_fits(h.L, true);
        hs[i] = &h;
        rows += h.L.n_rsb;
    }
    if (M <= config().gemv_max_m) { out[0] = QL_KERNEL_DECODE; return 1; }
    const Layout& L = layers[0].L;
    const NarrowPlan pl = plan_narrow(L, gated ? L.n_rsb : rows, gated, M, num_sms);
    const ql_kernel kernel = gemm_route(hs, n, M, gated);
    int32_t width = 0, parts = 1;
    if (kernel == QL_KERNEL_NARROW) { width = pl.bn; parts = pl.cl; }
    if (kernel == QL_KERNEL_SINGLE) width = gemm_pick_bn(L, M, num_sms);
    if (kernel == QL_KERNEL_PAIR_TA) {
        const TaPlan pl = gated ? gemm_pair_ta_gated_plan(L, M, num_sms) : gemm_pair_ta_plan(rows / 2, M, (L.K + kGemmKStep - 1) / kGemmKStep, 1, false, num_sms, true);
        width = pl.bn;
        parts = pl.split;
    }
    const double other = takes_mid(hs, n, M, gated) ? mid_us(hs, n, M, gated) : prefill_us(prefill_kernel(hs, n, M, gated), hs, n, M, gated);
    const int32_t v[5] = {kernel, width, parts, (int32_t)(1000 * narrow_us(hs, n, M, gated)), (int32_t)(1000 * other)};
    const int k = n_out < 5 ? n_out : 5;
    for (int i = 0; i < k; ++i) out[i] = v[i];
    return k;
}

extern "C" int32_t qlinear_debug_plan_a8(const qlinear_desc* d, int32_t M, int32_t num_sms, int32_t* out, int32_t n_out)
{
    Layout L;
    if (!d || M < 1 || num_sms < 2 || !out || !make_layout(d->N, d->K, d->bits, d->group, &L)) return 0;
    int32_t v[4];
    if (M <= config().gemv_max_m) {
        const GemvPlan pl = plan_gemv(L, (L.N + kRbRows - 1) / kRbRows, M, num_sms, false, true);
        if (pl.grid <= 0) return 0;
        v[0] = QL_KERNEL_DECODE; v[1] = pl.grid; v[2] = pl.cl; v[3] = pl.ks_cta;
    } else {
        const A8Scratch sc = a8_scratch(M, L.K, num_sms);
        if (L.grouped || (L.K % 128) || !gemm_pair_applicable(L, M) || !sc.fits) return 0;
        const bool ta = gemm_config().ta && w_map_fits(L, true);
        const TaPlan pl = ta ? gemm_pair_ta_i8_plan(L, M, num_sms, sc.parts) : TaPlan{(M + 255) / 256, 256, 1};
        v[0] = ta ? QL_KERNEL_PAIR_TA : QL_KERNEL_PAIR; v[1] = pl.bn; v[2] = pl.split; v[3] = pl.n_mblk;
    }
    const int k = std::min(n_out, 4);
    for (int i = 0; i < k; ++i) out[i] = v[i];
    return k;
}

extern "C" ql_status qlinear_debug_kv_hold(const qlinear_t* hs, int32_t n, void* stream, int32_t* first, int32_t* end)
{
    if (!hs || !first || !end || n < 1 || n > kGemvMaxBatch) return QL_ERR_INVALID_ARG;
    for (int i = 0; i < n; ++i)
        if (!hs[i] || hs[i]->device != hs[0]->device) return QL_ERR_INVALID_ARG;
    DeviceGuard guard(hs[0]->device);
    if (!guard.ok) { cudaGetLastError(); return QL_ERR_CUDA; }
    held_tokens(hs, n, static_cast<cudaStream_t>(stream), first, end);
    return QL_OK;
}

extern "C" int32_t qlinear_debug_takes_batch_kernel(const qlinear_t* hs, int32_t n, int32_t M)
{
    if (!hs || n < 1 || n > kGemvMaxGroup || M < 1) return 0;
    for (int i = 0; i < n; ++i)
        if (!hs[i]) return 0;
    return M > hs[0]->gemv_max_m && !(n == 1 && takes_rows(hs[0]->L)) && takes_mid(hs, n, M);
}

extern "C" uint32_t qlinear_debug_config_reads(void) { config(); return g_getenv_reads.load(); }

extern "C" const char* qlinear_status_string(ql_status s)
{
    switch (s) {
        case QL_OK: return "ok";
        case QL_ERR_INVALID_ARG: return "invalid argument";
        case QL_ERR_UNSUPPORTED: return "unsupported shape or quantisation scheme";
        case QL_ERR_ALLOC: return "host allocation failed";
        case QL_ERR_CUDA: return "CUDA call failed";
        case QL_ERR_DEVICE_TIMEOUT: return "a bounded wait inside a kernel expired";
        case QL_ERR_ARCH: return "device is not compute capability 10.x (sm_100)";
    }
    return "unknown status";
}


extern "C" uint32_t qlinear_version(void) { return (1u << 16) | 0u; }
