// SVIP speculative-decoding epilogues for sm_100a: the host side and the C ABI (see include/svip.h).
//
// The kernels live in the headers included below:
//   svip_device.cuh    the streaming core: row geometry, cp.async ring, online reduction, warp / block
//                      scans, picking the segment that holds a sample
//   svip_draft.cuh     draft_step_kernel (Algorithm 1 inner loop + Eq. 7) and row_stats_kernel (softmax
//                      normalisers or argmax of target rows; of draft rows when the caller has no q_stats)
//   svip_verify.cuh    verify_finish_kernel (Algorithms 2 and 4 + the loop of Algorithm 1: ratio tests by
//                      one warp, first rejection, residual or bonus token) and verify_greedy_kernel
//                      (Algorithms 3 and 5)
//   svip_analysis.cuh  pair_stats_kernel (Eq. 1-6)
//   svip_policy.cuh    vocabulary-parallel combine, draft-length policies, ragged packing
//   svip_select.cuh    row_threshold_kernel (top-k / nucleus truncation)
//   svip_tree.cuh      verify_tree_kernel (several candidates per position: recursive rejection sampling)
#include "svip_device.cuh"

#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <new>

#include "svip.h"

#include "svip_draft.cuh"
#include "svip_verify.cuh"
#include "svip_analysis.cuh"
#include "svip_policy.cuh"

#include "svip_select.cuh"
#include "svip_tree.cuh"

// ==================================================================== host side / C ABI

// -DSVIP_NVTX: a named range around every entry point's host work, for timelines.
#ifdef SVIP_NVTX
#include <nvtx3/nvToolsExt.h>
namespace {
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
};
}  // namespace
#define SVIP_RANGE(name) NvtxRange svip_nvtx_range_(name)
#else
#define SVIP_RANGE(name) do { } while (0)
#endif

using namespace svip;

struct svip_ctx {
    int device;
    int max_rows;
    int num_sms;
    int cluster_override;
    int max_clusters[kMaxCluster + 1];   // clusters of each size that fit the GPU at once (two blocks per SM)
    long launches;
    int last_cuda;
    int capturing;
    float2* p_stats;
    float2* q_stats;
    int32_t* p_argmax;
    unsigned* status;
    unsigned long long* loop_arrived;   // device: sequences counted by the draft kernel of the drafting loop being replayed,
                                        // zero between launches; behind it ...
    int* loop_iter;                     // ... the iteration counter of that loop (both cleared when a replay enters it)
    cudaGraphNode_t loop_draft_node;    // the last draft step recorded in the loop body, if nothing came after it ...
    DraftArgs loop_draft_args;          // ... and its arguments
    int loop_draft_rows;
    cudaStream_t loop_stream;  // records the body of a drafting loop
    int loop_open;             // a loop body is being recorded
    int loop_decided;          // the body already holds the kernel that decides the loop
    int loop_failed;           // a loop of the graph being recorded is not closed properly
    LoopCtl loop;
    const int32_t* loop_n_active;
    int profiling;
    int prof_used;
    cudaEvent_t* prof_start;
    cudaEvent_t* prof_stop;
};

constexpr int kProfilePairs = 4096;
constexpr size_t kLoopStateBytes = 16;    // loop_arrived and loop_iter

struct svip_graph {
    cudaGraphExec_t exec;
    cudaGraph_t graph;
};

namespace {

// SVIP_NO_PDL=1 in the environment launches every kernel fully serialized (for A/B timing).
const bool g_use_pdl = [] {
    const char* v = std::getenv("SVIP_NO_PDL");
    return !(v && v[0] == '1');
}();

// Set while the calling thread records the body of a drafting loop: kernels inside a conditional
// node are launched without the programmatic-serialization attribute.
thread_local bool t_plain_launches = false;

int cuda_fail(svip_ctx* ctx, cudaError_t e) {
    if (ctx) ctx->last_cuda = static_cast<int>(e);
    return SVIP_ERR_CUDA;
}

// Every kernel goes through here: optional cluster dimension, dynamic shared memory, and the
// programmatic-serialization attribute that lets the kernel be scheduled while its predecessor in
// the stream drains (the kernels wait for the predecessor themselves, see pdl_wait()).
template <class... KArgs, class... Args>
cudaError_t launch_ex(void (*kernel)(KArgs...), unsigned grid, unsigned block, int S, size_t dyn_smem,
                      cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = dyn_smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (S > 0) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = S;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (g_use_pdl && !t_plain_launches) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <class Args>
cudaError_t launch_clustered(void (*kernel)(Args), long units, int S, const Args& args, cudaStream_t st,
                             size_t dyn_smem) {
    return launch_ex(kernel, static_cast<unsigned>(units * S), kThreads, S, dyn_smem, st, args);
}

// Blocks per row.  Small launches are latency-bound: spread a row over as many blocks (1..8, any
// size) as still lets the whole grid sit on the GPU at once (two blocks per SM) while every thread
// keeps a vector; a second wave of clusters would double the time of such a launch.
int pick_cluster(const svip_ctx* ctx, long rows, int V, int dtype) {
    if (ctx->cluster_override > 0) return ctx->cluster_override;
    long nvec = (static_cast<long>(V) * (dtype == SVIP_BF16 ? 2 : 4) + 15) / 16;
    // measured: grids up to about 7/4 blocks per SM run as one wave next to the blocks of the
    // following launch that programmatic launch makes resident early; fuller grids run as two
    long by_grid = rows > 0 ? (7L * ctx->num_sms / 4) / rows : kMaxCluster;
    long by_work = nvec / kThreads;
    long S = by_grid < by_work ? by_grid : by_work;
    if (S > kMaxCluster) S = kMaxCluster;
    if (S < 1) S = 1;
    // measured: clusters of 5 and 7 blocks are placed badly (48 rows of 304 KB: 11.4 us with 5 blocks per row,
    // 9.8 with 4); the next smaller even size is used instead
    if (S == 5 || S == 7) S -= 1;
    // many long rows (more than a wave of blocks anyway): rows above 512 KB are cut so that the
    // two blocks of an SM finish close together (measured on 256 x 1 MB: 64 -> 55 us)
    const long row_bytes = nvec * 16;
    if (S == 1 && rows > ctx->num_sms && row_bytes > (512L << 10)) {
        S = (row_bytes + (512L << 10) - 1) / (512L << 10);
        if (S > 4) S = 4;
    }
    return static_cast<int>(S);
}

// Blocks per row of a draft step (and of svip_vp_locate, the same kernel).  Where pick_cluster gives 6 or 8, rows of up to
// 128 KB (below 8 rows up to 64 KB) take 4, or 2 from about a fifth as many rows as SMs on (30 to 43 rows).  us with 2, 4, 6
// and 8 blocks, launches of equal size:
//                 16 rows                  24 rows                  32 rows                  38 rows
//      64 KB  3.63 3.35 4.03 4.05      3.70 3.63 4.14 4.11      3.78 4.21 4.28 4.49      3.89 4.28 4.38 5.48
//      96 KB  4.05 3.60 4.06 4.31      4.05 3.79 4.22 4.39      4.05 4.50 4.29 4.78      4.25 4.57 4.40 5.85
//     128 KB  4.38 3.77 4.15 4.30      4.37 4.04 4.57 4.37      4.38 4.73 4.59 4.82      4.58 4.82 4.66 5.76
// A grid between a half and one block per SM is faster
// still as long as every launch has the same size, because all blocks of the next launch then find a place and prefetch, but
// not when the batch shrinks from launch to launch and two blocks of a launch meet on one SM (112 rows of 304 KB: one
// block per row 10.5 us against 13.6, two 11.0 either way), so it is not sought.
// Long rows, somewhat more than SMs (149 to 197): 3 blocks per row, which is at most two full rounds of two blocks per SM; fewer
// and longer blocks leave much of the GPU idle at the end.  us with 1, 2, 3 and 4 blocks:
//                      149 rows                     160 rows                     197 rows                  198 rows (not)
//     390 KB (not)  15.8 15.5 14.9 15.9        16.1 16.0 15.9 16.3        17.4 16.9 18.4 18.2        17.5 17.0 18.5 18.3
//     449 KB        18.4 17.0 16.0 17.6        20.0 17.7 17.2 18.4        21.0 19.0 20.5 20.5        21.0 19.0 20.6 20.5
//     500 KB fp32   18.5 19.4 17.6 19.7        18.6 20.8 19.0 21.1        21.5 21.6 21.6 23.5        21.6 21.6 21.7 23.6
//     500 KB bf16   25.4 26.3 21.2 26.5        25.8 27.7 23.1 26.8        26.3 28.4 25.5 31.8        26.3 28.6 25.6 32.0
//     594 KB        22.4 21.3 19.4 20.1        23.2 22.9 20.9 20.9        24.8 24.4 23.9 24.5        25.0 24.7 24.1 24.5
//     1000 KB       36.2 34.2 29.0 29.6        38.0 36.8 31.2 32.3        41.0 39.0 36.3 38.1        41.5 39.2 36.6 38.4
int pick_draft_cluster(const svip_ctx* ctx, long rows, int V, int dtype) {
    const int S = pick_cluster(ctx, rows, V, dtype);
    const long nvec = (static_cast<long>(V) * (dtype == SVIP_BF16 ? 2 : 4) + 15) / 16;
    if (ctx->cluster_override == 0 && rows > ctx->num_sms && 3 * rows <= 4L * ctx->num_sms && nvec * 16 > (448L << 10)) return 3;
    const bool shorter = nvec < 8L * kThreads || (nvec <= 16L * kThreads && rows >= 8);
    if (ctx->cluster_override > 0 || S <= 4 || !shorter) return S;
    return rows * 5 > ctx->num_sms ? 2 : 4;
}

// Blocks per row of the threshold kernel.  Its blocks hold over 100 KB of shared memory and its rows take several
// exchanges, so a cluster that finds no place until another one has left costs a whole second round: a size is used
// only if all clusters fit at once, with two left as slack for the blocks of the neighbouring launches (33 clusters of 8
// fit: 32 rows of 304 KB take 9.1 us as clusters of 8, 7.6 as clusters of 6).  Up to that the largest size of a list:
//   top-k    powers of two (16 rows of 64 KB: 6.5 us with 2, 6.7 with 3 or 4, 7.0 with 6 or 8; 16 of 390 KB 7.3 with 8, 7.6 with 4,
//            8.8 with 6); 6 where with 4 the segments do not fit the ring, so that stretches are fetched again (32 rows of
//            304 KB: 7.6 us with 6, 8.8 with 4; 36 of 1 MB 12.0 and 13.7).  For 32 to 64 rows of 64 KB 2 would be faster than 4, which
//            the list takes (6.4 and 7.2 us), for longer rows 4 (64 of 1 MB 16.1 and 17.4)
//   nucleus  6, 4, 3 for long rows, 2 (16 rows of 304 KB: 8.6 us with 6, 9.4 with 4, 12.3 with 2; 64 of 1 MB 22.9 with 4, 25.1 with 2; 72 of
//            128 KB 9.2 with 2 and 9.9 with 3, but 72 of 304 KB also 13.9 with 2 and 14.8 with 3); 8 up to 8 rows, for likely and flat
//            rows alike (8 rows of 608 KB 8.6 us with 8, 8.8 with 6, flat 41.5 and 47.7; of 512 KB 7.6 and 8.5, flat 36.1 and
//            43.7; of 1 MB 10.1 and 10.6, flat 53.6 and 63.6; but 16 rows of 608 KB 10.7 and 10.1, flat 55 either way)
// and 2 rather than 1 as long as it fits (nucleus, 144 rows of 304 KB: 19.3 against 20.3 us).  Launches that fit with no size
// are cut as those of the other kernels, but the nucleus alone, whose second pass over the row is as long as the first, takes 3
// where that is at most two full rounds of blocks (rows of 384 KB up to 6/5 rows per SM, of 768 KB up to 4/3), and again from two
// rows per SM on where the rows are so long (896 KB) that fewer blocks per row would bring more rows than L2 holds between the two
// passes; between these flat rows lose more than the others gain.  us with the number of the other kernels and with 3, for rows
// with a few likely tokens and for flat rows, which take the descent:
//                               likely        flat                                       likely        flat
//     160 x 250 KB fp32 (not)  20.3  21.9   117  116          180 x 1000 KB fp32        68.9  53.8   345  324
//     160 x 297 KB bf16 (not)  28.1  28.0   159  140          200 x 1000 KB fp32 (not)  74.4  67.7   348  392
//     160 x 390 KB bf16        34.5  32.6   201  172          200 x 1000 KB bf16 (not)  70.7  74.9   417  466
//     177 x 390 KB bf16        35.0  33.1   201  173          280 x 1000 KB fp32 (not)  89.6  83.6   427  515
//     160 x 500 KB fp32        32.4  31.5   209  181          300 x 1000 KB fp32       103.0  88.1   538  536
//     160 x 703 KB fp32        44.9  40.5   252  238          300 x 1000 KB bf16       106.4  96.2   642  626
//     280 x 781 KB fp32 (not)  68.8  70.1   343  424          600 x 1000 KB fp32       182.6 153.4   929  999
//     280 x 781 KB bf16 (not)  71.9  77.9   404  494          600 x  781 KB fp32 (not) 137.1 128.4   745  817
int pick_threshold_cluster(const svip_ctx* ctx, long rows, int V, int dtype, bool top_k) {
    if (ctx->cluster_override > 0) return ctx->cluster_override;
    const long nvec = (static_cast<long>(V) * (dtype == SVIP_BF16 ? 2 : 4) + 15) / 16;
    const auto resident = [&](int S) { return nvec <= static_cast<long>(S) * kWarps * 32 * kStages; };
    const int sizes[] = {8, 6, 4, 3, 2};
    for (const int S : sizes) {
        if (rows > ctx->max_clusters[S] - 2 || nvec < static_cast<long>(S) * kThreads) continue;
        if (top_k ? S == 3 || (S == 6 && resident(4)) : (S == 8 && rows > 8) || (S == 3 && nvec * 16 < (256L << 10))) continue;
        return S;
    }
    const long kb = nvec * 16 >> 10;
    if (!top_k) {
        if (3 * rows <= 4L * ctx->num_sms && kb >= (5 * rows <= 6L * ctx->num_sms ? 384 : 768)) return 3;
        if (rows >= 2L * ctx->num_sms && kb >= 896) return 3;
    }
    return pick_cluster(ctx, rows, V, dtype);
}

// Bytes from the start of the first row to the end of the last one.
[[maybe_unused]] size_t rows_extent(long n_rows, long row_stride, int V, size_t esz) {
    if (n_rows < 1) return 0;
    return (static_cast<size_t>(n_rows - 1) * static_cast<size_t>(row_stride) + static_cast<size_t>(V)) * esz;
}

// -DSVIP_DEBUG_BOUNDS: the extents of the (up to two) logits buffers of a call go into constant memory
// ahead of its kernels, which then refuse loads outside them (see debug_ok).  The vector loads start at the
// 16-byte boundary below a row and end at the one above it, hence the rounding.
#ifdef SVIP_DEBUG_BOUNDS
cudaError_t debug_ranges(const svip_ctx* ctx, cudaStream_t st, const void* p0, size_t bytes0, const void* p1 = nullptr,
                         size_t bytes1 = 0) {
    DebugRange r[2];
    const void* p[2] = {p0, p1};
    const size_t n[2] = {bytes0, bytes1};
    for (int i = 0; i < 2; ++i) {
        const unsigned long long a = reinterpret_cast<unsigned long long>(p[i]);
        r[i].lo = p[i] ? (a & ~15ull) : 0;
        r[i].hi = p[i] ? ((a + n[i] + 15ull) & ~15ull) : 0;
        if (p[i] && n[i] == ~static_cast<size_t>(0)) { r[i].lo = 0; r[i].hi = ~0ull; }   // extent not known
    }
    if (ctx->capturing) return cudaSuccess;      // no copies from host memory into a graph; see debug_no_ranges
    return cudaMemcpyToSymbolAsync(g_debug_range, r, sizeof r, 0, cudaMemcpyHostToDevice, st);
}
// Ahead of the replay of a graph, whose buffers are not known any more: its loads are not those of the last call made singly.
cudaError_t debug_no_ranges(cudaStream_t st) {
    DebugRange r[2];
    r[0].lo = r[1].lo = r[1].hi = 0;
    r[0].hi = ~0ull;
    return cudaMemcpyToSymbolAsync(g_debug_range, r, sizeof r, 0, cudaMemcpyHostToDevice, st);
}
#define SVIP_DEBUG_RANGES(...) do { if (debug_ranges(__VA_ARGS__) != cudaSuccess) return SVIP_ERR_CUDA; } while (0)
#else
#define SVIP_DEBUG_RANGES(...) do { } while (0)
#endif

template <bool kDraft>
auto threshold_kernel(svip_dtype dtype, const ThresholdArgs& a) -> void (*)(ThresholdArgs) {
    if (a.top_k > 0) return dtype == SVIP_BF16 ? row_threshold_kernel<kBF16, kDraft, true> : row_threshold_kernel<kF32, kDraft, true>;
    return dtype == SVIP_BF16 ? row_threshold_kernel<kBF16, kDraft, false> : row_threshold_kernel<kF32, kDraft, false>;
}

// The node that a stream under capture has recorded last, if its next one would depend on that one alone.
cudaGraphNode_t last_node(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    const cudaGraphNode_t* deps = nullptr;
    size_t n = 0;
    if (cudaStreamGetCaptureInfo(st, &status, nullptr, nullptr, &deps, &n) != cudaSuccess) return nullptr;
    return status == cudaStreamCaptureStatusActive && n == 1 ? deps[0] : nullptr;
}

// A policy step that directly follows the position-indexed draft step of the same sequences in the body of a drafting
// loop is taken by that kernel (advance_one): one kernel per drafted token instead of two.  Returns false if it does not
// fit (then the step stays a kernel of its own).
bool join_draft_step(svip_ctx* ctx, const AdvanceArgs& a) {
    if (!ctx->loop_draft_node || last_node(ctx->loop_stream) != ctx->loop_draft_node) return false;
    DraftArgs d = ctx->loop_draft_args;
    if (d.pos != a.draft_len || d.active != a.active || ctx->loop_draft_rows != a.B) return false;
    if (a.policy == SVIP_POLICY_ENTROPY && d.stop != a.stop) return false;
    d.adv = a;
    d.adv.arrived = ctx->loop_arrived;
    cudaKernelNodeParams p = {};
    if (cudaGraphKernelNodeGetParams(ctx->loop_draft_node, &p) != cudaSuccess) { cudaGetLastError(); return false; }
    void* args[] = {&d};
    p.kernelParams = args;
    p.extra = nullptr;
    if (cudaGraphKernelNodeSetParams(ctx->loop_draft_node, &p) != cudaSuccess) { cudaGetLastError(); return false; }
    ctx->loop_draft_node = nullptr;
    return true;
}

bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

float scale_for(float T) { return static_cast<float>(1.4426950408889634 / (T > 0.f ? static_cast<double>(T) : 1.0)); }

}  // namespace

extern "C" {

const char* svip_strerror(int status) {
    switch (status) {
        case SVIP_OK: return "ok";
        case SVIP_ERR_INVALID_ARG: return "invalid argument";
        case SVIP_ERR_UNSUPPORTED: return "unsupported dtype or device";
        case SVIP_ERR_WORKSPACE: return "more rows than the context's workspace holds";
        case SVIP_ERR_CUDA: return "CUDA runtime error";
        case SVIP_ERR_STATE: return "call not valid in the context's current state";
        default: return "unknown status";
    }
}

int svip_version(void) { return 200; }

int svip_last_cuda_error(const svip_ctx* ctx) { return ctx ? ctx->last_cuda : 0; }

int svip_create(svip_ctx** out, int device, int max_rows) {
    if (!out || max_rows < 1 || device < 0) return SVIP_ERR_INVALID_ARG;
    int prev = 0;
    if (cudaGetDevice(&prev) != cudaSuccess) { cudaGetLastError(); return SVIP_ERR_CUDA; }
    if (cudaSetDevice(device) != cudaSuccess) { cudaGetLastError(); return SVIP_ERR_CUDA; }
    int rc = SVIP_OK;
    svip_ctx* c = new (std::nothrow) svip_ctx();
    if (!c) { cudaSetDevice(prev); return SVIP_ERR_CUDA; }
    c->device = device;
    c->max_rows = max_rows;
    int major = 0, sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) rc = SVIP_ERR_CUDA;
    else if (major != 10) rc = SVIP_ERR_UNSUPPORTED;
    c->num_sms = sms;
    if (rc == SVIP_OK) {
        // the cp.async rings need more dynamic shared memory than the default limit
        const void* ringed[] = {
            (const void*)draft_step_kernel<kBF16, true, 2>, (const void*)draft_step_kernel<kBF16, false, 2>,
            (const void*)draft_step_kernel<kF32, true, 2>,  (const void*)draft_step_kernel<kF32, false, 2>,
            (const void*)draft_step_kernel<kBF16, true, 3>, (const void*)draft_step_kernel<kBF16, false, 3>,
            (const void*)draft_step_kernel<kF32, true, 3>,  (const void*)draft_step_kernel<kF32, false, 3>,
            (const void*)draft_step_kernel<kBF16, true, 2, true>, (const void*)draft_step_kernel<kBF16, false, 2, true>,
            (const void*)draft_step_kernel<kF32, true, 2, true>,  (const void*)draft_step_kernel<kF32, false, 2, true>,
            (const void*)row_stats_kernel<kBF16, 0>,     (const void*)row_stats_kernel<kBF16, 1>,
            (const void*)row_stats_kernel<kF32, 0>,      (const void*)row_stats_kernel<kF32, 1>,
            (const void*)verify_finish_kernel<kBF16>,    (const void*)verify_finish_kernel<kF32>,
            (const void*)row_stats_kernel<kBF16, 2>,     (const void*)row_stats_kernel<kF32, 2>,
            (const void*)row_threshold_kernel<kBF16, false, false>, (const void*)row_threshold_kernel<kF32, false, false>,
            (const void*)row_threshold_kernel<kBF16, false, true>,  (const void*)row_threshold_kernel<kF32, false, true>,
            (const void*)row_threshold_kernel<kBF16, true, false>,  (const void*)row_threshold_kernel<kF32, true, false>,
            (const void*)row_threshold_kernel<kBF16, true, true>,   (const void*)row_threshold_kernel<kF32, true, true>,
            (const void*)draft_step_kernel<kBF16, false, 2, false, true>, (const void*)draft_step_kernel<kF32, false, 2, false, true>,
            (const void*)row_stats_kernel<kBF16, 1, true>, (const void*)row_stats_kernel<kF32, 1, true>,
            (const void*)verify_finish_kernel<kBF16, true>, (const void*)verify_finish_kernel<kF32, true>,
            (const void*)pair_stats_kernel<kBF16>, (const void*)pair_stats_kernel<kF32>,
            (const void*)pair_stats_kernel<kBF16, true>, (const void*)pair_stats_kernel<kF32, true>,
            (const void*)verify_scan_kernel<kBF16, false>, (const void*)verify_scan_kernel<kF32, false>,
            (const void*)verify_scan_kernel<kBF16, true>, (const void*)verify_scan_kernel<kF32, true>};
        for (const void* k : ringed)
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes) != cudaSuccess)
                rc = SVIP_ERR_CUDA;
    }
    for (int S = 1; S <= kMaxCluster && rc == SVIP_OK; ++S) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(static_cast<unsigned>(S), 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = kRingBytes;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = static_cast<unsigned>(S);
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&c->max_clusters[S], (const void*)row_threshold_kernel<kF32, true, true>, &cfg) != cudaSuccess)
            rc = SVIP_ERR_CUDA;
    }
    if (rc == SVIP_OK) {
        size_t n = static_cast<size_t>(max_rows);
        if (cudaMalloc(&c->p_stats, n * sizeof(float2)) != cudaSuccess ||
            cudaMalloc(&c->q_stats, n * sizeof(float2)) != cudaSuccess ||
            cudaMalloc(&c->p_argmax, n * sizeof(int32_t)) != cudaSuccess ||
            cudaMalloc(&c->status, sizeof(unsigned)) != cudaSuccess ||
            cudaMemset(c->status, 0, sizeof(unsigned)) != cudaSuccess ||
            cudaMalloc(&c->loop_arrived, kLoopStateBytes) != cudaSuccess ||
            cudaMemset(c->loop_arrived, 0, kLoopStateBytes) != cudaSuccess) {
            rc = SVIP_ERR_CUDA;
        }
        c->loop_iter = reinterpret_cast<int*>(c->loop_arrived + 1);
    }
    if (rc != SVIP_OK) {
        cudaGetLastError();
        cudaFree(c->p_stats); cudaFree(c->q_stats); cudaFree(c->p_argmax); cudaFree(c->status);
        cudaFree(c->loop_arrived);
        delete c;
    } else {
        *out = c;
    }
    cudaSetDevice(prev);
    return rc;
}

int svip_destroy(svip_ctx* ctx) {
    if (!ctx) return SVIP_ERR_INVALID_ARG;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(ctx->device);
    cudaFree(ctx->p_stats); cudaFree(ctx->q_stats); cudaFree(ctx->p_argmax); cudaFree(ctx->status);
    cudaFree(ctx->loop_arrived);
    if (ctx->loop_stream) cudaStreamDestroy(ctx->loop_stream);
    if (ctx->prof_start) {
        for (int k = 0; k < kProfilePairs; ++k) {
            cudaEventDestroy(ctx->prof_start[k]);
            cudaEventDestroy(ctx->prof_stop[k]);
        }
        delete[] ctx->prof_start;
        delete[] ctx->prof_stop;
    }
    cudaSetDevice(prev);
    delete ctx;
    return SVIP_OK;
}

int svip_set_cluster_size(svip_ctx* ctx, int cluster_size) {
    if (!ctx) return SVIP_ERR_INVALID_ARG;
    if (cluster_size < 0 || cluster_size > kMaxCluster) return SVIP_ERR_INVALID_ARG;
    ctx->cluster_override = cluster_size;
    return SVIP_OK;
}

long svip_launch_count(const svip_ctx* ctx) { return ctx ? ctx->launches : 0; }

int svip_read_status(svip_ctx* ctx, unsigned* flags, void* stream) {
    if (!ctx || !flags) return SVIP_ERR_INVALID_ARG;
    if (ctx->capturing) return SVIP_ERR_STATE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, ctx->status, sizeof v, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->status, 0, sizeof v, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
#ifdef SVIP_DEBUG_BOUNDS
    unsigned oob = 0, zero = 0;
    e = cudaMemcpyFromSymbol(&oob, g_debug_oob, sizeof oob);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_debug_oob, &zero, sizeof zero);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if (oob) v |= SVIP_STATUS_DEBUG_OOB;
#endif
    *flags = v;
    return SVIP_OK;
}

static int draft_impl(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                      long pos_stride, const int32_t* pos, long slot_stride, float T, float thresh,
                      const float* uniforms, const uint8_t* active, const float* thr, int32_t* token,
                      float* entropy, uint8_t* stop, float* row_stats, void* stream);

int svip_draft_step(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                    float T, float thresh, const float* uniforms, int32_t* token, float* entropy,
                    uint8_t* stop, float* row_stats, void* stream) {
    return svip_draft_step_masked(ctx, logits, dtype, B, V, row_stride, T, thresh, uniforms, nullptr, token,
                                  entropy, stop, row_stats, stream);
}

int svip_draft_step_masked(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                           float T, float thresh, const float* uniforms, const uint8_t* active,
                           int32_t* token, float* entropy, uint8_t* stop, float* row_stats, void* stream) {
    return svip_draft_step_at(ctx, logits, dtype, B, V, row_stride, 0, nullptr, 0, T, thresh, uniforms, active,
                              token, entropy, stop, row_stats, stream);
}

int svip_draft_step_at(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                       long pos_stride, const int32_t* pos, long slot_stride, float T, float thresh,
                       const float* uniforms, const uint8_t* active, int32_t* token, float* entropy,
                       uint8_t* stop, float* row_stats, void* stream) {
    return draft_impl(ctx, logits, dtype, B, V, row_stride, pos_stride, pos, slot_stride, T, thresh, uniforms, active,
                      nullptr, token, entropy, stop, row_stats, stream);
}

int svip_draft_step_filtered(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                             float T, float thresh, const float* uniforms, const uint8_t* active, const float* thr,
                             int32_t* token, float* entropy, uint8_t* stop, float* row_stats, void* stream) {
    if (!thr || !(T > 0.f)) return SVIP_ERR_INVALID_ARG;
    return draft_impl(ctx, logits, dtype, B, V, row_stride, 0, nullptr, 0, T, thresh, uniforms, active, thr, token,
                      entropy, stop, row_stats, stream);
}

static int draft_impl(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                      long pos_stride, const int32_t* pos, long slot_stride, float T, float thresh,
                      const float* uniforms, const uint8_t* active, const float* thr, int32_t* token,
                      float* entropy, uint8_t* stop, float* row_stats, void* stream) {
    if (!ctx || !logits || !token || !entropy || !stop) return SVIP_ERR_INVALID_ARG;
    if (pos_stride < 0 || slot_stride < 0) return SVIP_ERR_INVALID_ARG;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (B < 0 || V < 1 || V > 0x7fffffe0 || row_stride < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T >= 0.f) || std::isinf(T) || std::isnan(thresh)) return SVIP_ERR_INVALID_ARG;
    if (T > 0.f && !uniforms) return SVIP_ERR_INVALID_ARG;
    if (!aligned_to(logits, dtype == SVIP_BF16 ? 2 : 4)) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    SVIP_RANGE("svip_draft_step");
    SVIP_DEBUG_RANGES(ctx, static_cast<cudaStream_t>(stream), logits,
                      pos ? ~static_cast<size_t>(0) : rows_extent(B, row_stride, V, dtype == SVIP_BF16 ? 2 : 4));
    DraftArgs a;
    a.logits = logits; a.row_stride = row_stride; a.V = V; a.c = scale_for(T); a.thresh = thresh;
    a.greedy = T > 0.f ? 0 : 1; a.uniforms = uniforms; a.token = token; a.entropy = entropy;
    a.stop = stop; a.row_stats = row_stats; a.status = ctx->status; a.active = active;
    a.ext_target = nullptr; a.token_offset = 0;
    a.pos = pos; a.pos_stride = pos_stride; a.slot_stride = slot_stride; a.thr = thr; a.adv.arrived = nullptr;
    const int S = pick_draft_cluster(ctx, B, V, dtype);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool waves = static_cast<long>(B) * S > 2L * ctx->num_sms;
    void (*k)(DraftArgs);
    if (dtype == SVIP_BF16)
        k = a.greedy ? (waves ? draft_step_kernel<kBF16, true, 3> : draft_step_kernel<kBF16, true, 2>)
                     : (waves ? draft_step_kernel<kBF16, false, 3> : draft_step_kernel<kBF16, false, 2>);
    else
        k = a.greedy ? (waves ? draft_step_kernel<kF32, true, 3> : draft_step_kernel<kF32, true, 2>)
                     : (waves ? draft_step_kernel<kF32, false, 3> : draft_step_kernel<kF32, false, 2>);
    if (pos) {
        if (dtype == SVIP_BF16) k = a.greedy ? draft_step_kernel<kBF16, true, 2, true> : draft_step_kernel<kBF16, false, 2, true>;
        else k = a.greedy ? draft_step_kernel<kF32, true, 2, true> : draft_step_kernel<kF32, false, 2, true>;
    }
    if (thr) k = dtype == SVIP_BF16 ? draft_step_kernel<kBF16, false, 2, false, true> : draft_step_kernel<kF32, false, 2, false, true>;
    cudaError_t e = launch_clustered(k, B, S, a, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    if (pos && ctx->loop_open && st == ctx->loop_stream) {      // svip_policy_advance may join this kernel
        ctx->loop_draft_node = last_node(st);
        ctx->loop_draft_args = a;
        ctx->loop_draft_rows = B;
    }
    return SVIP_OK;
}

int svip_row_threshold(svip_ctx* ctx, const void* logits, svip_dtype dtype, int n_rows, int V, long row_stride,
                       float T, int top_k, float top_p, float* thr, float* stats, void* stream) {
    if (!ctx || !logits || !thr) return SVIP_ERR_INVALID_ARG;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (n_rows < 0 || V < 1 || V > 0x7fffffe0 || row_stride < 0 || top_k < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T > 0.f) || std::isinf(T) || !(top_p > 0.f)) return SVIP_ERR_INVALID_ARG;
    if (!aligned_to(logits, dtype == SVIP_BF16 ? 2 : 4)) return SVIP_ERR_INVALID_ARG;
    if (n_rows == 0) return SVIP_OK;
    SVIP_RANGE("svip_row_threshold");
    SVIP_DEBUG_RANGES(ctx, static_cast<cudaStream_t>(stream), logits, rows_extent(n_rows, row_stride, V, dtype == SVIP_BF16 ? 2 : 4));
    ThresholdArgs a;
    a.logits = logits; a.row_stride = row_stride; a.V = V; a.c = scale_for(T);
    a.top_k = (top_k >= 1 && top_k < V) ? top_k : 0; a.top_p = top_p; a.thr = thr;
    a.stats = reinterpret_cast<float2*>(stats);
    if (stats && !aligned_to(stats, 8)) return SVIP_ERR_INVALID_ARG;
    a.uniforms = nullptr; a.active = nullptr; a.thresh = 0.f; a.token = nullptr; a.entropy = nullptr;
    a.stop = nullptr; a.status = ctx->status;
    const int S = pick_threshold_cluster(ctx, n_rows, V, dtype, a.top_k > 0);
    a.groups = choose_groups(S, a.top_k);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = launch_clustered(threshold_kernel<false>(dtype, a), n_rows, S, a, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_draft_step_truncated(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V, long row_stride,
                              float T, float thresh, int top_k, float top_p, const float* uniforms,
                              const uint8_t* active, float* thr, int32_t* token, float* entropy, uint8_t* stop,
                              float* row_stats, void* stream) {
    if (!ctx || !logits || !thr || !token || !entropy || !stop || !uniforms) return SVIP_ERR_INVALID_ARG;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (B < 0 || V < 1 || V > 0x7fffffe0 || row_stride < 0 || top_k < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T > 0.f) || std::isinf(T) || !(top_p > 0.f) || std::isnan(thresh)) return SVIP_ERR_INVALID_ARG;
    if (!aligned_to(logits, dtype == SVIP_BF16 ? 2 : 4)) return SVIP_ERR_INVALID_ARG;
    if (row_stats && !aligned_to(row_stats, 8)) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    SVIP_RANGE("svip_draft_step_truncated");
    SVIP_DEBUG_RANGES(ctx, static_cast<cudaStream_t>(stream), logits, rows_extent(B, row_stride, V, dtype == SVIP_BF16 ? 2 : 4));
    ThresholdArgs a;
    a.logits = logits; a.row_stride = row_stride; a.V = V; a.c = scale_for(T);
    a.top_k = (top_k >= 1 && top_k < V) ? top_k : 0; a.top_p = top_p; a.thr = thr;
    a.stats = reinterpret_cast<float2*>(row_stats);
    a.uniforms = uniforms; a.active = active; a.thresh = thresh; a.token = token; a.entropy = entropy;
    a.stop = stop; a.status = ctx->status;
    const int S = pick_threshold_cluster(ctx, B, V, dtype, a.top_k > 0);
    a.groups = choose_groups(S, a.top_k);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = launch_clustered(threshold_kernel<true>(dtype, a), B, S, a, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_pack_ragged(svip_ctx* ctx, const int32_t* draft_len, int B, int K_max, int32_t* cu_rows,
                     int32_t* row_seq, int32_t* row_pos, void* stream) {
    if (!ctx || !draft_len || !cu_rows) return SVIP_ERR_INVALID_ARG;
    if (B < 1 || B > 65536 || K_max < 1) return SVIP_ERR_INVALID_ARG;
    if (static_cast<long>(B) * (static_cast<long>(K_max) + 1) >= 0x7fffffffL) return SVIP_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = launch_ex(pack_ragged_kernel, 1, kPackThreads, 0, 0, st, draft_len, B, K_max, cu_rows, row_seq,
                              row_pos, ctx->status);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

// The verification round; q_thr / p_thr are both NULL (plain distributions) or both given
// (distributions truncated at those per-row thresholds).
static int verify_impl(svip_ctx* ctx, const int32_t* draft_tokens, const void* q_logits, long q_row_stride,
                       const float* q_stats, long q_seq_stride, long q_pos_stride, const void* target_logits,
                       long t_row_stride, svip_dtype dtype, const int32_t* cu_rows, int B, int K,
                       int n_target_rows, int V, float T, const float* uniforms, int32_t* n_accepted,
                       int32_t* next_token, void* stream, const float* q_thr, const float* p_thr,
                       const float* p_stats_user, bool early_exit = false) {
    if (!ctx || !draft_tokens || !target_logits || !n_accepted || !next_token) return SVIP_ERR_INVALID_ARG;
    const bool truncated = q_thr != nullptr;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (B < 0 || K < 1 || V < 1 || V > 0x7fffffe0 || t_row_stride < 0 || q_row_stride < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T >= 0.f) || std::isinf(T)) return SVIP_ERR_INVALID_ARG;
    const bool sampling = T > 0.f;
    if (sampling && (!q_logits || !uniforms)) return SVIP_ERR_INVALID_ARG;
    if (q_seq_stride < 0 && q_seq_stride != SVIP_Q_PACKED) return SVIP_ERR_INVALID_ARG;
    if (q_seq_stride >= 0 && q_pos_stride < 0) return SVIP_ERR_INVALID_ARG;
    const size_t esz = dtype == SVIP_BF16 ? 2 : 4;
    if (!aligned_to(target_logits, esz) || (q_logits && !aligned_to(q_logits, esz))) return SVIP_ERR_INVALID_ARG;
    if (static_cast<long>(B) * (static_cast<long>(K) + 1) >= 0x7fffffffL) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return n_target_rows == 0 ? SVIP_OK : SVIP_ERR_INVALID_ARG;
    if (n_target_rows < 2 * B || n_target_rows > B * (K + 1)) return SVIP_ERR_INVALID_ARG;
    if (!cu_rows && n_target_rows != B * (K + 1)) return SVIP_ERR_INVALID_ARG;
    if (n_target_rows > ctx->max_rows) return SVIP_ERR_WORKSPACE;

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const float c = scale_for(T);
    cudaError_t e;
    SVIP_RANGE("svip_verify");
    {
        [[maybe_unused]] const long q_rows =
            q_seq_stride < 0 ? n_target_rows - B : (B - 1) * q_seq_stride + (static_cast<long>(K) - 1) * q_pos_stride + 1;
        SVIP_DEBUG_RANGES(ctx, st, target_logits, rows_extent(n_target_rows, t_row_stride, V, esz), q_logits,
                          rows_extent(q_rows, q_row_stride, V, esz));
    }

    StatsArgs s;
    s.logits = target_logits; s.row_stride = t_row_stride; s.V = V; s.c = c; s.draft_rows = 0; s.K = K;
    s.cu = cu_rows; s.q_seq_stride = q_seq_stride; s.q_pos_stride = q_pos_stride;
    s.out_stats = ctx->p_stats; s.out_argmax = sampling ? nullptr : ctx->p_argmax; s.status = ctx->status;
    s.out_partial = nullptr; s.idx_offset = 0; s.thr = p_thr;
    int S = pick_cluster(ctx, n_target_rows, V, dtype);
    const bool timed = ctx->profiling && !ctx->capturing && ctx->prof_used < kProfilePairs;
    if (early_exit) {
        // the draft rows' normalisers first (the accept test of a position needs them), then one cluster
        // per sequence walks the target rows up to the first rejection
        if (sampling && !q_stats) {
            StatsArgs d = s;
            d.logits = q_logits; d.row_stride = q_row_stride; d.draft_rows = 1;
            d.out_stats = ctx->q_stats; d.out_argmax = nullptr; d.thr = nullptr;
            const int Sd = pick_cluster(ctx, n_target_rows - B, V, dtype);
            e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1>, static_cast<long>(B) * K, Sd, d, st, kRingBytes)
                                   : launch_clustered(row_stats_kernel<kF32, 1>, static_cast<long>(B) * K, Sd, d, st, kRingBytes);
            if (e != cudaSuccess) return cuda_fail(ctx, e);
            ctx->launches += 1;
        }
        FinishArgs w;
        w.draft_tokens = draft_tokens; w.q_logits = q_logits; w.q_row_stride = q_row_stride;
        w.q_stats_user = reinterpret_cast<const float2*>(q_stats); w.q_stats_ws = ctx->q_stats;
        w.q_seq_stride = q_seq_stride; w.q_pos_stride = q_pos_stride; w.t_logits = target_logits;
        w.t_row_stride = t_row_stride; w.p_stats = ctx->p_stats; w.p_stats_out = ctx->p_stats;
        w.cu = cu_rows; w.K = K; w.V = V; w.c = c;
        w.uniforms = uniforms; w.n_accepted = n_accepted; w.next_token = next_token; w.status = ctx->status;
        w.p_thr = nullptr; w.q_thr = nullptr; w.after_stats = 0;
        // one cluster per sequence, cut as for the finish kernel (measured on 256 sequences of 1 MB rows: 2 or 4
        // blocks per sequence are equally fast, 8 are slower; on 32 sequences of 304 KB rows 8 are fastest)
        int Sw = pick_cluster(ctx, B, V, dtype);
        if (ctx->cluster_override == 0) {
            const long row_bytes = static_cast<long>(V) * static_cast<long>(esz);
            while (Sw < 4 && 2 * row_bytes / Sw > (512L << 10)) Sw *= 2;
        }
        if (timed) cudaEventRecord(ctx->prof_start[ctx->prof_used], st);
        if (sampling)
            e = dtype == SVIP_BF16 ? launch_clustered(verify_scan_kernel<kBF16, false>, B, Sw, w, st, kRingBytes)
                                   : launch_clustered(verify_scan_kernel<kF32, false>, B, Sw, w, st, kRingBytes);
        else
            e = dtype == SVIP_BF16 ? launch_clustered(verify_scan_kernel<kBF16, true>, B, Sw, w, st, kRingBytes)
                                   : launch_clustered(verify_scan_kernel<kF32, true>, B, Sw, w, st, kRingBytes);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        ctx->launches += 1;
        if (timed) cudaEventRecord(ctx->prof_stop[ctx->prof_used++], st);
        return SVIP_OK;
    } else {
    if (timed) cudaEventRecord(ctx->prof_start[ctx->prof_used], st);
    if (p_stats_user)
        e = cudaSuccess;   // the caller already holds (m, Z) of every target row
    else if (truncated)
        e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1, true>, n_target_rows, S, s, st, kRingBytes)
                               : launch_clustered(row_stats_kernel<kF32, 1, true>, n_target_rows, S, s, st, kRingBytes);
    else if (sampling)
        e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1>, n_target_rows, S, s, st, kRingBytes)
                               : launch_clustered(row_stats_kernel<kF32, 1>, n_target_rows, S, s, st, kRingBytes);
    else
        e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 0>, n_target_rows, S, s, st, kRingBytes)
                               : launch_clustered(row_stats_kernel<kF32, 0>, n_target_rows, S, s, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if (!p_stats_user) ctx->launches += 1;
    if (timed) cudaEventRecord(ctx->prof_stop[ctx->prof_used++], st);

    }
    if (!sampling) {
        GreedyArgs g;
        g.draft_tokens = draft_tokens; g.p_argmax = ctx->p_argmax; g.cu = cu_rows;
        g.q_seq_stride = q_seq_stride; g.q_pos_stride = q_pos_stride; g.B = B; g.K = K;
        g.n_accepted = n_accepted; g.next_token = next_token;
        e = launch_ex(verify_greedy_kernel, static_cast<unsigned>((B + kWarps - 1) / kWarps), kThreads, 0, 0, st, g);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        ctx->launches += 1;
        return SVIP_OK;
    }

    if (!q_stats) {
        StatsArgs d = s;
        d.logits = q_logits; d.row_stride = q_row_stride; d.draft_rows = 1;
        d.out_stats = ctx->q_stats; d.out_argmax = nullptr; d.thr = q_thr;
        long units = static_cast<long>(B) * K;
        int Sd = pick_cluster(ctx, n_target_rows - B, V, dtype);
        if (truncated)
            e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1, true>, units, Sd, d, st, kRingBytes)
                                   : launch_clustered(row_stats_kernel<kF32, 1, true>, units, Sd, d, st, kRingBytes);
        else
            e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1>, units, Sd, d, st, kRingBytes)
                                   : launch_clustered(row_stats_kernel<kF32, 1>, units, Sd, d, st, kRingBytes);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        ctx->launches += 1;
    }

    FinishArgs f;
    f.draft_tokens = draft_tokens; f.q_logits = q_logits; f.q_row_stride = q_row_stride;
    f.q_stats_user = reinterpret_cast<const float2*>(q_stats); f.q_stats_ws = ctx->q_stats;
    f.q_seq_stride = q_seq_stride; f.q_pos_stride = q_pos_stride; f.t_logits = target_logits;
    f.t_row_stride = t_row_stride;
    f.p_stats = p_stats_user ? reinterpret_cast<const float2*>(p_stats_user) : ctx->p_stats;
    f.cu = cu_rows; f.K = K; f.V = V; f.c = c;
    f.uniforms = uniforms; f.n_accepted = n_accepted; f.next_token = next_token; f.status = ctx->status;
    f.p_thr = p_thr; f.q_thr = q_thr;
    f.p_stats_out = nullptr;
    f.after_stats = !p_stats_user || !q_stats;
    // up to two rows per sequence are streamed: long rows are cut finer than the one-wave policy
    // asks for (this kernel runs for many microseconds, so several waves are fine)
    int Sf = pick_cluster(ctx, B, V, dtype);
    if (ctx->cluster_override == 0) {
        const long row_bytes = static_cast<long>(V) * static_cast<long>(esz);
        while (Sf < kMaxCluster && 2 * row_bytes / Sf > (512L << 10)) Sf *= 2;
        if (Sf > kMaxCluster) Sf = kMaxCluster;
    }
    if (truncated)
        e = dtype == SVIP_BF16 ? launch_clustered(verify_finish_kernel<kBF16, true>, B, Sf, f, st, kRingBytes)
                               : launch_clustered(verify_finish_kernel<kF32, true>, B, Sf, f, st, kRingBytes);
    else
        e = dtype == SVIP_BF16 ? launch_clustered(verify_finish_kernel<kBF16>, B, Sf, f, st, kRingBytes)
                               : launch_clustered(verify_finish_kernel<kF32>, B, Sf, f, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_verify(svip_ctx* ctx, const int32_t* draft_tokens, const void* q_logits, long q_row_stride,
                const float* q_stats, long q_seq_stride, long q_pos_stride, const void* target_logits,
                long t_row_stride, svip_dtype dtype, const int32_t* cu_rows, int B, int K,
                int n_target_rows, int V, float T, const float* uniforms, int32_t* n_accepted,
                int32_t* next_token, void* stream) {
    return verify_impl(ctx, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                       target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                       n_accepted, next_token, stream, nullptr, nullptr, nullptr);
}

int svip_verify_early_exit(svip_ctx* ctx, const int32_t* draft_tokens, const void* q_logits, long q_row_stride,
                           const float* q_stats, long q_seq_stride, long q_pos_stride, const void* target_logits,
                           long t_row_stride, svip_dtype dtype, const int32_t* cu_rows, int B, int K,
                           int n_target_rows, int V, float T, const float* uniforms, int32_t* n_accepted,
                           int32_t* next_token, void* stream) {
    return verify_impl(ctx, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                       target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                       n_accepted, next_token, stream, nullptr, nullptr, nullptr, true);
}

int svip_verify_filtered(svip_ctx* ctx, const int32_t* draft_tokens, const void* q_logits, long q_row_stride,
                         const float* q_stats, const float* q_thr, long q_seq_stride, long q_pos_stride,
                         const void* target_logits, long t_row_stride, const float* p_thr, const float* p_stats,
                         svip_dtype dtype, const int32_t* cu_rows, int B, int K, int n_target_rows, int V, float T,
                         const float* uniforms, int32_t* n_accepted, int32_t* next_token, void* stream) {
    if (!q_thr || !p_thr || !(T > 0.f)) return SVIP_ERR_INVALID_ARG;
    if (p_stats && !aligned_to(p_stats, 8)) return SVIP_ERR_INVALID_ARG;
    return verify_impl(ctx, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                       target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                       n_accepted, next_token, stream, q_thr, p_thr, p_stats);
}

int svip_profile_enable(svip_ctx* ctx, int on) {
    if (!ctx) return SVIP_ERR_INVALID_ARG;
    if (ctx->capturing) return SVIP_ERR_STATE;
    if (on && !ctx->prof_start) {
        int prev = 0;
        cudaGetDevice(&prev);
        cudaSetDevice(ctx->device);
        ctx->prof_start = new (std::nothrow) cudaEvent_t[kProfilePairs]();
        ctx->prof_stop = new (std::nothrow) cudaEvent_t[kProfilePairs]();
        cudaError_t e = (ctx->prof_start && ctx->prof_stop) ? cudaSuccess : cudaErrorMemoryAllocation;
        for (int k = 0; k < kProfilePairs && e == cudaSuccess; ++k) {
            e = cudaEventCreate(&ctx->prof_start[k]);
            if (e == cudaSuccess) e = cudaEventCreate(&ctx->prof_stop[k]);
        }
        cudaSetDevice(prev);
        if (e != cudaSuccess) {
            delete[] ctx->prof_start; delete[] ctx->prof_stop;   // events created so far leak with the context
            ctx->prof_start = ctx->prof_stop = nullptr;
            return cuda_fail(ctx, e);
        }
    }
    ctx->profiling = on ? 1 : 0;
    ctx->prof_used = 0;
    return SVIP_OK;
}

int svip_profile_read(svip_ctx* ctx, double* total_ms, long* launches) {
    if (!ctx || !total_ms || !launches) return SVIP_ERR_INVALID_ARG;
    if (ctx->capturing) return SVIP_ERR_STATE;
    double sum = 0.0;
    for (int k = 0; k < ctx->prof_used; ++k) {
        cudaError_t e = cudaEventSynchronize(ctx->prof_stop[k]);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ctx->prof_start[k], ctx->prof_stop[k]);
        if (e != cudaSuccess) { ctx->prof_used = 0; return cuda_fail(ctx, e); }
        sum += ms;
    }
    *total_ms = sum;
    *launches = ctx->prof_used;
    ctx->prof_used = 0;
    return SVIP_OK;
}

int svip_verify_tree(svip_ctx* ctx, const int32_t* tokens, const int32_t* parent, const void* q_logits,
                     long q_row_stride, const float* q_stats, const void* target_logits, long t_row_stride,
                     svip_dtype dtype, int B, int N, int V, float T, const float* uniforms,
                     int32_t* n_accepted, int32_t* path, int32_t* next_token, void* stream) {
    if (!ctx || !tokens || !parent || !target_logits || !n_accepted || !path || !next_token) return SVIP_ERR_INVALID_ARG;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (B < 0 || N < 1 || V < 1 || V > 0x7fffffe0 || t_row_stride < 0 || q_row_stride < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T >= 0.f) || std::isinf(T)) return SVIP_ERR_INVALID_ARG;
    const bool sampling = T > 0.f;
    if (sampling && (!q_logits || !uniforms)) return SVIP_ERR_INVALID_ARG;
    const size_t esz = dtype == SVIP_BF16 ? 2 : 4;
    if (!aligned_to(target_logits, esz) || (q_logits && !aligned_to(q_logits, esz))) return SVIP_ERR_INVALID_ARG;
    if (q_stats && !aligned_to(q_stats, 8)) return SVIP_ERR_INVALID_ARG;
    if (static_cast<long>(B) * (static_cast<long>(N) + 1) >= 0x7fffffffL) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    const long n_rows = static_cast<long>(B) * (N + 1);
    if (n_rows > ctx->max_rows) return SVIP_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const float c = scale_for(T);
    cudaError_t e;
    SVIP_RANGE("svip_verify_tree");
    SVIP_DEBUG_RANGES(ctx, st, target_logits, rows_extent(n_rows, t_row_stride, V, esz), q_logits,
                      rows_extent(n_rows, q_row_stride, V, esz));

    StatsArgs s;
    s.logits = target_logits; s.row_stride = t_row_stride; s.V = V; s.c = c; s.draft_rows = 0; s.K = 1;
    s.cu = nullptr; s.q_seq_stride = 0; s.q_pos_stride = 0;
    s.out_stats = ctx->p_stats; s.out_argmax = sampling ? nullptr : ctx->p_argmax; s.status = ctx->status;
    s.out_partial = nullptr; s.idx_offset = 0; s.thr = nullptr;
    const int S = pick_cluster(ctx, n_rows, V, dtype);
    if (sampling)
        e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1>, n_rows, S, s, st, kRingBytes)
                               : launch_clustered(row_stats_kernel<kF32, 1>, n_rows, S, s, st, kRingBytes);
    else
        e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 0>, n_rows, S, s, st, kRingBytes)
                               : launch_clustered(row_stats_kernel<kF32, 0>, n_rows, S, s, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;

    if (!sampling) {
        TreeGreedyArgs g;
        g.tokens = tokens; g.parent = parent; g.p_argmax = ctx->p_argmax; g.B = B; g.N = N;
        g.n_accepted = n_accepted; g.path = path; g.next_token = next_token;
        e = launch_ex(verify_tree_greedy_kernel, static_cast<unsigned>((B + kPolicyThreads - 1) / kPolicyThreads),
                      kPolicyThreads, 0, 0, st, g);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        ctx->launches += 1;
        return SVIP_OK;
    }

    if (!q_stats) {
        StatsArgs d = s;
        d.logits = q_logits; d.row_stride = q_row_stride; d.out_stats = ctx->q_stats; d.out_argmax = nullptr;
        e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 1>, n_rows, S, d, st, kRingBytes)
                               : launch_clustered(row_stats_kernel<kF32, 1>, n_rows, S, d, st, kRingBytes);
        if (e != cudaSuccess) return cuda_fail(ctx, e);
        ctx->launches += 1;
    }

    TreeArgs t;
    t.tokens = tokens; t.parent = parent; t.q_logits = q_logits; t.q_row_stride = q_row_stride;
    t.q_stats = q_stats ? reinterpret_cast<const float2*>(q_stats) : ctx->q_stats;
    t.t_logits = target_logits; t.t_row_stride = t_row_stride; t.p_stats = ctx->p_stats;
    t.N = N; t.V = V; t.c = c; t.uniforms = uniforms; t.n_accepted = n_accepted; t.path = path;
    t.next_token = next_token; t.status = ctx->status;
    // the walk is a chain of passes over two rows: spread a sequence over as many blocks as the batch leaves room for
    int Sf = pick_cluster(ctx, B, V, dtype);
    if (ctx->cluster_override == 0) {
        const long row_bytes = static_cast<long>(V) * static_cast<long>(esz);
        while (Sf < kMaxCluster && 2 * row_bytes / Sf > (512L << 10)) Sf *= 2;
        if (Sf > kMaxCluster) Sf = kMaxCluster;
    }
    e = dtype == SVIP_BF16 ? launch_clustered(verify_tree_kernel<kBF16>, B, Sf, t, st, 0)
                           : launch_clustered(verify_tree_kernel<kF32>, B, Sf, t, st, 0);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_selftest_wait_timeout(svip_ctx* ctx, long wait_ns, void* stream) {
    if (!ctx || wait_ns < 1 || wait_ns > 100000000L) return SVIP_ERR_INVALID_ARG;
    cudaError_t e = launch_ex(wait_timeout_kernel, 1, 32, 0, 0, static_cast<cudaStream_t>(stream),
                              static_cast<unsigned long long>(wait_ns), ctx->status);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_policy_advance(svip_ctx* ctx, int policy, const uint8_t* stop, const int32_t* gamma,
                        int32_t* draft_len, uint8_t* active, int B, int K_cap, int32_t* n_active,
                        void* stream) {
    if (!ctx || !draft_len || !active || B < 0 || K_cap < 1) return SVIP_ERR_INVALID_ARG;
    if (policy != SVIP_POLICY_ENTROPY && policy != SVIP_POLICY_CONSTANT && policy != SVIP_POLICY_HEURISTIC)
        return SVIP_ERR_INVALID_ARG;
    if (policy == SVIP_POLICY_ENTROPY ? !stop : !gamma) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    AdvanceArgs a;
    a.policy = policy; a.stop = stop; a.gamma = gamma; a.draft_len = draft_len; a.active = active;
    a.B = B; a.K_cap = K_cap; a.n_active = n_active;
    a.loop.iter = nullptr; a.loop.max_iters = 0; a.loop.handle = 0;
    const bool decides = ctx->loop_open && n_active && n_active == ctx->loop_n_active &&
                         static_cast<cudaStream_t>(stream) == ctx->loop_stream;
    if (decides) a.loop = ctx->loop;
    a.arrived = nullptr;
    if (decides && join_draft_step(ctx, a)) {
        ctx->loop_decided = 1;      // no kernel of its own: nothing to count
        return SVIP_OK;
    }
    cudaError_t e = launch_ex(policy_advance_kernel, 1, kPolicyThreads, 0, 0, static_cast<cudaStream_t>(stream), a);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if (decides) ctx->loop_decided = 1;
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_policy_update(svip_ctx* ctx, int policy, const int32_t* n_accepted, int32_t* draft_len,
                       int32_t* gamma, uint8_t* active, int B, int K_cap, void* stream) {
    if (!ctx || !draft_len || !active || B < 0 || K_cap < 1) return SVIP_ERR_INVALID_ARG;
    if (policy != SVIP_POLICY_ENTROPY && policy != SVIP_POLICY_CONSTANT && policy != SVIP_POLICY_HEURISTIC)
        return SVIP_ERR_INVALID_ARG;
    if (policy == SVIP_POLICY_HEURISTIC && (!gamma || !n_accepted)) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    UpdateArgs a;
    a.policy = policy; a.n_accepted = n_accepted; a.draft_len = draft_len; a.gamma = gamma; a.active = active;
    a.B = B; a.K_cap = K_cap;
    cudaError_t e = launch_ex(policy_update_kernel, static_cast<unsigned>((B + kPolicyThreads - 1) / kPolicyThreads),
                              kPolicyThreads, 0, 0, static_cast<cudaStream_t>(stream), a);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_vp_partial(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V_shard, long row_stride,
                    float T, int vocab_offset, float* partial, void* stream) {
    if (!ctx || !logits || !partial) return SVIP_ERR_INVALID_ARG;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (B < 0 || V_shard < 1 || V_shard > 0x7fffffe0 || row_stride < 0 || vocab_offset < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T >= 0.f) || std::isinf(T)) return SVIP_ERR_INVALID_ARG;
    if (!aligned_to(logits, dtype == SVIP_BF16 ? 2 : 4) || !aligned_to(partial, 16)) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    SVIP_DEBUG_RANGES(ctx, static_cast<cudaStream_t>(stream), logits, rows_extent(B, row_stride, V_shard, dtype == SVIP_BF16 ? 2 : 4));
    StatsArgs s;
    s.logits = logits; s.row_stride = row_stride; s.V = V_shard; s.c = scale_for(T); s.draft_rows = 0; s.K = 1;
    s.cu = nullptr; s.q_seq_stride = 0; s.q_pos_stride = 0; s.out_stats = nullptr; s.out_argmax = nullptr;
    s.status = ctx->status; s.out_partial = reinterpret_cast<float4*>(partial); s.idx_offset = vocab_offset;
    const int S = pick_cluster(ctx, B, V_shard, dtype);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = dtype == SVIP_BF16 ? launch_clustered(row_stats_kernel<kBF16, 2>, B, S, s, st, kRingBytes)
                                       : launch_clustered(row_stats_kernel<kF32, 2>, B, S, s, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_vp_combine(svip_ctx* ctx, const float* partials, int G, int rank, int B, float T, float thresh,
                    const float* uniforms, float* entropy, uint8_t* stop, int32_t* token, int32_t* owner,
                    float* local_target, uint8_t* active, void* stream) {
    if (!ctx || !partials || !entropy || !stop || !token || !owner || !local_target || !active)
        return SVIP_ERR_INVALID_ARG;
    if (G < 1 || rank < 0 || rank >= G || B < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T >= 0.f) || std::isinf(T) || std::isnan(thresh) || (T > 0.f && !uniforms)) return SVIP_ERR_INVALID_ARG;
    if (!aligned_to(partials, 16)) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    VpCombineArgs a;
    a.partials = reinterpret_cast<const float4*>(partials); a.G = G; a.B = B; a.rank = rank; a.c = scale_for(T);
    a.thresh = thresh; a.greedy = T > 0.f ? 0 : 1; a.uniforms = uniforms; a.entropy = entropy; a.stop = stop;
    a.token = token; a.owner = owner; a.ext_target = local_target; a.active = active; a.status = ctx->status;
    cudaError_t e = launch_ex(vp_combine_kernel, static_cast<unsigned>((B + kPolicyThreads - 1) / kPolicyThreads),
                              kPolicyThreads, 0, 0, static_cast<cudaStream_t>(stream), a);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_vp_locate(svip_ctx* ctx, const void* logits, svip_dtype dtype, int B, int V_shard, long row_stride,
                   float T, const float* local_target, const uint8_t* active, int vocab_offset,
                   int32_t* token, void* stream) {
    if (!ctx || !logits || !local_target || !active || !token) return SVIP_ERR_INVALID_ARG;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (B < 0 || V_shard < 1 || V_shard > 0x7fffffe0 || row_stride < 0 || vocab_offset < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T > 0.f) || std::isinf(T)) return SVIP_ERR_INVALID_ARG;
    if (!aligned_to(logits, dtype == SVIP_BF16 ? 2 : 4)) return SVIP_ERR_INVALID_ARG;
    if (B == 0) return SVIP_OK;
    SVIP_DEBUG_RANGES(ctx, static_cast<cudaStream_t>(stream), logits, rows_extent(B, row_stride, V_shard, dtype == SVIP_BF16 ? 2 : 4));
    DraftArgs a;
    a.logits = logits; a.row_stride = row_stride; a.V = V_shard; a.c = scale_for(T); a.thresh = 0.f; a.greedy = 0;
    a.uniforms = nullptr; a.token = token; a.entropy = nullptr; a.stop = nullptr; a.row_stats = nullptr;
    a.status = ctx->status; a.active = active; a.ext_target = local_target; a.token_offset = vocab_offset;
    a.pos = nullptr; a.pos_stride = 0; a.slot_stride = 0; a.thr = nullptr; a.adv.arrived = nullptr;
    const int S = pick_draft_cluster(ctx, B, V_shard, dtype);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = dtype == SVIP_BF16 ? launch_clustered(draft_step_kernel<kBF16, false, 2>, B, S, a, st, kRingBytes)
                                       : launch_clustered(draft_step_kernel<kF32, false, 2>, B, S, a, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_pair_stats(svip_ctx* ctx, const void* q_logits, long q_row_stride, const void* target_logits,
                    long t_row_stride, svip_dtype dtype, int n_pairs, int V, float T, float c_bound,
                    float* out, void* stream) {
    return svip_pair_stats_given(ctx, q_logits, q_row_stride, nullptr, target_logits, t_row_stride, nullptr, dtype,
                                 n_pairs, V, T, c_bound, out, stream);
}

int svip_pair_stats_given(svip_ctx* ctx, const void* q_logits, long q_row_stride, const float* q_stats,
                          const void* target_logits, long t_row_stride, const float* p_stats, svip_dtype dtype,
                          int n_pairs, int V, float T, float c_bound, float* out, void* stream) {
    if (!ctx || !q_logits || !target_logits || !out) return SVIP_ERR_INVALID_ARG;
    if ((q_stats == nullptr) != (p_stats == nullptr)) return SVIP_ERR_INVALID_ARG;
    if (q_stats && (!aligned_to(q_stats, 8) || !aligned_to(p_stats, 8))) return SVIP_ERR_INVALID_ARG;
    const bool given = q_stats != nullptr;
    if (dtype != SVIP_F32 && dtype != SVIP_BF16) return SVIP_ERR_UNSUPPORTED;
    if (n_pairs < 0 || V < 1 || V > 0x7fffffe0 || q_row_stride < 0 || t_row_stride < 0) return SVIP_ERR_INVALID_ARG;
    if (!(T > 0.f) || std::isinf(T) || !(c_bound >= 0.f)) return SVIP_ERR_INVALID_ARG;
    const size_t esz = dtype == SVIP_BF16 ? 2 : 4;
    if (!aligned_to(target_logits, esz) || !aligned_to(q_logits, esz)) return SVIP_ERR_INVALID_ARG;
    if (n_pairs == 0) return SVIP_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SVIP_RANGE("svip_pair_stats");
    SVIP_DEBUG_RANGES(ctx, st, target_logits, rows_extent(n_pairs, t_row_stride, V, esz), q_logits,
                      rows_extent(n_pairs, q_row_stride, V, esz));
    // More pairs than fit at once: a block gets at most about 320 KB of the two rows, so that the pairs in flight stay
    // near the size of L2 for the second pass, but no pair more than 4 blocks (1024 pairs of 256000 fp32 logits 580 us with 2
    // blocks per pair, 476 with 4, 491 with 8; 512 pairs of 152064 bf16 88 us with 1, 83 with 2, 108 with 4; 1024 of
    // 50021 fp32 305 with 1, 263 with 2; short rows are best left whole: 32000 bf16 45 us with 1, 64 with 2).  Fewer
    // pairs: one wave.
    int S = pick_cluster(ctx, n_pairs, V, dtype);
    if (!given && ctx->cluster_override == 0 && n_pairs > 2 * ctx->num_sms) {
        const long pair_bytes = 2L * V * static_cast<long>(esz);
        S = 1;
        while (S < 4 && pair_bytes / S > (320L << 10)) S *= 2;
    }
    PairArgs p;
    p.t_logits = target_logits; p.t_row_stride = t_row_stride; p.q_logits = q_logits; p.q_row_stride = q_row_stride;
    p.V = V; p.c = scale_for(T); p.c_bound = c_bound; p.out = out; p.status = ctx->status;
    p.p_stats = reinterpret_cast<const float2*>(p_stats); p.q_stats = reinterpret_cast<const float2*>(q_stats);
    cudaError_t e;
    if (given)
        e = dtype == SVIP_BF16 ? launch_clustered(pair_stats_kernel<kBF16, true>, n_pairs, S, p, st, kRingBytes)
                               : launch_clustered(pair_stats_kernel<kF32, true>, n_pairs, S, p, st, kRingBytes);
    else
        e = dtype == SVIP_BF16 ? launch_clustered(pair_stats_kernel<kBF16>, n_pairs, S, p, st, kRingBytes)
                               : launch_clustered(pair_stats_kernel<kF32>, n_pairs, S, p, st, kRingBytes);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches += 1;
    return SVIP_OK;
}

int svip_graph_begin(svip_ctx* ctx, void* stream) {
    if (!ctx) return SVIP_ERR_INVALID_ARG;
    if (ctx->capturing) return SVIP_ERR_STATE;
    cudaError_t e = cudaSuccess;
    if (!ctx->loop_stream) {   // made now: no stream is created while a capture is open
        e = cudaStreamCreateWithFlags(&ctx->loop_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) { ctx->loop_stream = nullptr; return cuda_fail(ctx, e); }
    }
    e = cudaStreamBeginCapture(static_cast<cudaStream_t>(stream), cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->capturing = 1;
    return SVIP_OK;
}

int svip_graph_loop_begin(svip_ctx* ctx, void* stream, const int32_t* n_active, int max_iters, void** body_stream) {
    if (!ctx || !n_active || !body_stream || max_iters < 1) return SVIP_ERR_INVALID_ARG;
    if (!ctx->capturing || ctx->loop_open) return SVIP_ERR_STATE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // both counters start at zero at every replay, whatever the one before has left
    cudaError_t e = cudaMemsetAsync(ctx->loop_arrived, 0, kLoopStateBytes, st);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t n_deps = 0;
    e = cudaStreamGetCaptureInfo(st, &status, nullptr, &graph, &deps, &n_deps);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    if (status != cudaStreamCaptureStatusActive || !graph) return SVIP_ERR_STATE;
    // the body runs once before the first decision (the do-while of Algorithm 1): default value 1
    cudaGraphConditionalHandle handle;
    e = cudaGraphConditionalHandleCreate(&handle, graph, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    cudaGraphNodeParams params = {};
    params.type = cudaGraphNodeTypeConditional;
    params.conditional.handle = handle;
    params.conditional.type = cudaGraphCondTypeWhile;
    params.conditional.size = 1;
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddNode(&node, graph, deps, n_deps, &params);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    cudaGraph_t body = params.conditional.phGraph_out[0];
    // from here on the graph holds a loop: if its body cannot be recorded, svip_graph_end refuses
    // to hand the graph out (a loop without a deciding kernel would never end)
    // what is recorded on `stream` from here on comes after the loop
    e = cudaStreamUpdateCaptureDependencies(st, &node, 1, cudaStreamSetCaptureDependencies);
    if (e != cudaSuccess) { ctx->loop_failed = 1; return cuda_fail(ctx, e); }
    e = cudaStreamBeginCaptureToGraph(ctx->loop_stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) { ctx->loop_failed = 1; return cuda_fail(ctx, e); }
    ctx->loop.handle = handle;
    ctx->loop.iter = ctx->loop_iter;
    ctx->loop.max_iters = max_iters;
    ctx->loop_n_active = n_active;
    ctx->loop_open = 1;
    ctx->loop_decided = 0;
    ctx->loop_draft_node = nullptr;
    t_plain_launches = true;
    *body_stream = ctx->loop_stream;
    return SVIP_OK;
}

int svip_graph_loop_end(svip_ctx* ctx) {
    if (!ctx) return SVIP_ERR_INVALID_ARG;
    if (!ctx->loop_open) return SVIP_ERR_STATE;
    cudaError_t e = cudaSuccess;
    if (!ctx->loop_decided) {   // no svip_policy_advance on the loop's counter in the body: decide here
        e = launch_ex(loop_decide_kernel, 1, 32, 0, 0, ctx->loop_stream, ctx->loop, ctx->loop_n_active);
        if (e == cudaSuccess) ctx->launches += 1;
    }
    cudaGraph_t body = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(ctx->loop_stream, &body);
    ctx->loop_open = 0;
    t_plain_launches = false;
    if (e != cudaSuccess) { ctx->loop_failed = 1; return cuda_fail(ctx, e); }
    if (e2 != cudaSuccess) { ctx->loop_failed = 1; return cuda_fail(ctx, e2); }
    return SVIP_OK;
}

int svip_graph_end(svip_ctx* ctx, void* stream, svip_graph** graph) {
    if (!ctx || !graph) return SVIP_ERR_INVALID_ARG;
    if (!ctx->capturing) return SVIP_ERR_STATE;
    // a loop whose body was left open, or whose decision kernel could not be recorded, would
    // never end at replay: such a graph is not handed out
    bool broken = ctx->loop_failed != 0;
    if (ctx->loop_open) {
        cudaGraph_t body = nullptr;
        cudaStreamEndCapture(ctx->loop_stream, &body);
        ctx->loop_open = 0;
        t_plain_launches = false;
        broken = true;
    }
    ctx->loop_failed = 0;
    ctx->capturing = 0;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(static_cast<cudaStream_t>(stream), &g);
    if (broken) {
        if (g) cudaGraphDestroy(g);
        cudaGetLastError();
        return SVIP_ERR_STATE;
    }
    if (e != cudaSuccess || !g) return cuda_fail(ctx, e);
    cudaGraphExec_t ex = nullptr;
    e = cudaGraphInstantiate(&ex, g, 0);
    if (e != cudaSuccess) { cudaGraphDestroy(g); return cuda_fail(ctx, e); }
    svip_graph* out = new (std::nothrow) svip_graph();
    if (!out) { cudaGraphExecDestroy(ex); cudaGraphDestroy(g); return SVIP_ERR_CUDA; }
    out->exec = ex; out->graph = g;
    *graph = out;
    return SVIP_OK;
}

int svip_graph_launch(svip_graph* graph, void* stream) {
    if (!graph) return SVIP_ERR_INVALID_ARG;
#ifdef SVIP_DEBUG_BOUNDS
    if (debug_no_ranges(static_cast<cudaStream_t>(stream)) != cudaSuccess) return SVIP_ERR_CUDA;
#endif
    return cudaGraphLaunch(graph->exec, static_cast<cudaStream_t>(stream)) == cudaSuccess ? SVIP_OK : SVIP_ERR_CUDA;
}

int svip_graph_destroy(svip_graph* graph) {
    if (!graph) return SVIP_ERR_INVALID_ARG;
    cudaGraphExecDestroy(graph->exec);
    cudaGraphDestroy(graph->graph);
    delete graph;
    return SVIP_OK;
}

// ------------------------------------------------------------------ verify without allocation
//
// Workspace of svip_verify_noalloc: one fixed array in the library's device image instead of
// cudaMalloc'ed memory.  Layout: [p_stats | q_stats | p_argmax | status word].  Every call on a
// device reuses it, so calls that overlap on the GPU race (see include/svip.h).

namespace {

constexpr size_t kNoAllocRows = SVIP_NOALLOC_MAX_ROWS;
constexpr size_t kNoAllocStatsBytes = kNoAllocRows * sizeof(float2);
constexpr size_t kNoAllocBytes = 2 * kNoAllocStatsBytes + kNoAllocRows * sizeof(int32_t) + 256;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;

struct NoAllocDevice {
    int ready;
    int num_sms;
    unsigned char* base;   // device address of g_noalloc_scratch on this device
};
NoAllocDevice g_noalloc_dev[kNoAllocMaxDevices];
std::mutex g_noalloc_mutex;   // the per-device set-up may be reached from several host threads

// Once per device, with that device current: the host-side name g_noalloc_scratch is not a device
// address, so ask the runtime for the address the kernels must be given.
int noalloc_setup(int device, NoAllocDevice** out) {
    if (device < 0 || device >= kNoAllocMaxDevices) return SVIP_ERR_INVALID_ARG;
    NoAllocDevice* d = &g_noalloc_dev[device];
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!d->ready) {
        int current = -1;
        if (cudaGetDevice(&current) != cudaSuccess) { cudaGetLastError(); return SVIP_ERR_CUDA; }
        if (current != device) return SVIP_ERR_INVALID_ARG;
        int major = 0, sms = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
            cudaGetLastError();
            return SVIP_ERR_CUDA;
        }
        if (major != 10) return SVIP_ERR_UNSUPPORTED;
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return SVIP_ERR_CUDA;
        }
        const void* ringed[] = {
            (const void*)row_stats_kernel<kBF16, 0>, (const void*)row_stats_kernel<kBF16, 1>,
            (const void*)row_stats_kernel<kF32, 0>,  (const void*)row_stats_kernel<kF32, 1>,
            (const void*)verify_finish_kernel<kBF16>, (const void*)verify_finish_kernel<kF32>};
        for (const void* k : ringed)
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes) != cudaSuccess) {
                cudaGetLastError();
                return SVIP_ERR_CUDA;
            }
        d->num_sms = sms;
        d->base = static_cast<unsigned char*>(ptr);
        d->ready = 1;
    }
    *out = d;
    return SVIP_OK;
}

}  // namespace

int svip_verify_noalloc(int device, const int32_t* draft_tokens, const void* q_logits, long q_row_stride,
                        const float* q_stats, long q_seq_stride, long q_pos_stride,
                        const void* target_logits, long t_row_stride, svip_dtype dtype,
                        const int32_t* cu_rows, int B, int K, int n_target_rows, int V, float T,
                        const float* uniforms, int32_t* n_accepted, int32_t* next_token,
                        unsigned* status, void* stream) {
    if (n_target_rows > SVIP_NOALLOC_MAX_ROWS) return SVIP_ERR_WORKSPACE;
    NoAllocDevice* d = nullptr;
    int rc = noalloc_setup(device, &d);
    if (rc != SVIP_OK) return rc;
    // A context that lives on this call's stack and points into the fixed array; nothing is allocated.
    svip_ctx view = {};
    view.device = device;
    view.max_rows = SVIP_NOALLOC_MAX_ROWS;
    view.num_sms = d->num_sms;
    view.p_stats = reinterpret_cast<float2*>(d->base);
    view.q_stats = reinterpret_cast<float2*>(d->base + kNoAllocStatsBytes);
    view.p_argmax = reinterpret_cast<int32_t*>(d->base + 2 * kNoAllocStatsBytes);
    unsigned* own_status = reinterpret_cast<unsigned*>(d->base + 2 * kNoAllocStatsBytes +
                                                       kNoAllocRows * sizeof(int32_t));
    view.status = status ? status : own_status;
    // the status word must start at zero; everything else in the array is written before it is read
    if (cudaMemsetAsync(view.status, 0, sizeof(unsigned), static_cast<cudaStream_t>(stream)) != cudaSuccess) {
        cudaGetLastError();
        return SVIP_ERR_CUDA;
    }
    return svip_verify(&view, draft_tokens, q_logits, q_row_stride, q_stats, q_seq_stride, q_pos_stride,
                       target_logits, t_row_stride, dtype, cu_rows, B, K, n_target_rows, V, T, uniforms,
                       n_accepted, next_token, stream);
}

}  // extern "C"

