// Shared declarations of the k-MIP attention kernels (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kmip.h"
#include "kmip_test.h"

namespace kmip {

// ---------------------------------------------------------------------------------------------
// Workspace layout.  The first 256 bytes are the status block; everything else is carved by the
// host-side planners below with 256-byte alignment.
// ---------------------------------------------------------------------------------------------
constexpr size_t kStatusBytes = 256;
constexpr size_t kAlign = 256;

// -DKMIP_CHECKS builds (libkmip_checks.so) stand in for a memory checker: every workspace region is
// preceded by a 256-byte canary block that a tail kernel verifies, and the kernels test the indices they
// are about to follow.  A failed test RECORDS KMIP_ERR_CHECK in the status word and skips the access;
// nothing traps.  Release builds compile all of it away.
#ifdef KMIP_CHECKS
constexpr bool kChecks = true;
#else
constexpr bool kChecks = false;
#endif
constexpr size_t kCanaryBytes = kChecks ? 256 : 0;
constexpr uint32_t kCanaryWord = 0xC0DEFACEu;
constexpr int kMaxCanaries = 24;

// Offsets of the canary blocks of a workspace (checks builds; n = 0 otherwise).
struct Canaries {
    size_t off[kMaxCanaries];
    int n = 0;
};

constexpr int kRedoSplitMax = 48;

// Which kernels a forward call ran (StatusBlock::route; the values of kmip_test.h).
enum Route {
    kRouteSmall = KMIP_ROUTE_SMALL, kRouteFilter = KMIP_ROUTE_FILTER, kRouteTensorCore = KMIP_ROUTE_TENSOR_CORE,
    kRouteTiled = KMIP_ROUTE_TILED, kRouteRows = KMIP_ROUTE_ROWS
};

struct StatusBlock {
    int status;      // kmip_status_t recorded by the device (first error wins)
    int detail;      // where it happened (kernel-specific code)
    int n_items;     // forward: number of work items the plan kernel produced
    int n_long;      // backward: number of long key segments
    // pruned sweep: key tiles of all work items, tiles loaded (end-of-item markers included),
    // (key tile, query tile) pairs, pairs scored - summed over the CTAs (kmip_attn_sweep_counters)
    unsigned long long counters[4];
    int n_redo;      // forward, fp16 prefilter: rows the rescoring kernel sent to the exact kernel
    int redo_done[kRedoSplitMax];  // parts finished of each of the first redo rows (score_select_exact.cu)
    int route;       // forward: Route, written by the plan kernel (a lone small graph: by its own kernel)
    int reserved[50 - kRedoSplitMax];
};
static_assert(sizeof(StatusBlock) == kStatusBytes, "status block size");

// One unit of work of a sweep: up to 384 consecutive query rows of one
// graph and that graph's key range (Eq. 1 restricted to the graph by the CSR offsets).
struct WorkItem {
    int row0;    // first query row
    int nrows;   // 1..384 (128 x the query tiles per CTA of the launched configuration)
    int key_lo;  // graph's first row
    int key_hi;  // one past the graph's last row
    int tile0;   // number of the graph's first 128-key tile in the per-tile statistics (pruned sweep)
};

__host__ __device__ inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }

struct FwdWorkspace {
    size_t items_off;  // WorkItem[max_items]
    size_t kpack_off;  // [H, N, d], 2 bytes per element: K regrouped by head for the tensor-core sweeps (bf16, or
                       // scaled fp16 for the half-precision prefilter; 0 bytes without a tensor-core sweep)
    size_t qperm_off;  // [N, H, d], 2 bytes per element: Q in the sweep's row order (bf16, only when `reorder`;
                       // scaled fp16 whenever `f16`)
    size_t perm_off;   // int  [N]: original row of each sweep row
    size_t code_off;   // u16  [N]: locality codes of the query rows
    // pruned sweep only (all 0 bytes otherwise):
    size_t kperm_off;   // int   [N]: original key of each sweep position
    size_t kcode_off;   // u16   [N]: key codes (norm class, nearest pivot), by node
    size_t kcs_off;     // u16   [N]: the same in sweep order
    size_t knorm_off;   // float [N]: squared norm of the node's whole key vector
    size_t gmax_off;    // u32   [G]: bits of each graph's largest squared key norm
    size_t qnorm_off;   // float [N, H]: norm of each query row's head slice, in sweep order
    size_t qstat_off;   // float [max_items, 3, H, d+4]: centroid, radius, centroid norm of each item's 128-row query tiles
    size_t kstat_off;   // float [max_tiles, H, d+4]: centroid, radius, centroid norm, largest norm of each key tile
    // half-precision prefilter only (all 0 bytes otherwise):
    size_t f16stat_off;    // F16HeadStat [H]: per-head norm maxima
    size_t cand_word_off;  // u32 [N, H, list]: the groups each row kept (first key of the 16-key window, bit 31 = odd keys)
    size_t cand_half_off;  // u16 [N, H, list]: their fp16 maxima
    size_t redo_off;       // int [N * H]: (row, head) pairs the rescoring kernel hands to the exact kernel
    size_t total;
    int max_items;
    int max_tiles;
    int item_tiles;    // 128-row query tiles per work item of the half-precision prefilter (set where the plan is used:
                       // sizing a workspace makes no CUDA call)
    int list;          // groups kept per row by the half-precision prefilter
    bool tc;           // a tensor-core sweep runs (bf16 storage and a supported (d, k))
    bool f16;          // the half-precision prefilter runs (bf16: instead of that sweep; fp32: instead of the CUDA-core ones)
    bool in_outputs;   // ... with its lists, the redo list and the operand copies that have no place here in the call's
                       // output arrays, which nothing else uses until the last stages write them (f16_buffers)
    bool reorder;      // the sweep runs the rows of large graphs in locality order (reorder.cu)
    bool direct = false;  // set by plan_forward (api.cu): a fallback of the small-graph kernel with few launches
    bool prune;        // the sweep skips key tiles that cannot hold a candidate (prune.cu)
    Canaries canaries;
};

constexpr int64_t kReorderMinNodes = 32768;  // below this the extra launches cost more than they can save

bool score_select_tc_supported(int32_t d, int32_t k);
bool score_select_f16_supported(int64_t N, int32_t d, int32_t k);
bool score_select_f16_in_outputs_supported(int64_t N, int32_t H, int32_t d, int32_t k, int mode);
int score_select_f16_list(int32_t k);
int score_select_f16_list_in_outputs(int32_t k);
int score_select_f16_item_tiles(int64_t N, int32_t G, int32_t H, int32_t d, int list);

// Which sweep the plan is for: the one the mode selects, or one a test entry point asks for.
enum PlanVariant { kPlanByMode = 0, kPlanNoTensorCore = 1, kPlanTcFp32Acc = 2, kPlanTcFp16Acc = 3,
                   kPlanTcFp32AccInOrder = 4 /* fp32-accumulate sweep over the rows in their own order */ };

inline FwdWorkspace plan_fwd_workspace(int64_t N, int32_t G, int32_t H, int32_t d, int32_t k, int mode,
                                       int variant = kPlanByMode) {
    FwdWorkspace w;
    // start of the next region after one that ends at `end`; checks builds put a canary block in front of it
    auto region = [&w](size_t end) {
        const size_t c = align_up(end);
        if (kChecks && w.canaries.n < kMaxCanaries) w.canaries.off[w.canaries.n++] = c;
        return c + kCanaryBytes;
    };
    const int32_t g = G > 0 ? G : 1;
    w.tc = variant == kPlanByMode ? (mode != KMIP_FP32_EXACT && score_select_tc_supported(d, k))
                                  : variant != kPlanNoTensorCore;
    w.f16 = variant == kPlanByMode ? (w.tc && mode == KMIP_BF16_TC && score_select_f16_supported(N, d, k))
                                   : variant == kPlanTcFp16Acc;
    w.in_outputs = variant == kPlanByMode && !w.f16 && score_select_f16_in_outputs_supported(N, H, d, k, mode);
    w.f16 = w.f16 || w.in_outputs;
    w.list = w.in_outputs ? score_select_f16_list_in_outputs(k) : w.f16 ? score_select_f16_list(k) : 0;
    w.item_tiles = 0;
    w.max_items = (int)(N / 128 + g + 1);
    w.items_off = region(kStatusBytes);
    w.kpack_off = region(w.items_off + sizeof(WorkItem) * (size_t)w.max_items);
    w.reorder = w.tc && N >= kReorderMinNodes && variant != kPlanTcFp32AccInOrder;
    w.qperm_off = region(w.kpack_off + (w.tc ? (size_t)N * H * d * 2 : 0));
    w.perm_off = region(w.qperm_off + ((w.reorder || (w.f16 && !w.in_outputs)) ? (size_t)N * H * d * 2 : 0));
    w.code_off = region(w.perm_off + (w.reorder ? (size_t)N * 4 : 0));
    w.prune = variant == kPlanByMode && mode == KMIP_BF16_TC_PRUNED && w.reorder;
    w.max_tiles = (int)(N / 128 + g + 2);  // tile0 of a graph = floor(first row / 128) + graph index
    const size_t p = w.prune ? 1 : 0, rec = (size_t)(d + 4) * 4;
    w.kperm_off = region(w.code_off + (w.reorder ? (size_t)N * 2 : 0));
    w.kcode_off = region(w.kperm_off + p * (size_t)N * 4);
    w.kcs_off = region(w.kcode_off + p * (size_t)N * 2);
    w.knorm_off = region(w.kcs_off + p * (size_t)N * 2);
    w.gmax_off = region(w.knorm_off + p * (size_t)N * 4);
    w.qnorm_off = region(w.gmax_off + p * (size_t)g * 4);
    w.qstat_off = region(w.qnorm_off + p * (size_t)N * H * 4);
    w.kstat_off = region(w.qstat_off + p * (size_t)w.max_items * 3 * H * rec);
    const size_t f = w.f16 && !w.in_outputs ? 1 : 0, rows = (size_t)N * H;
    w.f16stat_off = region(w.kstat_off + p * (size_t)w.max_tiles * H * rec);
    w.cand_word_off = region(w.f16stat_off + (w.f16 ? 16 : 0) * (size_t)H);
    w.cand_half_off = region(w.cand_word_off + f * rows * w.list * 4);
    w.redo_off = region(w.cand_half_off + f * rows * w.list * 2);
    w.total = region(w.redo_off + f * rows * 4);  // checks builds: a last canary block behind the last region
    return w;
}

struct BwdWorkspace {
    size_t p_off;         // float [N*H*k]   softmax weights
    size_t ds_off;        // float [N*H*k]   score gradients
    size_t seg_off;       // int   [N*H+1]   start of each (key, head) hit list
    size_t cursor_off;    // int   [N*H]     hit counts, then fill cursors
    size_t pairs_off;     // int4  [N*H*k]   hit lists: records {query row, p, dS, (key, head) number}
    size_t tmp_off;       // int4  [N*H*k]   the other buffer of the radix passes that build them
    size_t table_off;     // int   [high digits][blocks]  digit counts per block of the first sorting step, then offsets
    size_t tblsum_off;    // int   block sums of the scan over that table
    size_t blocksum_off;  // int   [scan blocks]
    size_t long_off;      // int   [N*H]     ids of long segments
    size_t total;
    int scan_blocks;
    Canaries canaries;
};

constexpr int kScanItemsPerBlock = 4096;
// The hit lists are built by a stable two-step radix sort of the selected pairs by (key, head) number, so every
// list comes out ordered by query row whatever the timing.  First step: a block owns kRadixPerWarp consecutive
// pairs per warp and sorts them by the high digit in shared memory before it writes them out.
constexpr int kRadixPerWarp = 512;
constexpr int kRadixMaxBits = 12, kRadixMaxBins = 1 << kRadixMaxBits;
struct RadixPlan {
    int bits, lo_bits, hi_bits;  // of the numbers 0 .. rows (rows = "no key"): low and high digit
    bool sorted;                 // false: more than 2 * kRadixMaxBits bits or 2^31 pairs, unordered lists instead
    int warps;                   // per block of the first step
    long long blocks;            // blocks of the first step
    size_t bins_hi;
};
inline RadixPlan plan_radix(long long rows, long long pairs) {
    RadixPlan r;
    r.bits = 1;
    while ((1ll << r.bits) <= rows) ++r.bits;
    r.hi_bits = r.bits / 2 > 0 ? r.bits / 2 : 1;
    r.lo_bits = r.bits - r.hi_bits;
    r.sorted = r.bits <= 2 * kRadixMaxBits && pairs < (1ll << 31);
    r.warps = 8;
    const long long per_block = (long long)r.warps * kRadixPerWarp;
    r.blocks = r.sorted ? (pairs + per_block - 1) / per_block : 1;
    if (r.blocks < 1) r.blocks = 1;
    r.bins_hi = r.sorted ? ((size_t)1 << r.hi_bits) : 1;
    return r;
}

inline BwdWorkspace plan_bwd_workspace(int64_t N, int32_t H, int32_t k) {
    BwdWorkspace w;
    const size_t rows = (size_t)N * H, pairs = rows * (size_t)k;
    w.scan_blocks = (int)((rows + 1 + kScanItemsPerBlock - 1) / kScanItemsPerBlock);
    auto region = [&w](size_t end) {
        const size_t c = align_up(end);
        if (kChecks && w.canaries.n < kMaxCanaries) w.canaries.off[w.canaries.n++] = c;
        return c + kCanaryBytes;
    };
    size_t o = region(kStatusBytes);
    w.p_off = o;        o = region(o + 4 * pairs);
    w.ds_off = o;       o = region(o + 4 * pairs);
    w.seg_off = o;      o = region(o + 4 * (rows + 1));
    w.cursor_off = o;   o = region(o + 4 * (rows + 1));
    w.pairs_off = o;    o = region(o + 16 * pairs);
    w.tmp_off = o;      o = region(o + 16 * pairs);
    const RadixPlan rp = plan_radix((long long)rows, (long long)pairs);
    w.table_off = o;    o = region(o + 4 * rp.bins_hi * (size_t)rp.blocks);
    w.tblsum_off = o;   o = region(o + 4 * (rp.bins_hi * (size_t)rp.blocks / kScanItemsPerBlock + 2));
    w.blocksum_off = o; o = region(o + 4 * (size_t)(w.scan_blocks + 1));
    w.long_off = o;     o = region(o + 4 * rows);
    w.total = o;
    return w;
}

// ---------------------------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------------------------
__device__ inline void record_status(StatusBlock* sb, int status, int detail) {
    if (atomicCAS(&sb->status, 0, status) == 0) sb->detail = detail;
}
// Checks builds: `cond` must hold before an index is followed; if it does not, the failure is recorded with
// `code` (which test, see the call sites) and the caller skips the access.  Release builds: always true, no code.
__device__ __forceinline__ bool kmip_check(bool cond, StatusBlock* sb, int code) {
    if (!kChecks) return true;
    if (!cond) record_status(sb, KMIP_ERR_CHECK, code);
    return cond;
}

// First thing in the kernels of the sweeps' routes: true if the plan kernel gave the batch to the small-graph kernel, or if
// the call failed before.  The wait is for launches that overlap the end of the kernel before them (launch_next).
// The tensor-core sweeps may record a problem while blocks of theirs still start, so they don't ask for the second: they find
// no work items when the plan failed.  The half-precision one asks for neither and finds no work items in both cases; the wait
// at its head would make no difference (100k nodes, H 1, d 16, k 16 774 us without and with it, H 4, d 32, k 16 3047 and 3052).
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ bool small_route(const StatusBlock* sb) {
    wait_for_previous();
    return sb->route == kRouteSmall;
}
__device__ __forceinline__ bool sweep_off(const StatusBlock* sb) { return small_route(sb) || sb->status != KMIP_OK; }
// ... and, in those that serve as the second sweep (FwdArgs::min_redo), whether the filter decided enough rows.
__device__ __forceinline__ bool decided(const StatusBlock* sb, int min_redo) { return min_redo >= 0 && sb->n_redo <= min_redo; }

template <typename T> struct Elem;
template <> struct Elem<float> {
    static constexpr int kVec = 4;  // elements per 16-byte vector
    __device__ static inline float load(const float* p) { return __ldg(p); }
    __device__ static inline void store(float* p, float v) { *p = v; }
    __device__ static inline void load_vec(const float* p, float (&v)[4]) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    }
    __device__ static inline void store_vec(float* p, const float (&v)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct Elem<__nv_bfloat16> {
    static constexpr int kVec = 8;
    __device__ static inline float load(const __nv_bfloat16* p) {
        return __uint_as_float(((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p))) << 16);
    }
    __device__ static inline void store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
    __device__ static inline void load_vec(const __nv_bfloat16* p, float (&v)[8]) {
        const uint4 t = __ldg(reinterpret_cast<const uint4*>(p));
        const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
        }
    }
    __device__ static inline void store_vec(__nv_bfloat16* p, const float (&v)[8]) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// ---------------------------------------------------------------------------------------------
// Kernel launchers (defined in the .cu files; all asynchronous on `stream`)
// ---------------------------------------------------------------------------------------------
struct FwdArgs {
    const void *Q, *K, *V;
    const int32_t* graph_offsets;  // may be null
    int32_t G;
    int64_t N;
    int32_t H, d, k;
    int mode;
    void* out;
    int32_t* topk_idx;
    float* topk_score;
    unsigned char* ws;
    cudaStream_t stream;
    float drop_p = 0.0f;             // attention dropout on the k weights (0 = none)
    unsigned long long seed = 0ull;  // of its counter-based draws
    // per-call test options (kmip_test.h); the public entry points leave the defaults
    long long wait_limit_cycles = 0;  // bound of every device-side wait in SM clocks; <= 0: kDefaultWaitLimitCycles
    int drop_first_tile = 0;          // leave one key tile of CTA 0 unloaded, so that the waits on it run out
    bool maybe_small = false;         // the plan kernel decides between the small-graph kernel and the sweep's kernels
    int redo_limit = 0x7FFFFFFF;      // undecided rows that the exact pass takes; beyond, everything is swept again
    int min_redo = -1;                // >= 0: the kernels of that second sweep return unless more rows than this are undecided
    bool keys_in_place = false;       // the fp32-accumulate sweep and its rescoring read K as it lies, without a copy by head
    bool in_place = false;            // `out` overlaps Q or K: nothing may be written there before the last stage
    int fp32_path = 0;                // fp32 mode: 0 = sweep chosen by problem size, 1 = one warp per row, 2 = tiled
};

constexpr long long kDefaultWaitLimitCycles = 8000000000ll;  // about 4 s of SM clocks

struct BwdArgs {
    const void *Q, *K, *V, *d_out;
    int64_t N;
    int32_t H, d, k;
    int mode;
    const int32_t* topk_idx;
    const float* topk_score;
    void *dQ, *dK, *dV;
    unsigned char* ws;
    cudaStream_t stream;
    float drop_p = 0.0f;
    unsigned long long seed = 0ull;
};

// Launches a kernel that begins with sweep_off, small_route or wait_for_previous: it may start while the one before it ends.
// One that finds nothing to do then costs 1.3 us instead of 2.5.
// The shared memory that a kernel may ask for at a launch is set before, to the most that any call asks of it: it is state of
// the kernel, and a call in another host thread may set it between this one's setting and its launch.
template <typename... P, typename... A>
inline cudaError_t launch_next(const FwdArgs& a, void (*kern)(P...), dim3 grid, int threads, size_t smem, A&&... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = a.stream;
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &overlap;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}
// plan.cu, checks builds: write the canary blocks of a workspace / verify them (detail = 900 + block number)
cudaError_t launch_canary_fill(unsigned char* ws, const Canaries& c, cudaStream_t stream);
cudaError_t launch_canary_check(unsigned char* ws, const Canaries& c, cudaStream_t stream);
// plan.cu: clears the status block, validates the offsets and writes the work items of the sweep
enum SmallUse { kSmallNever = 0, kSmallAlways = 1, kSmallDecide = 2 };
cudaError_t launch_plan(const FwdArgs& a, const FwdWorkspace& w, int rows_per_item, int small_use, int route);
// plan.cu, after the exact pass: items of the second sweep (min_redo; route: kRouteTensorCore or kRouteTiled)
cudaError_t launch_resweep_plan(const FwdArgs& a, const FwdWorkspace& w, int rows_per_item, int route);
// plan.cu: K [N, H, d] -> [H, N, d] so that a head's key tile is one contiguous block for TMA
cudaError_t launch_pack_keys(const FwdArgs& a, const FwdWorkspace& w);
// reorder.cu: counters of the bucket sort (before launch_plan: they lie in an output array); locality codes, per-graph
// bucket sort, row-permuted copy of Q (after launch_plan)
cudaError_t launch_reorder_clear(const FwdArgs& a, const FwdWorkspace& w);
cudaError_t launch_reorder_queries(const FwdArgs& a, const FwdWorkspace& w);
// reorder.cu, pruned sweep: keys of large graphs sorted by (norm class, locality code) and regrouped by
// head in that order (replaces launch_pack_keys; after launch_reorder_queries, which owns the code buffer first)
cudaError_t launch_reorder_keys(const FwdArgs& a, const FwdWorkspace& w);
// prune.cu: centroid / radius / norm statistics of every item's query rows and of every key tile
cudaError_t launch_prune_stats(const FwdArgs& a, const FwdWorkspace& w);
constexpr int kMinRowsToSort = 8192;  // smaller graphs keep their row and key order
// Smallest N * H with 32 < k <= 103 that runs the half-precision prefilter (us for the forward pass, fp32-accumulate sweep / filter): 1024 rows, d 16, k 45:
// 165 / 113; d 32, k 80: 171 / 139; 10 000 rows, d 16, k 45: 348 / 218; smaller calls were not measured.
constexpr int64_t kF16MinRowsLong = 1024;
// score_select_exact.cu: CUDA-core scores + running top-k, any supported (d, k), fp32 or bf16 storage
cudaError_t launch_score_select_exact(const FwdArgs& a);
int sm_count();  // multiprocessors of the current device (cached per device)
// Blocks of a grid-stride kernel with `want` blocks of work, of which `per_sm` fit an SM.
inline int grid_blocks(const FwdArgs& a, long long want, int per_sm) {
    // a launch that may have nothing to do has no more blocks than fit the chip at once
    const long long most = (long long)sm_count() * (a.maybe_small || a.min_redo >= 0 ? per_sm : 32);
    return (int)(want < most ? want : most);
}
// score_select_tc.cu: tcgen05 scores + running top-k (bf16 storage); returns cudaErrorNotSupported
// when (d, k) is outside what the tensor-core kernel covers
int score_select_tc_rows_per_item(int32_t d, int32_t k);
cudaError_t launch_score_select_tc(const FwdArgs& a, const FwdWorkspace& w);
cudaError_t launch_score_dump_tc(const FwdArgs& a, const FwdWorkspace& w, float* dump);
// Half-precision prefilter (bf16 and fp32 storage; head widths 16, 32, 64 with k <= 32, 16 and 32 with k <= 103):
// f16_convert.cu (norm maxima, scaled fp16 copies of K and Q), score_select_f16.cu (sweep),
// refine_f16.cu (exact rescoring, redo list), score_select_exact.cu (the listed rows again, from all keys)

// The groups a row kept: `slots` entries per (node, head) row, the group and the fp16 maximum of its scores.
//   compact = 0  32-bit words (first key of the 16-key window, bit 31 = its odd keys)
//   compact = 1  16-bit numbers inside the graph: 2 * window + (odd keys)
struct GroupLists {
    unsigned char* word;
    unsigned char* half;
    long long word_pitch, half_pitch;  // bytes from row to row
    int slots, compact;
};
struct F16Buffers {
    void *k16, *q16;        // [H, N, d] and [N, H, d] (sweep order) fp16
    GroupLists lists;
    int* redo;              // [N * H]
    void* scratch;          // of the redo pass, 8-byte entries
    long long scratch_words;
};
inline F16Buffers f16_buffers(const FwdArgs& a, const FwdWorkspace& w) {
    const size_t rows = (size_t)a.N * a.H, copy = rows * a.d * 2, out_bytes = rows * a.d * (a.mode == KMIP_FP32_EXACT ? 4 : 2);
    unsigned char* out = static_cast<unsigned char*>(a.out);
    F16Buffers b;
    b.k16 = a.ws + w.kpack_off;
    b.q16 = a.ws + w.qperm_off;
    b.lists = {a.ws + w.cand_word_off, a.ws + w.cand_half_off, 4ll * w.list, 2ll * w.list, w.list, 0};
    b.redo = reinterpret_cast<int*>(a.ws + w.redo_off);
    size_t used = 0;  // bytes of `out` taken after the sweep
    if (w.in_outputs) {
        // until the sweep is done `out` holds the copies; then the redo list and the redo pass's scratch
        if (a.mode == KMIP_FP32_EXACT) { b.k16 = out; b.q16 = out + copy; }
        else if (!w.reorder) b.q16 = out;
        b.lists = {reinterpret_cast<unsigned char*>(a.topk_idx), reinterpret_cast<unsigned char*>(a.topk_score), 4ll * a.k, 4ll * a.k, w.list, 1};
        b.redo = reinterpret_cast<int*>(out);
        used = align_up(rows * 4, 16);
    }
    b.scratch = out + used;
    b.scratch_words = out_bytes > used && !a.in_place ? (long long)((out_bytes - used) / 8) : 0;
    return b;
}
cudaError_t launch_f16_convert(const FwdArgs& a, const FwdWorkspace& w);
cudaError_t launch_score_select_f16(const FwdArgs& a, const FwdWorkspace& w);
cudaError_t launch_score_dump_f16(const FwdArgs& a, const FwdWorkspace& w, float* dump);
cudaError_t launch_refine_f16(const FwdArgs& a, const FwdWorkspace& w);
cudaError_t launch_score_select_exact_redo(const FwdArgs& a, const FwdWorkspace& w);
// refine.cu: rescoring of the k best 8-key groups left by the tensor-core sweep -> final top-k
cudaError_t launch_refine_topk(const FwdArgs& a, const FwdWorkspace& w);
cudaError_t launch_refine_topk_fp32(const FwdArgs& a);
// topk_mass.cu: share of the full softmax held by the kept scores on CUDA cores (fp32 storage); needs 128-row
// work items in the workspace.  score_select_tc.cu: the same on the tensor cores (bf16 storage, every head width)
cudaError_t launch_topk_mass(const FwdArgs& a, const FwdWorkspace& w, float* mass);
cudaError_t launch_topk_mass_tc(const FwdArgs& a, const FwdWorkspace& w, float* mass);
// tiled CUDA-core sweep of fp32 mode (score_select_fp32.cu): 128-row work items, then launch_refine_topk_fp32
bool score_select_fp32_tiled_supported(int32_t d, int32_t k);
cudaError_t launch_score_select_fp32_tiled(const FwdArgs& a, const FwdWorkspace& w);
// small_graphs.cu: the whole forward pass of batches of small graphs (any graph size, k <= 32, d <= 64); after the plan
// kernel, which validates the offsets
int small_graphs_use(int64_t N, int32_t G, int32_t H, int32_t d, int32_t k);
// The rule, for `squares` = the sum of the squared graph sizes (the scores of a head); see small_graphs.cu
__host__ __device__ inline bool small_graphs_preferred(double squares, long long N, int H, int d, bool direct = false) {
    return squares * (d + 16) <= (direct && d > 16 ? 25000.0 : 15000.0) * (double)N || squares * H * (d + 16) <= 3.0e8;
}
cudaError_t launch_small_graphs(const FwdArgs& a);
// ... of one graph that fits its shared memory, without a plan kernel
bool one_graph_supported(int64_t N, int32_t G, int32_t H, int32_t d, int32_t k, int mode);
bool one_graph_preferred(int64_t N, int32_t H, int32_t d, int32_t k, int mode);
cudaError_t launch_one_graph(const FwdArgs& a);
// epilogue.cu: softmax over the k kept scores fused with the gather-V weighted sum
cudaError_t launch_softmax_gather(const FwdArgs& a);
// backward.cu
// ev (optional): three events recorded after the rows, inverse-index and segment stages
cudaError_t launch_backward(const BwdArgs& a, const BwdWorkspace& w, cudaEvent_t* ev);

// gemm_tn.cu: C_z = A_z B_z^T on the tensor cores (bf16 operands, fp32 accumulation); see there
struct GemmCall {
    const void *A[4], *B[4];
    void* C[4];
    int M, N, K, lda, ldb, ldc;
    bool a_mn = false, b_mn = false;  // stored [K, M] / [K, N] instead of [M, K] / [N, K]
    bool out_f32 = false;
    int n_batch = 1, n_kseg = 1, n_split = 1;
    const StatusBlock* merge_from = nullptr;  // a device-side problem recorded there is copied into the call's status block
};
cudaError_t launch_gemm(const GemmCall& g, StatusBlock* sb, cudaStream_t stream);
// parts of the K axis for a split launch whose partial sums have to fit `partial_bytes`
int gemm_splits(int M, int N, int K, int n_batch, size_t partial_bytes);
struct ReduceOut {
    void* dst[4];
    float scale[4];
    int transposed[4];
};
cudaError_t launch_reduce_partials(const float* partial, int n_split, int M, int N, int pad, int real, int n_batch, const ReduceOut& out,
                                   cudaStream_t stream);

// layer.cu: the full layer of Eq. 2 (bf16).  All pointers are device memory.
struct LayerArgs {
    const void *x, *w_q, *w_k, *w_v, *w_o;  // [N, d_model], [H*d_head, d_model] x 3, [d_model, H*d_head]
    void *q, *k_proj, *v, *o;               // [N, H, d_pad]: written by the forward pass, read by the backward pass
    int32_t* topk_idx;                      // [N, H, k]
    float* topk_score;                      // [N, H, k]
    void* y;                                // forward: [N, d_model]
    const void* d_y;                        // backward: upstream gradient [N, d_model]
    void *d_x, *dw_q, *dw_k, *dw_v, *dw_o;  // backward: gradients in the shapes of x and the weights
    const int32_t* graph_offsets;
    int32_t G;
    int64_t N;
    int32_t d_model, H, d_head, k;
    unsigned char* ws;
    cudaStream_t stream;
};
struct LayerWorkspace {
    size_t wq_pad, wk_pad, wv_pad, wo_pad;         // padded weights (unused when the head width needs no padding)
    size_t d_o, d_q, d_k, d_v;                     // [N, H*d_pad] gradients around the attention core
    size_t partial, partial_bytes;                 // fp32 partial sums of the weight gradients
    size_t attn, attn_bytes;                       // workspace of the attention call
    size_t total;
};
int layer_pad_width(int d_head);
LayerWorkspace plan_layer_workspace(int64_t N, int32_t G, int32_t d_model, int32_t H, int32_t d_head, int32_t k, int pass);
int layer_forward(const LayerArgs& a);   // kmip_status_t
int layer_backward(const LayerArgs& a);

}  // namespace kmip
