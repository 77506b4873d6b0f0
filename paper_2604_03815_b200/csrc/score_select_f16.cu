// Half-precision prefilter sweep (Algorithm 1 lines 2-3): k <= 32, head widths 16, 32 and 64; k <= 103, widths 16 and 32; bf16 and fp32 storage.
//
// The paper lists half-precision arithmetic and tensor-core support as the engineering it left open
// (Sec. 6; closing remark of the FlashAttention comparison in the appendix).  The sweep of
// score_select_tc.cu is bound by the instructions that reduce the fp32 scores to group maxima, not by
// the tensor cores.  This kernel runs the same pipeline (TMA -> shared memory ring -> tcgen05.mma ->
// tensor memory -> selection warps, one thread per query row) with fp16 operands and fp16 accumulators:
// a selection thread pulls its 128 scores of a (key tile, query tile) pair out of tensor memory packed
// two to a register and reduces them with packed three-input maxima - half the registers and half the
// instructions per score.  What it computes is a FILTER, not the answer:
//   * Q and K are converted to fp16 after a power-of-two scaling per head that puts the largest row
//     norm into [32, 64) (f16_convert.cu), so nothing overflows and a bf16 value converts exactly except for
//     elements below 2^-14 of that;
//   * a candidate is a group of 8 keys - the even or the odd keys of a window of 16 consecutive keys,
//     which is what one packed register chain covers - ranked by the fp16 maximum of its scores;
//   * every row keeps at least k + slack of its best groups (select_rows below); whatever it drops has a
//     maximum at most the smallest one kept;
//   * refine_f16.cu rescoring decides: it computes the exact fp32 scores of the kept groups' keys, proves
//     from the error bound of the fp16 scores that no dropped group can hold one of the k best keys, and
//     sends the rare row for which it cannot to the exact CUDA-core kernel.
// The tensor cores round an fp16 accumulator to nearest after each 16-deep step (checked against the
// exact sums on the device); f16_filter.cuh has the bound.
//
// Pipeline.  Up to three 128-row query tiles per CTA (384 rows per work item, 12 selection warps), each with an accumulator
// buffer, an issuer warp and barriers of its own: independent pipelines that meet only at the key stages.  A selection warp
// hands its buffer back as soon as the scores are in registers and its issuer multiplies the next key tile while the
// warp reduces the current one.  The query tiles are the MMA's operand in tensor memory, beside the accumulators: each
// selection thread puts its row there once per work item.  From shared memory the two operands of a 128 x 128 tile take
// all of its bandwidth while the MMA runs (a load or barrier poll then waits 69 clocks instead of 29, 45 with the query
// tile in tensor memory), and the memory they took is room for the rows' lists.
//
// Selection.  A row's entries (fp16 maximum, group number) sit in one column of shared memory.  A group that beats the
// row's threshold is appended, nothing else; when a row runs out of room, all rows of the CTA raise their thresholds and
// drop what falls below, each lane for its own row (all together: a query tile that stalls alone stalls the others
// later, at the key stages).  Appending costs a few instructions, and the expected number of such rounds is the
// logarithm of the number of tiles (a row of random scores appends L per e-fold of keys seen).  Appending stores without a
// predicate and advances with one: a predicated store costs a warp 12 clocks, a plain one 5 (both sides of a tile's 16
// stores, one warp: 201 and 86 clocks).
//
// Measured (us, events around the launch; before: four query tiles from shared memory, three issuers that were one warp short,
// predicated appends, the ragged last tile masked inside the loop): 100k nodes, H 4, d 32, k 16 3450 -> 3050, k 30
// 4220 -> 3390; H 1, d 16, k 10 915 -> 770, k 45 1051 -> 898; 50k nodes, H 4, d 64, k 20 1348 -> 1061; point clouds, H 4, d 32,
// k 32, 200k nodes 12 180 -> 9300, 500k nodes 65 500 -> 53 000.  Where items of 512 rows just filled one wave and those of 384 do
// not, the whole forward pass is up to 6 % slower: 31 623 nodes, H 2, d 16, k 8 333 -> 351, 15 000, H 4, d 32 251 -> 265.  A round (one key tile, three query tiles, d 32) takes 546 clocks with thresholds
// that nothing beats, 384 of them MMA, and 920 where every tile has hits: three chains of load, maxima, append a
// scheduler, which fill 61 % of its issue slots.  What did not pay there (100k nodes, H 4, d 32, k 16, us, against 3060 in the
// same runs):
// four query tiles of 112 keys in 96 registers 3360, two tiles with two buffers each 4140, five of 80 keys 3760, six of 64
// keys 4010, the hits of a half tile kept aside and appended in batches 3670, one vote per half tile 3200, two key tiles per
// vote 3650, six key stages 3080.
//
// Persistent CTAs, head-major visiting order, the split tail of the schedule and the bounded waits are those of
// score_select_tc.cu.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "f16_filter.cuh"
#include "ptx.cuh"

#include <cuda_fp16.h>

namespace kmip {

namespace {

constexpr int BM = 128;  // query rows per tile = TMEM lanes
constexpr int BN = 128;  // keys per tile = accumulator columns
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int kRelaxedPollNs = 100;
constexpr uint32_t kTmemCols = 512;  // all of tensor memory: an accumulator buffer of BN columns per query tile, then the query tiles
// The service warps: the TMA producer and an issuer per query tile.
// The time from a buffer's release to the next commit is on every pipeline's critical path, so an issuer runs its loop
// as a whole warp (operands in uniform registers, an elected lane issues), has everything ready before it waits, and
// does nothing else.  With two query tiles on one of them its loop was as long as a round.
constexpr int kServiceWarps = 4, kIssuers = kServiceWarps - 1;
constexpr int threads16(int nqt) { return (4 * nqt + kServiceWarps) * 32; }

template <int D>
struct Shape16 {
    static_assert(D == 16 || D == 32 || D == 64, "head widths of the fp16 prefilter");
    static constexpr int RB = D * 2;                       // bytes per operand row = swizzle span
    static constexpr uint32_t LAYOUT = RB == 128 ? 2u : RB == 64 ? 4u : 6u;  // UMMA swizzle code (128 / 64 / 32 bytes)
    static constexpr int KSTEPS = D / 16;                  // one tcgen05.mma covers 16 halves of depth
    static constexpr int TILE_BYTES = 128 * RB;
};

// Shared-memory matrix descriptor of a K-major, swizzled operand whose 8-row groups are contiguous.
template <int D>
__device__ __forceinline__ uint64_t make_desc16(uint32_t saddr) {
    using Sh = Shape16<D>;
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((8 * Sh::RB) >> 4) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of sm_100
    d |= (uint64_t)Sh::LAYOUT << 61;
    return d;
}

// Instruction descriptor: fp16 accumulate (format 0), fp16 A and B (format 0), both K-major, M = 128, N = BN.
constexpr uint32_t kInstrDesc16 = ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

// CAP entries of 4 bytes per row: a warp's block of shared memory is slot-major (entry s of lane l at s * 128 + 4 l), so
// that no access conflicts.
template <int CAP, int NQT, int S>
struct Plan16 {
    static constexpr int WARP_BYTES = CAP * 128;
    static constexpr int NBARS = 1 + 2 * S + 3 * NQT;
};

struct Bars {
    uint32_t base;
    int S, NQT;
    __device__ uint32_t done() const { return base; }
    __device__ uint32_t k_full(int s) const { return base + 8 * (1 + s); }
    __device__ uint32_t k_empty(int s) const { return base + 8 * (1 + S + s); }
    __device__ uint32_t t_full(int qt) const { return base + 8 * (1 + 2 * S + qt); }
    __device__ uint32_t t_empty(int qt) const { return base + 8 * (1 + 2 * S + NQT + qt); }
    __device__ uint32_t q_full(int qt) const { return base + 8 * (1 + 2 * S + 2 * NQT + qt); }
};

template <int SLEEP_NS = 0>
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                              StatusBlock* sb, int who, long long limit) {
    if (ptx::mbar_wait_bounded<SLEEP_NS>(bar, parity, abort_flag, limit)) return true;
    record_status(sb, KMIP_ERR_TIMEOUT, who);
    return false;
}

// fp16 bits <-> 16-bit unsigned integers that order like the numbers (0 = empty list slot).
__device__ __forceinline__ uint32_t order16(uint32_t h) { return (h ^ ((h & 0x8000u) ? 0xFFFFu : 0x8000u)) & 0xFFFFu; }
__device__ __forceinline__ uint32_t unorder16(uint32_t x) { return (x ^ ((x & 0x8000u) ? 0x8000u : 0xFFFFu)) & 0xFFFFu; }
constexpr uint32_t kHalfNegInf2 = 0xFC00FC00u, kHalfPosInf2 = 0x7C007C00u;

constexpr uint32_t kEmptyEntry = 0x7FFF0000u;  // not a number: no comparison keeps it, no maximum returns it

// Groups of a graph are numbered 2 * (16-key window) + (odd keys); an entry holds the low 16 bits.  Graphs of more than
// 2^19 keys have 2^16 groups per segment: the high bits of a KEPT entry wait in the row's own list in global memory (one
// byte each), and rows are selected at every segment's end, so that all entries behind the kept ones are of the
// current segment.
constexpr int kSegTiles = (1 << 19) / BN;

constexpr int kDenseTiles = 16;  // a warp's appends are counted over this many tiles

struct RowSel16 {
    uint32_t pend;   // shared address of the row's next free entry
    uint32_t tau2;   // the row's threshold in both halves
    uint32_t n_old;  // entries that were there after the last selection (segmented graphs)
};

struct SelectTargets {
    int lo, hi;  // entries a row should be left with: at least lo, at most hi (all, where it has fewer)
};

// All lanes raise their rows' thresholds such that between lo and hi entries reach them, and drop the others.  The
// threshold of a row is searched between its smallest and its largest entry, counting packed halves in registers: three
// steps that interpolate (the entries above a threshold thin out exponentially), then bisection over the ordered 16-bit
// values.  Where many entries tie and no threshold leaves a number in range, the smallest tied ones past `hi` are
// dropped too.  `seg` >= 0: also keeps the high bytes at `hi_bytes` (the first n_old entries have one).
// Its instructions grow with CAP: a load, two extrema and up to 19 counts for every two entries.
// Out of line: the loop that calls it rarely keeps its registers.
template <int CAP>
__device__ __noinline__ RowSel16 select_rows(RowSel16 r, uint32_t base, SelectTargets t, bool raise, unsigned char* hi_bytes, int seg) {
    constexpr int NP = CAP / 2;
    static_assert(CAP % 8 == 0, "entries are moved eight at a time");
    const int cnt = (int)((r.pend - base) >> 7);
    const int maxcnt = __reduce_max_sync(FULL, cnt);
    uint32_t pk[NP];  // the maxima, two entries to a register
    uint32_t top = kHalfNegInf2, bot = kHalfPosInf2;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        uint32_t a = kEmptyEntry, b = kEmptyEntry;
        if (2 * i < cnt) a = ptx::lds_u32(base + (uint32_t)(2 * i) * 128u);
        if (2 * i + 1 < cnt) b = ptx::lds_u32(base + (uint32_t)(2 * i + 1) * 128u);
        pk[i] = __byte_perm(a, b, 0x7632);
        top = ptx::hmax2(top, pk[i]);
        bot = ptx::hmin2(bot, pk[i]);
    }
    auto value = [](uint32_t ordered) { return __half2float(__ushort_as_half((unsigned short)unorder16(ordered))); };
    // invariants of the search: c_lo > t.hi entries reach `lo`, c_hi < t.lo reach `hi`
    uint32_t lo = min(order16(bot & 0xFFFFu), order16(bot >> 16)), hi = max(order16(top & 0xFFFFu), order16(top >> 16)) + 1u;
    float c_lo = (float)cnt, c_hi = 0.0f;
    uint32_t thr = lo;
    const bool keep_all = cnt <= t.hi && !(raise && cnt >= t.lo);
    bool done = cnt <= t.hi, tie = false;  // a row with lo .. hi entries only raises its threshold to the smallest
    const float want = 0.5f * (float)(t.lo + t.hi);
#pragma unroll 1
    for (int step = 0; !__all_sync(FULL, done); ++step) {
        uint32_t mid = (lo + hi) >> 1;
        if (step < 3) {
            const float f = __logf(c_lo / want) / __logf(c_lo / fmaxf(c_hi, 0.7f));
            const float x = value(lo), g = x + f * (value(hi) - x);
            mid = min(max(order16(__half_as_ushort(__float2half_rn(g))), lo + 1u), hi - 1u);
        }
        const uint32_t h = unorder16(mid), h2 = h | (h << 16);
        uint32_t c2[4] = {0u, 0u, 0u, 0u};  // counts as packed fp16 numbers: exact up to 2048
#pragma unroll
        for (int i = 0; i < NP; ++i) c2[i & 3] = ptx::hadd2(c2[i & 3], ptx::hge2(pk[i], h2));
        const float c = ptx::half_sum(ptx::hadd2(ptx::hadd2(c2[0], c2[1]), ptx::hadd2(c2[2], c2[3])));
        if (!done) {
            if (c >= (float)t.lo && c <= (float)t.hi) { thr = mid; done = true; }
            else if (c > (float)t.hi) { lo = mid; c_lo = c; }
            else { hi = mid; c_hi = c; }
            if (!done && hi - lo <= 1u) { thr = lo; done = tie = true; }
        }
    }
    const uint32_t th = keep_all ? 0xFC00u : unorder16(thr), th2 = th | (th << 16);
    uint32_t out = base, off = 0u;
    if (seg < 0 && !__any_sync(FULL, tie)) {
#pragma unroll
        for (int i = 0; i < NP; i += 4) {
            if (2 * i < maxcnt) {  // warp-uniform
                uint32_t e[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) e[x] = ptx::lds_u32(base + (uint32_t)(2 * i + x) * 128u);
#pragma unroll
                for (int x = 0; x < 4; ++x)  // as in append_groups16; what lies at or behind `off` has been read
                    asm volatile(
                        "{\n\t"
                        ".reg .pred p, q;\n\t"
                        ".reg .b32 t, u;\n\t"
                        "setp.ge.f16x2 p|q, %1, %2;\n\t"
                        "add.u32 t, %0, %5;\n\t"
                        "@p add.u32 %0, %0, 128;\n\t"
                        "add.u32 u, %0, %5;\n\t"
                        "@q add.u32 %0, %0, 128;\n\t"
                        "st.shared.b32 [t], %3;\n\t"
                        "st.shared.b32 [u], %4;\n\t"
                        "}"
                        : "+r"(off)
                        : "r"(pk[i + x]), "r"(th2), "r"(e[2 * x]), "r"(e[2 * x + 1]), "r"(base)
                        : "memory");
            }
        }
        out = base + off;
    } else {
        // rare: ties, or a graph of several segments
        uint32_t c2 = 0u;
#pragma unroll
        for (int i = 0; i < NP; ++i) c2 = ptx::hadd2(c2, ptx::hgt2(pk[i], th2));
        int budget = tie ? t.hi - (int)ptx::half_sum(c2) : CAP;  // of entries equal to the threshold (zeros of either sign too)
        int n_new = 0;
#pragma unroll 1
        for (int s = 0; s < cnt; ++s) {
            const uint32_t e = ptx::lds_u32(base + (uint32_t)s * 128u);
            bool keep = ptx::half_ge(e >> 16, th);
            if (keep && ptx::half_ge(th, e >> 16) && budget-- <= 0) keep = false;
            if (keep) {
                ptx::sts_u32(out, e);
                if (seg >= 0) hi_bytes[n_new] = s < (int)r.n_old ? hi_bytes[s] : (unsigned char)seg;
                out += 128u;
                ++n_new;
            }
        }
        __syncwarp();
    }
    r.pend = out;
    r.n_old = (out - base) >> 7;
    if (!keep_all) r.tau2 = th2;
    return r;
}

// Columns at or past `nvalid` do not exist (end of the key range).
__device__ __forceinline__ void mask_ragged16(uint32_t (&v)[64], int nvalid) {
#pragma unroll
    for (int x = 0; x < 64; ++x) {
        if (2 * x >= nvalid) v[x] = kHalfNegInf2;
        else if (2 * x + 1 >= nvalid) v[x] = (v[x] & 0xFFFFu) | 0xFC000000u;
    }
}
// Packed maxima of a row's 128 scores: w[j] covers the 16-key window j (low half: its even keys, high half: its odd
// keys), m the tile.
__device__ __forceinline__ void tile_maxima16(const uint32_t (&v)[64], uint32_t (&w)[8], uint32_t& m) {
    uint32_t a[8], b[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int o = 8 * j;
        a[j] = ptx::hmax3(v[o], v[o + 1], v[o + 2]);
        b[j] = ptx::hmax3(v[o + 3], v[o + 4], v[o + 5]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = ptx::hmax3(v[8 * j + 6], v[8 * j + 7], a[j]);
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = ptx::hmax2(a[j], b[j]);
    m = ptx::hmax2(ptx::hmax3(ptx::hmax3(w[0], w[1], w[2]), w[3], w[4]), ptx::hmax3(w[5], w[6], w[7]));
}

// Appends the groups of a row's tile whose maximum beats tau (at most 16): per window one packed compare and two
// (4-byte store, pointer bump) pairs.  Every entry is stored where the next one goes, and stays if the pointer moves on:
// room for 16 is demanded before.  The addresses are copies, so that no bump waits for the store before it to have read
// its register (in place: 100k nodes, H 4, d 32, k 16 3330 us instead of 3060).  `id`: number of the tile's first group (its low 16
// bits count).
__device__ __forceinline__ void append_groups16(const uint32_t (&w)[8], uint32_t tau2, uint32_t id, uint32_t base, uint32_t& pend) {
    uint32_t ids = (id & 0xFFFFu) | ((id + 1u) << 16);  // of the even and the odd keys of a window
    uint32_t off = pend - base;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        asm volatile(
            "{\n\t"
            ".reg .pred p, q;\n\t"
            ".reg .b32 a, b, t, u;\n\t"
            "setp.gt.f16x2 p|q, %1, %2;\n\t"
            "prmt.b32 a, %3, %1, 0x5410;\n\t"
            "prmt.b32 b, %3, %1, 0x7632;\n\t"
            "add.u32 t, %0, %4;\n\t"
            "@p add.u32 %0, %0, 128;\n\t"
            "add.u32 u, %0, %4;\n\t"
            "@q add.u32 %0, %0, 128;\n\t"
            "st.shared.b32 [t], a;\n\t"
            "st.shared.b32 [u], b;\n\t"
            "}"
            : "+r"(off)
            : "r"(w[j]), "r"(tau2), "r"(ids + (uint32_t)j * 0x00020002u), "r"(base)
            : "memory");
    }
    pend = base + off;
}

template <int D, int CAP, int NQT, int S, bool DUMP>
__global__ void __launch_bounds__(threads16(NQT), 1)
score_select_f16_kernel(const __half* __restrict__ q16, const __grid_constant__ CUtensorMap tmK,
                        const WorkItem* __restrict__ items, StatusBlock* __restrict__ sb, int H,
                        const GroupLists lists, SelectTargets target, int item_tiles, float* __restrict__ dump, int n_total /* = N */, long long wait_limit, int drop_first_tile,
                        const int* __restrict__ perm) {
    using Sh = Shape16<D>;
    using Sp = Plan16<CAP, NQT, S>;
    constexpr int NEPI = 4 * NQT;
    constexpr uint32_t Q_COL = NQT * BN, Q_COLS = D / 2;  // the query tiles, two halves to a column
    static_assert(NQT <= kIssuers, "an issuer per query tile");
    static_assert(Q_COL + NQT * Q_COLS <= kTmemCols, "accumulators and query tiles in tensor memory");

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sK = smem;
    uint8_t* sRows = sK + S * Sh::TILE_BYTES;
    uint64_t* sBars = reinterpret_cast<uint64_t*>(sRows + NEPI * Sp::WARP_BYTES);
    uint32_t* sTmem = reinterpret_cast<uint32_t*>(sBars + Sp::NBARS);
    volatile int* sAbort = reinterpret_cast<volatile int*>(sTmem + 1);
    volatile int* sSelectReq = reinterpret_cast<volatile int*>(sTmem + 2);

    const int warp = __shfl_sync(FULL, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    Bars bars{ptx::smem_u32(sBars), S, NQT};

    if (threadIdx.x == 0) {
        ptx::mbar_init(bars.done(), NQT);
        for (int s = 0; s < S; ++s) {
            ptx::mbar_init(bars.k_full(s), 1);
            ptx::mbar_init(bars.k_empty(s), NQT);
        }
        for (int q = 0; q < NQT; ++q) {
            ptx::mbar_init(bars.t_full(q), 1);
            ptx::mbar_init(bars.t_empty(q), 4);  // the four selection warps of the query tile
            ptx::mbar_init(bars.q_full(q), 4);
        }
        *sAbort = 0;
        *sSelectReq = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async();
    }
    if (warp == NEPI + 1) {
        ptx::tmem_alloc(ptx::smem_u32(sTmem), kTmemCols);
        ptx::tmem_relinquish();
    }
    if (warp == NEPI && lane == 0) ptx::prefetch_tensormap(&tmK);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(FULL, *sTmem, 0);

    const int n_items = sb->n_items;
    const long long total = (long long)n_items * H;
    // Tail of the persistent schedule: the units (work item, head) past the last full wave of CTAs are cut into pieces of
    // fewer query tiles, one CTA each, as far as the pieces fit one wave.
    long long n_whole = total, n_units = total;
    int pieces = 1, piece_rows = item_tiles * BM;
    if (!DUMP && total > (long long)gridDim.x) {
        const int left = (int)(total % gridDim.x);
        if (left > 0) {
            const int tiles = (item_tiles + min(item_tiles, (int)gridDim.x / left) - 1) / min(item_tiles, (int)gridDim.x / left);
            pieces = (item_tiles + tiles - 1) / tiles;
            piece_rows = tiles * BM;
            n_whole = total - left;
            n_units = n_whole + (long long)left * pieces;
        }
    }
    auto unit = [&](long long w, int& h, WorkItem& it) -> bool {
        long long base = w;
        int piece = -1;
        if (w >= n_whole && pieces > 1) { base = n_whole + (w - n_whole) / pieces; piece = (int)((w - n_whole) % pieces); }
        h = (int)(base / n_items);
        it = items[base % n_items];
        if (piece >= 0) { it.row0 += piece * piece_rows; it.nrows = min(piece_rows, it.nrows - piece * piece_rows); }
        return it.nrows > 0;
    };

    if (warp == NEPI) {
        // ------------------------------------------------------------------ TMA producer
        // Every work item begins with stage 0, so that the issuers' loops know the stage of a step at compile time.
        int ic = 0;
        uint32_t k_phase = 0u, loaded = 0u;  // bit s: parity of stage s, a tile was loaded into stage s
        bool ok = true;
        for (long long w = blockIdx.x; ok && w < n_units; w += gridDim.x) {
            int h;
            WorkItem it;
            if (!unit(w, h, it)) continue;
            const int ntiles = (it.key_hi - it.key_lo + BN - 1) / BN;
            int s = 0;
            for (int j = 0; j < ntiles; ++j) {
                ok = __all_sync(FULL, wait_or_abort<kRelaxedPollNs>(bars.k_empty(s), ((k_phase >> s) & 1u) ^ 1u, sAbort, sb, 2, wait_limit));
                if (!ok) break;
                k_phase ^= 1u << s;
                // failure-detection test option: CTA 0 never loads its first key tile
                if (!(drop_first_tile && blockIdx.x == 0 && ic == 0 && j == 0)) {
                    if (ptx::elect_one()) {
                        ptx::mbar_arrive_expect_tx(bars.k_full(s), Sh::TILE_BYTES);
                        ptx::tma_load_2d(ptx::smem_u32(sK + s * Sh::TILE_BYTES), &tmK, 0, h * n_total + it.key_lo + j * BN, bars.k_full(s));
                    }
                    loaded |= 1u << s;
                }
                __syncwarp();
                if (++s == S) s = 0;
            }
            ++ic;
        }
        if (!ok && lane == 0) {
            // give copies that are still in flight a bounded time to land before the CTA exits
            const long long t0 = clock64();
            for (int s = 0; s < S; ++s)
                if ((loaded >> s) & 1u)
                    while (!ptx::mbar_try_wait(bars.k_full(s), ((k_phase >> s) & 1u) ^ 1u) && clock64() - t0 < 40000000ll) {}
        }
        __syncwarp();
    } else if (warp > NEPI) {
        // ------------------------------------------------------------------ MMA issuers
        // Query tile qt is multiplied with every key tile into accumulator buffer qt, committed to a barrier of its own,
        // and its four selection warps hand the buffer back as soon as the scores are in their registers.  Every issuer
        // waits for every key tile (a parity wait is sound only on a barrier whose every phase the waiter observes).
        const int qt = warp - NEPI - 1;
        if (qt < NQT) {  // one without a query tile would not be waited for at the key stages: it stays out
            const uint64_t desc_k0 = make_desc16<D>(ptx::smem_u32(sK));
            const uint32_t d_tmem = tmem_base + (uint32_t)(qt * BN), q_tmem = tmem_base + Q_COL + (uint32_t)qt * Q_COLS;
            const uint32_t full_bar = bars.t_full(qt), empty_bar = bars.t_empty(qt);
            uint32_t k_phase = 0u, t_par = 1u;
            int ic = 0;
            bool ok = true;
            for (long long w = blockIdx.x; ok && w < n_units; w += gridDim.x) {
                int h_unused;
                WorkItem it;
                if (!unit(w, h_unused, it)) continue;
                ok = __all_sync(FULL, wait_or_abort<0>(bars.q_full(qt), ic & 1, sAbort, sb, 3, wait_limit));
                ptx::tc_fence_after();
                const int ntiles = (it.key_hi - it.key_lo + BN - 1) / BN;
                const bool active = qt * BM < it.nrows;
                for (int j0 = 0; ok && j0 < ntiles; j0 += S) {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        if (j0 + s >= ntiles) break;
                        const uint64_t desc_k = desc_k0 + (uint64_t)((s * Sh::TILE_BYTES) >> 4);
                        if (!__all_sync(FULL, ptx::mbar_try_wait(bars.k_full(s), (k_phase >> s) & 1u)))
                            ok = __all_sync(FULL, wait_or_abort<0>(bars.k_full(s), (k_phase >> s) & 1u, sAbort, sb, 4, wait_limit));
                        if (!ok) break;
                        if (!__all_sync(FULL, ptx::mbar_try_wait(empty_bar, t_par)))
                            ok = __all_sync(FULL, wait_or_abort<0>(empty_bar, t_par, sAbort, sb, 5, wait_limit));
                        if (!ok) break;
                        ptx::tc_fence_after();
                        if (ptx::elect_one()) {
                            if (active) {
#pragma unroll
                                for (int ks = 0; ks < Sh::KSTEPS; ++ks)  // 16 values of depth = 32 bytes of a key row, 8 columns of the query tile
                                    ptx::mma_f16_ts(d_tmem, q_tmem + 8u * ks, desc_k + (uint64_t)(2 * ks), kInstrDesc16, ks > 0 ? 1u : 0u);
                            }
                            ptx::mma_commit(full_bar);
                            // the scores of the tile before have been read, so its stage has been read too
                            if (s > 0) ptx::mbar_arrive(bars.k_empty(s > 0 ? s - 1 : 0));
                            else if (j0 > 0) ptx::mbar_arrive(bars.k_empty(S - 1));
                        }
                        __syncwarp();
                        k_phase ^= 1u << s;
                        t_par ^= 1u;
                    }
                }
                if (!ok) break;
                // the next item begins with stage 0, which may be the one that the last tile is in
                if (ntiles > 0 && ptx::elect_one()) ptx::mma_commit(bars.k_empty((ntiles - 1) % S));
                __syncwarp();
                ++ic;
            }
            if (ptx::elect_one()) {
                ptx::mma_commit(bars.done());
                const long long t0 = clock64();
                while (!ptx::mbar_try_wait(bars.done(), 0) && clock64() - t0 < 2000000000ll) {}
            }
            __syncwarp();
        }
    } else {
        // ------------------------------------------------------------------ selection warps
        const int qt = warp >> 2, quarter = warp & 3;
        const uint32_t row_base = ptx::smem_u32(sRows + (size_t)warp * Sp::WARP_BYTES) + 4u * lane;  // the row's first entry
        const uint32_t full_bar = bars.t_full(qt), empty_bar = bars.t_empty(qt);
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(qt * BN);
        const uint32_t select_req_s = ptx::smem_u32(const_cast<int*>(sSelectReq));
        RowSel16 rs;
        int select_seen = 0;
        int tcnt = 0;
        bool ok = true;
        for (long long w = blockIdx.x; ok && w < n_units; w += gridDim.x) {
            int h;
            WorkItem it;
            if (!unit(w, h, it)) continue;
            const bool active = qt * BM < it.nrows;
            const int local = qt * BM + quarter * 32 + lane;
            const bool rvalid = local < it.nrows;
            // the row's part of the query tile (every MMA of the item before is done: its last scores have been read)
            const uint4* q_row = reinterpret_cast<const uint4*>(q16 + ((size_t)(it.row0 + local) * H + h) * D);
#pragma unroll
            for (int ks = 0; ks < Sh::KSTEPS; ++ks) {
                uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
                if (rvalid) { a = q_row[2 * ks]; b = q_row[2 * ks + 1]; }
                ptx::tmem_st_32x8(tmem_base + ((uint32_t)(quarter * 32) << 16) + Q_COL + (uint32_t)qt * Q_COLS + 8u * ks, a, b);
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bars.q_full(qt));
            // the row's place in the list arrays: sweep order in, the row's own place out
            long long list_row = 0;
            if (!DUMP && rvalid) {
                const int srow = it.row0 + local;
                const int orow = perm ? __ldg(perm + srow) : srow;
                // checks builds: a row of the batch (a row that fails keeps to row 0's slots of the scratch list)
                if (kmip_check(orow >= 0 && orow < n_total, sb, 103)) list_row = (long long)orow * H + h;
            }
            unsigned char* const list_word = lists.word + list_row * lists.word_pitch;
            rs.pend = row_base;
            rs.tau2 = rvalid ? kHalfNegInf2 : kHalfPosInf2;
            __syncwarp();
            const int ntiles = (it.key_hi - it.key_lo + BN - 1) / BN;
            if (DUMP || !active) {
                for (int j = 0; j < ntiles; ++j, ++tcnt) {
                    ok = wait_or_abort(full_bar, (uint32_t)tcnt & 1u, sAbort, sb, 6, wait_limit);
                    ok = __all_sync(FULL, ok);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (DUMP && active) {
                        const int key0 = it.key_lo + j * BN;
                        const int ncol = min(BN, it.key_hi - key0);
                        uint32_t v[64];
                        ptx::tmem_ld_32x128_pack16_sync(taddr, v);
                        if (rvalid) {
#pragma unroll
                            for (int x = 0; x < 64; ++x) {
                                float* o = dump + ((size_t)h * n_total + it.row0 + local) * n_total + key0 + 2 * x;
                                if (2 * x < ncol) o[0] = __half2float(__ushort_as_half((unsigned short)(v[x] & 0xFFFFu)));
                                if (2 * x + 1 < ncol) o[1] = __half2float(__ushort_as_half((unsigned short)(v[x] >> 16)));
                            }
                        }
                    }
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(empty_bar);
                }
            } else {
                const int n_keys = it.key_hi - it.key_lo;
                const bool segmented = ntiles > kSegTiles;
                rs.n_old = 0u;
                uint32_t par = (uint32_t)tcnt & 1u;
                // The scores of the next key tile in registers, the buffer back to its issuer; false: gave up.
                auto fetch = [&](uint32_t (&v)[64]) -> bool {
                    if (!__all_sync(FULL, ptx::mbar_try_wait(full_bar, par))) {
                        if (!__all_sync(FULL, wait_or_abort(full_bar, par, sAbort, sb, 6, wait_limit))) return false;
                    }
                    ptx::tc_fence_after();
                    ptx::tmem_ld_32x128_pack16_sync(taddr, v);
                    ptx::tc_fence_before();
                    __syncwarp();
                    ptx::mbar_arrive_if(empty_bar, lane == 0);
                    par ^= 1u;
                    return true;
                };
                // a part: the key tiles of a segment, or all of them
                for (int j = 0, seg = 0; ok && j < ntiles; ++seg) {
                    const int part_end = segmented ? min((seg + 1) * kSegTiles, ntiles) : ntiles;
                    // After an append: selects where a row may have no room for another tile, or another warp asked for it.
                    auto make_room = [&](int req) {
                        bool select = req != select_seen;
                        if (__any_sync(FULL, rs.pend > row_base + (uint32_t)(CAP - 16) * 128u)) {
                            select = true;
                            if (req == select_seen) {  // the whole CTA selects now: the pipelines stall together, not in turn
                                if (lane == 0) atomicAdd(const_cast<int*>(sSelectReq), 1);
                                ++select_seen;
                            }
                        }
                        if (select) {
                            rs = select_rows<CAP>(rs, row_base, target, true, list_word, segmented ? seg : -1);
                            select_seen = max(select_seen, req);
                        }
                    };
                    if constexpr (NQT == 2) {
                        // Dense phase, while nearly every tile has a hit in some row of the warp: the groups of tile j are
                        // appended, without asking, while tile j + 1 is reduced.  Two warps a scheduler wait for their own
                        // chains (31 623 nodes, d 16, k 10: 147 -> 133 us); three fill each other's gaps, and have no
                        // registers for it.
                        if (j < part_end - 2) {
                            uint32_t wa[8], wb[8], m;
                            {
                                uint32_t v[64];
                                ok = fetch(v);
                                if (ok) tile_maxima16(v, wa, m);
                            }
                            auto step = [&](const uint32_t (&wp)[8], uint32_t (&wn)[8]) -> bool {
                                uint32_t v[64];
                                if (!fetch(v)) return false;
                                const int req = (int)ptx::lds_u32(select_req_s);
                                append_groups16(wp, rs.tau2, (uint32_t)j * 16u, row_base, rs.pend);
                                tile_maxima16(v, wn, m);
                                ++j;
                                make_room(req);
                                return true;
                            };
                            uint32_t mark = rs.pend;
                            int check = j + kDenseTiles;
                            while (ok && j < part_end - 2) {  // the groups of tile j wait in wa
                                ok = step(wa, wb);
                                if (!ok) break;
                                if (j >= part_end - 2) {
#pragma unroll
                                    for (int x = 0; x < 8; ++x) wa[x] = wb[x];
                                    break;
                                }
                                ok = step(wb, wa);
                                if (j >= check) {
                                    const int grown = __reduce_add_sync(FULL, (int)(rs.pend - mark) >> 7);  // negative after a selection
                                    if (grown >= 0 && grown < kDenseTiles / 2) break;
                                    mark = rs.pend;
                                    check = j + kDenseTiles;
                                }
                            }
                            if (!ok) break;
                            append_groups16(wa, rs.tau2, (uint32_t)j * 16u, row_base, rs.pend);
                            ++j;
                            make_room(select_seen);
                        }
                    }
                    for (; j < part_end - 1; ++j) {
                        uint32_t v[64], wm[8], m;
                        ok = fetch(v);
                        if (!ok) break;
                        const int req = (int)ptx::lds_u32(select_req_s);
                        tile_maxima16(v, wm, m);
                        // some lane of the warp has a hit in this tile, or it is time to select
                        if (!ptx::warp_any_half_gt_or(m, rs.tau2, req != select_seen)) continue;
                        append_groups16(wm, rs.tau2, (uint32_t)j * 16u, row_base, rs.pend);
                        make_room(req);
                    }
                    if (!ok) break;
                    // the part's last tile, outside the loop: it may be ragged (the mask in the loop cost 18 % at d 16, taken or
                    // not), and the rows are selected after it; at the end a row keeps all that its list can hold
                    uint32_t v[64], wm[8], m;
                    ok = fetch(v);
                    if (!ok) break;
                    const bool last = j == ntiles - 1;
                    if (last && (n_keys & (BN - 1))) mask_ragged16(v, n_keys - j * BN);
                    tile_maxima16(v, wm, m);
                    append_groups16(wm, rs.tau2, (uint32_t)j * 16u, row_base, rs.pend);
                    const SelectTargets t = last ? SelectTargets{lists.slots - 2, lists.slots} : target;
                    rs = select_rows<CAP>(rs, row_base, t, !last, list_word, segmented ? seg : -1);
                    ++j;
                }
                tcnt += ntiles;
                if (ok && rvalid) {
                    // each lane stores its row's groups and maxima, two at a time (unsorted; an empty slot is marked by the
                    // half 0xFFFF and its group is not written)
                    unsigned char* const list_half = lists.half + list_row * lists.half_pitch;
                    const int cnt = (int)((rs.pend - row_base) >> 7);
                    // high bytes first: they lie where the words go, and word s only covers bytes 4 s and up
                    for (int s = (lists.slots - 1) & ~1; s >= 0; s -= 2) {
                        uint32_t e[2];
#pragma unroll
                        for (int x = 0; x < 2; ++x) e[x] = s + x < cnt ? ptx::lds_u32(row_base + (uint32_t)(s + x) * 128u) : 0xFFFF0000u;
                        *reinterpret_cast<uint32_t*>(list_half + 2 * s) = __byte_perm(e[0], e[1], 0x7632);
                        if (s >= cnt) continue;
                        if (lists.compact) {
                            *reinterpret_cast<uint32_t*>(list_word + 2 * s) = __byte_perm(e[0], e[1], 0x5410);
                        } else {
                            uint32_t word[2];
#pragma unroll
                            for (int x = 0; x < 2; ++x) {
                                uint32_t id = e[x] & 0xFFFFu;
                                if (segmented && s + x < cnt) id |= (uint32_t)list_word[s + x] << 16;
                                word[x] = ((uint32_t)it.key_lo + (id >> 1) * 16u) | (id << 31);
                            }
                            *reinterpret_cast<uint2*>(list_word + 4 * s) = make_uint2(word[0], word[1]);
                        }
                    }
                }
                __syncwarp();
            }
            if (!ok) break;
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == NEPI + 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------- host
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Tensor map over an fp16 matrix of `rows` rows of D elements; a box is 128 rows.
template <int D>
bool make_tensor_map16(CUtensorMap* tm, const void* base, int64_t rows) {
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)D, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)D * 2};
    const cuuint32_t box[2] = {(cuuint32_t)D, 128u};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUtensorMapSwizzle sw = D == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : D == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Entries a row is left with before the end: about as many as its list holds at the end (k + slack: fewer would send
// more rows to the exact kernel, more would be appended more often).  The width of the range saves search steps: lists filled
// to their last slot send fewer rows there (point cloud of 200k nodes, H 4, d 32, k 32: 0 instead of 7 of 800 000) but cost
// the sweep more than those rows do (us, sweep + rescoring: 12 605 + 2583 instead of 11 951 + 2666; 20 graphs of 3000, d 16,
// k 8: 111 + 172 instead of 99 + 170).
SelectTargets select_targets(int slots) { return {slots - 2, slots + 6}; }

template <int D, int CAP, int NQT, int S, bool DUMP>
cudaError_t launch_cfg(const FwdArgs& a, const FwdWorkspace& w, float* dump) {
    using Sh = Shape16<D>;
    using Sp = Plan16<CAP, NQT, S>;
    constexpr size_t smem_bytes = 1024 + (size_t)S * Sh::TILE_BYTES + (size_t)4 * NQT * Sp::WARP_BYTES +
                                  (size_t)Sp::NBARS * 8 + 64;
    static_assert(smem_bytes <= 232448, "shared memory budget of one CTA");
    CUtensorMap tmK;
    const F16Buffers buf = f16_buffers(a, w);
    if (!make_tensor_map16<D>(&tmK, buf.k16, a.N * a.H)) return cudaErrorInvalidValue;
    auto kern = score_select_f16_kernel<D, CAP, NQT, S, DUMP>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    if (err != cudaSuccess) return err;
    const long long max_total = (long long)w.max_items * a.H;
    const int grid = (int)std::min<long long>(sm_count(), max_total);
    kern<<<grid, threads16(NQT), smem_bytes, a.stream>>>(
        static_cast<const __half*>(buf.q16), tmK, reinterpret_cast<const WorkItem*>(a.ws + w.items_off), reinterpret_cast<StatusBlock*>(a.ws), a.H,
        buf.lists, select_targets(w.list), w.item_tiles, dump, (int)a.N, a.wait_limit_cycles > 0 ? a.wait_limit_cycles : kDefaultWaitLimitCycles, a.drop_first_tile,
        (w.reorder && !DUMP) ? reinterpret_cast<const int*>(a.ws + w.perm_off) : nullptr);
    return cudaGetLastError();
}

// Long lists, measured (us for the sweep, fp32-accumulate sweep / this one): 100k nodes, H 1, d 16, k 45 2098 / 1070, k 100
// 5513 / 1859; 50k nodes, H 2, d 32, k 64 1627 / 939, k 100 3946 / 1180.
// Query tiles per CTA, at most: a row needs room for a good number of groups beyond its list, or the CTA selects too often.
int most_query_tiles(int32_t d, int list) { return list > (d == 16 ? 80 : 64) ? 2 : 3; }

// The kernel for as many query tiles as the work items have; entries per row as far as shared memory goes.
template <int D>
cudaError_t launch_d(const FwdArgs& a, const FwdWorkspace& w) {
    if (w.item_tiles == 3) return launch_cfg<D, D == 64 ? 96 : 128, 3, 4, false>(a, w, nullptr);
    return launch_cfg<D, D == 64 ? 144 : 184, 2, 4, false>(a, w, nullptr);
}

}  // namespace

// Lists in the workspace (bf16 storage); a graph has at most 256 segments.
bool score_select_f16_supported(int64_t N, int32_t d, int32_t k) { return (d == 16 || d == 32) && k <= 32 && N <= 256ll * kSegTiles * BN; }
int score_select_f16_list(int32_t k) { return k <= 8 ? 16 : k <= 16 ? 24 : kF16List32; }

// Lists in the output arrays: a row's topk_idx and topk_score hold 2 k entries of two 16-bit numbers, so the groups are
// numbered inside their graph (up to 2^16 of 8 keys) and k + slack <= 2 k, which wants k >= 4.
// Beyond 32 the slack grows slower than k: far down the list the scores lie close together, but L / k of them fit into
// the error bound all the same.
int score_select_f16_list_in_outputs(int32_t k) {
    if (k > 32) return std::max(kF16List32, (k + k / 8 + 4 + 7) / 8 * 8);
    return std::min(2 * k, k <= 8 ? 16 : k <= 16 ? 24 : kF16List32);
}
bool score_select_f16_in_outputs_supported(int64_t N, int32_t H, int32_t d, int32_t k, int mode) {
    if (k < 4 || N > (1 << 19) || (d != 16 && d != 32 && d != 64)) return false;
    if (k > 32) return mode != KMIP_BF16_TC_PRUNED && d <= 32 && score_select_f16_list_in_outputs(k) <= kF16ListMost && N * H >= kF16MinRowsLong;
    return mode == KMIP_FP32_EXACT || (mode == KMIP_BF16_TC && d == 64);  // the smallest calls are the small-graph kernel's
}

// Query tiles per work item.  A round (one key tile against all query tiles of a CTA) is mostly the chain of one pipeline, so
// fewer tiles per item pay only where they fill idle SMs: the smallest number of rounds, weighted with their length,
// wins.  Measured, ns (18 816 keys, one work item per CTA, 1 / 2 / 3 tiles: d 16, k 8 550 605 717; d 32, k 16 613 661 766; d 64, k
// 16 618 669 780; longer lists d 32, k 32 743 773 939; d 16, k 45 744 827 1003; d 64, k 32 724 822 1094).  Graphs of one size are
// assumed.
int score_select_f16_item_tiles(int64_t N, int32_t G, int32_t H, int32_t d, int list) {
    const double kRound[4] = {0.0, list > 24 ? 0.74 : 0.79, list > 24 ? 0.8 : 0.86, 1.0};
    const int most = most_query_tiles(d, list);
    const int64_t grid = sm_count(), tiles = (N / std::max(G, 1) + BM - 1) / BM;  // query tiles of a graph
    int best = most;
    double best_cost = 0.0;
    for (int t = most; t >= 1; --t) {
        const int64_t units = (tiles + t - 1) / t * G * H, left = units % grid;
        double cost = (double)(units / grid) * kRound[t];
        if (left > 0) {
            const int64_t pieces = units > grid ? std::min<int64_t>(t, grid / left) : 1;  // the kernel cuts the tail
            cost += kRound[(t + pieces - 1) / pieces];
        }
        if (t == most || cost < best_cost) { best = t; best_cost = cost; }
    }
    return best;
}

cudaError_t launch_score_select_f16(const FwdArgs& a, const FwdWorkspace& w) {
    switch (a.d) {
        case 16: return launch_d<16>(a, w);
        case 32: return launch_d<32>(a, w);
        case 64: return launch_d<64>(a, w);
        default: return cudaErrorInvalidValue;
    }
}

// Test entry: the fp16 scores themselves (scaled as the converted operands are), dump[h][i][j], ld = N.
cudaError_t launch_score_dump_f16(const FwdArgs& a, const FwdWorkspace& w, float* dump) {
    return a.d == 16 ? launch_cfg<16, 64, 3, 4, true>(a, w, dump) : launch_cfg<32, 64, 3, 4, true>(a, w, dump);
}

}  // namespace kmip
