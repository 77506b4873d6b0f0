// Forward pass for small graphs in one kernel (Algorithm 1 lines 2-6): scores, selection, softmax and weighted sum.  Batches:
// a (query, head) row by one warp, against the graph's keys in shared memory; one graph: further down.
//
// On graphs of a few hundred nodes the filter of score_select_f16.cu saves nothing: its rescoring alone takes about 900
// instructions a row, and it needs seven launches.  Here a lane scores kU keys of a 256-key chunk (the same chains of
// fused multiply-adds in index order as every other kernel); the k-th largest of the 32 lane maxima is a lower bound of
// the row's k-th best score (k <= 32), so only the few scores that reach it are sorted, as (score, key) words.  Graphs of
// any size work, 256 keys at a time against the running list; small_graphs_preferred() has the line where the filter
// takes over.  Bound by instruction issue (about 1000 a row at n = 175, d = 16, k = 8; 0.72 of the issue slots).
// A block owns up to 8 * rows_per_warp consecutive rows of the batch and one head; rows of several graphs may meet in it.
#include <algorithm>
#include <cstddef>

#include "common.cuh"
#include "ptx.cuh"
#include "rowops.cuh"
#include "topk_buffer.cuh"

namespace kmip {

namespace {

constexpr int kWarps = 8;
constexpr int kMaxRowsPerWarp = 8;
constexpr int kU = 8;               // keys per lane and chunk
constexpr int kChunk = 32 * kU;     // keys per chunk
constexpr int kPend = kChunk + 32;  // candidates of a chunk
constexpr unsigned FULL = 0xFFFFFFFFu;

template <typename T, int D>
__host__ __device__ constexpr int row_stride() { return D * (int)sizeof(T) + 16; }  // an odd number of 16-byte units: a lane per row is conflict-free

// A query row in registers (bf16: two values to a register), and a key row in shared memory against it.
template <typename T, int D> struct RowDot;
template <int D> struct RowDot<__nv_bfloat16, D> {
    uint32_t q[D / 2];
    __device__ __forceinline__ void load(const __nv_bfloat16* p) {
#pragma unroll
        for (int v = 0; v < D / 8; ++v) {
            const uint4 t = __ldg(reinterpret_cast<const uint4*>(p + v * 8));
            q[v * 4] = t.x; q[v * 4 + 1] = t.y; q[v * 4 + 2] = t.z; q[v * 4 + 3] = t.w;
        }
    }
    __device__ __forceinline__ float dot(const unsigned char* kr) const {
        float s = 0.0f;
#pragma unroll
        for (int v = 0; v < D / 8; ++v) {
            const uint4 t = *reinterpret_cast<const uint4*>(kr + v * 16);
            const uint32_t kw[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) s = ptx::fma_bf16_pair(q[v * 4 + x], kw[x], s);
        }
        return s;
    }
};
template <int D> struct RowDot<float, D> {
    float q[D];
    __device__ __forceinline__ void load(const float* p) {
#pragma unroll
        for (int v = 0; v < D / 4; ++v) {
            const float4 t = __ldg(reinterpret_cast<const float4*>(p + v * 4));
            q[v * 4] = t.x; q[v * 4 + 1] = t.y; q[v * 4 + 2] = t.z; q[v * 4 + 3] = t.w;
        }
    }
    __device__ __forceinline__ float dot(const unsigned char* kr) const {
        float s = 0.0f;
#pragma unroll
        for (int v = 0; v < D / 4; ++v) {
            const float4 t = *reinterpret_cast<const float4*>(kr + v * 16);
            s = fmaf(q[v * 4], t.x, s);
            s = fmaf(q[v * 4 + 1], t.y, s);
            s = fmaf(q[v * 4 + 2], t.z, s);
            s = fmaf(q[v * 4 + 3], t.w, s);
        }
        return s;
    }
};

// `best` (sorted, a lane per entry, at most k) and up to 32 more candidates, unsorted: the best k of both.
__device__ __forceinline__ cand_t merge_sorted(cand_t best, cand_t more, int k, int lane) {
    cand_t v[1] = {more};
    warp_sort_desc<1>(v, lane);
    const cand_t rev = __shfl_sync(FULL, v[0], 31 - lane);
    cand_t m = cmax(lane < k ? best : 0ull, rev);
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const cand_t o = __shfl_xor_sync(FULL, m, j);
        m = ((lane & j) == 0) ? cmax(m, o) : cmin(m, o);
    }
    return m;
}

// The end of a row: softmax over the kept scores (`best`: sorted, one entry per lane, 0 = none) and the weighted sum of their
// V rows.
template <typename T, int D>
__device__ __forceinline__ void finish_row(cand_t best, const T* __restrict__ V, int H, int h, int k, int lane, size_t r, float scale,
                                           float drop_p, unsigned long long seed, T* __restrict__ out, int32_t* __restrict__ topk_idx,
                                           float* __restrict__ topk_score) {
    const float sc = best ? cand_score(best) : -CUDART_INF_F;
    if (lane < k) {
        topk_idx[r * k + lane] = best ? cand_index(best) : -1;
        topk_score[r * k + lane] = sc;
    }
    int jj[1] = {best ? cand_index(best) : -1};
    const float mx = __shfl_sync(FULL, sc, 0);
    float p[1] = {best ? __expf((sc - mx) * scale) : 0.0f};
    const float z = warp_sum(p[0]);
    p[0] *= z > 0.0f ? 1.0f / z : 0.0f;
    if (drop_p > 0.0f) {
        float f[1];
        dropout_factors((long long)r, k, lane, drop_p, seed, f);
        p[0] *= f[0];
    }
    // k > 16 known: half of the rounds go without a test (fp32, 22 400 rows, H 4, k 24: d 64 436 -> 391 us, d 16 211 -> 207;
    // bf16 has half as many rounds and gains nothing, d 32 loses 12 %)
    if (sizeof(T) == 4 && k > 16) gather_weighted_sum<T, D, 1, 32, 17>(V, H, h, k, lane, jj, p, out + r * D);
    else gather_weighted_sum<T, D>(V, H, h, k, lane, jj, p, out + r * D);
}

template <typename T, int D>
__global__ void __launch_bounds__(kWarps * 32)
small_forward_kernel(const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V, const int32_t* __restrict__ offs, int G,
                     int N, int H, int k, int rows_per_warp, float scale, float drop_p, unsigned long long seed, T* __restrict__ out,
                     int32_t* __restrict__ topk_idx, float* __restrict__ topk_score, StatusBlock* __restrict__ sb) {
    if (!small_route(sb) || sb->status != KMIP_OK) return;
    constexpr int P = D * (int)sizeof(T) / 16, kStride = row_stride<T, D>();
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char* sK = smem;                                          // [kChunk] padded key rows
    cand_t* sList = reinterpret_cast<cand_t*>(sK + kChunk * kStride);  // [rows of the block][32] running lists
    cand_t* sPend = sList + kWarps * rows_per_warp * 32;               // [kWarps][kPend]
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int rows = kWarps * rows_per_warp;
    const long long first = (long long)blockIdx.x * rows;
    const int row_lo = (int)first, row_hi = (int)min((long long)N, first + rows);
    cand_t* pend = sPend + wib * kPend;

    for (int h = blockIdx.y; h < H; h += gridDim.y) {
        int i0 = row_lo;
        while (i0 < row_hi) {  // one graph after the other; block-uniform
            int lo = 0, hi = N;
            if (offs != nullptr) {
                int a = 0, b = G;
                while (b - a > 1) {
                    const int m = (a + b) >> 1;
                    if (__ldg(offs + m) <= i0) a = m; else b = m;
                }
                lo = max(0, min(N, __ldg(offs + a)));
                hi = max(lo, min(N, __ldg(offs + a + 1)));
            }
            const int i1 = max(i0 + 1, min(hi, row_hi));  // rows [i0, i1) of the block belong to graph [lo, hi)
            for (int c0 = lo; c0 < hi || c0 == lo; c0 += kChunk) {
                const int nk = min(kChunk, hi - c0);
                __syncthreads();  // the chunk before has been read
                for (int x = threadIdx.x; x < nk * P; x += kWarps * 32) {
                    const int r = x / P, v = x % P;
                    ptx::cp_async_16(sK + r * kStride + v * 16,
                                     reinterpret_cast<const unsigned char*>(K + ((size_t)(c0 + r) * H + h) * D) + v * 16);
                }
                ptx::cp_async_commit();
                ptx::cp_async_wait<0>();
                __syncthreads();
                const bool first_chunk = c0 == lo, last_chunk = c0 + kChunk >= hi;
                for (int x = wib; x < i1 - i0; x += kWarps) {
                    const int i = i0 + x;
                    const size_t r = (size_t)i * H + h;
                    cand_t* list = sList + (size_t)(i - row_lo) * 32;
                    __syncwarp();
                    RowDot<T, D> q;
                    q.load(Q + r * D);
                    cand_t best = first_chunk || lane >= k ? 0ull : list[lane];  // sorted, one entry per lane
                    float s[kU];
                    float top = -CUDART_INF_F;
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        s[u] = -CUDART_INF_F;
                        if (u * 32 < nk) {  // warp-uniform
                            const float t = q.dot(sK + (u * 32 + lane) * kStride);
                            if (u * 32 + lane < nk) s[u] = t;
                            top = fmaxf(top, s[u]);
                        }
                    }
                    // k-th largest lane maximum
                    uint32_t w = order_bits(top);
#pragma unroll
                    for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
                        for (int j = kk >> 1; j > 0; j >>= 1) {
                            const uint32_t o = __shfl_xor_sync(FULL, w, j);
                            w = (((lane & j) == 0) == ((lane & kk) == 0)) ? max(w, o) : min(w, o);
                        }
                    }
                    const float bound = unorder_bits(__shfl_sync(FULL, w, k - 1));
                    // a later key with the score of the list's last entry loses to it, one with the bound's may be it;
                    // keys past the end have the score -infinity
                    const cand_t kth = __shfl_sync(FULL, best, k - 1);
                    const float tau = kth ? cand_score(kth) : -CUDART_INF_F;
                    int cnt = 0;
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        if (u * 32 < nk) {
                            // a score of -infinity (or a NaN) is nobody's choice, as in the other kernels
                            const bool pass = s[u] >= bound && s[u] > tau;
                            const unsigned m = __ballot_sync(FULL, pass);
                            if (m) {
                                if (pass) pend[cnt + __popc(m & ((1u << lane) - 1u))] = make_cand(s[u], c0 + u * 32 + lane);
                                cnt += __popc(m);
                            }
                        }
                    }
                    __syncwarp();
                    if (first_chunk && cnt <= 32) {
                        // the usual case: at most a warp of candidates, listed by key, so a candidate's place is the number
                        // of larger scores and of equal ones before it
                        const cand_t c = lane < cnt ? pend[lane] : 0ull;
                        const uint32_t mine = (uint32_t)(c >> 32);
                        int place = 0;
                        for (int j = 0; j < cnt; ++j) {
                            const uint32_t o = __shfl_sync(FULL, mine, j);
                            place += o > mine || (o == mine && j < lane) ? 1 : 0;
                        }
                        __syncwarp();
                        if (lane < cnt) pend[place] = c;
                        __syncwarp();
                        best = lane < cnt ? pend[lane] : 0ull;
                    } else {
                        for (int p0 = 0; p0 < cnt; p0 += 32) best = merge_sorted(best, p0 + lane < cnt ? pend[p0 + lane] : 0ull, k, lane);
                    }
                    if (lane >= k) best = 0ull;
                    if (!last_chunk) {
                        if (lane < k) list[lane] = best;
                        continue;
                    }
                    finish_row<T, D>(best, V, H, h, k, lane, r, scale, drop_p, seed, out, topk_idx, topk_score);
                }
            }
            i0 = i1;
        }
    }
}

// ------------------------------------------------------------------------------------------- one graph, few rows
// One graph of up to a few thousand nodes: too few rows to fill the chip with a warp each, so the latency of a row counts.
// A block of up to 32 warps owns R rows of a head.  A lane holds its key in registers, 64 bytes at a time, and the R query rows
// are broadcast from shared memory (a key row in shared memory would be read R times); the scores go to shared memory, WR warps
// select from a row's scores side by side, and their sorted lists are merged by rank.  Places in a list are counted with
// shuffles that do not wait for one another.  There is no plan kernel: a block checks the two offsets itself, and the first
// one writes the status block.
// Bound by latency: one pass over the phases, keys, scores, selection, V rows, in one wave of blocks.  Measured (us a call in a
// CUDA graph, a warp per row behind the plan kernel / this): fp32 H 1, d 16, k 10, 100 nodes 7.4 / 4.1, 256 7.8 / 5.1, 1024
// 19.0 / 10.2, 2048 36.5 / 17.4; d 32, k 16, 1024 22.3 / 13.3; d 64, k 20, 1024 30.0 / 19.2; bf16 H 4, d 16, k 10, 512 12.4 / 8.8,
// 1024 31.9 / 21.4.  Key rows read by a lane each (32 cache lines an instruction): d 32, 1024 15.5.
constexpr int kBlockWarps = 32;
constexpr size_t kMaxSmem = 227 * 1024;  // of a block

constexpr int kOneStageRow = 80, kOneStage = 32 * kOneStageRow;  // 64 bytes of a key row, padded: a lane per row is conflict-free
constexpr int kOnePend = 128;            // candidates of a warp before they are sorted
__host__ __device__ constexpr int one_graph_pitch(int N) { return (N + 31) / 32 * 32; }
__host__ __device__ constexpr size_t one_graph_smem(int N, int row_bytes, int R, int warps) {
    return (size_t)R * row_bytes + (size_t)(warps + R) * 32 * sizeof(cand_t) + (size_t)warps * kOneStage + (size_t)R * one_graph_pitch(N) * sizeof(float);
}

// Lanes' ranks by (value desc, lane asc).
__device__ __forceinline__ int lane_rank(uint32_t mine, int lane) {
    int place = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t o = __shfl_sync(FULL, mine, j);
        place += o > mine || (o == mine && j < lane) ? 1 : 0;
    }
    return place;
}

// A part of a key row (at most 64 bytes) in a lane's registers, and the chain of multiply-adds of a query row against it (index
// order, the same bits as every other kernel).
template <typename T, int D> struct KeyPart {
    static constexpr int kElems = D * (int)sizeof(T) < 64 ? D : 64 / (int)sizeof(T), kPieces = kElems * (int)sizeof(T) / 16;
    uint4 k[kPieces];
    __device__ __forceinline__ void load(const unsigned char* row) {
#pragma unroll
        for (int v = 0; v < kPieces; ++v) k[v] = *reinterpret_cast<const uint4*>(row + v * 16);
    }
    __device__ __forceinline__ float add(const T* q, float s) const {
#pragma unroll
        for (int v = 0; v < kPieces; ++v) {
            const uint4 t = *reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(q) + v * 16);
            const uint32_t a[4] = {t.x, t.y, t.z, t.w}, b[4] = {k[v].x, k[v].y, k[v].z, k[v].w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if constexpr (sizeof(T) == 4) s = fmaf(__uint_as_float(a[x]), __uint_as_float(b[x]), s);
                else s = ptx::fma_bf16_pair(a[x], b[x], s);
            }
        }
        return s;
    }
};

template <typename T, int D, int R, int WR>
__global__ void __launch_bounds__(R * WR * 32, kBlockWarps / (R * WR))
one_graph_forward_kernel(const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V, const int32_t* __restrict__ offs,
                         int N, int H, int k, float scale, float drop_p, unsigned long long seed, T* __restrict__ out,
                         int32_t* __restrict__ topk_idx, float* __restrict__ topk_score, StatusBlock* __restrict__ sb) {
    using Part = KeyPart<T, D>;
    static_assert(kOnePend * sizeof(cand_t) <= kOneStage, "candidates in the place of the key rows");
    static_assert(R * WR <= kBlockWarps && D % Part::kElems == 0, "warps of a block, whole parts per key");
    constexpr int P = D * (int)sizeof(T) / 16, threads = R * WR * 32;
    wait_for_previous();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, h = blockIdx.y, row0 = blockIdx.x * R;
    const bool bad = offs != nullptr && (__ldg(offs) != 0 || __ldg(offs + 1) != N);
    if (blockIdx.x == 0 && h == 0 && tid < (int)(kStatusBytes / 4)) {
        int v = 0;
        if (tid == (int)(offsetof(StatusBlock, status) / 4)) v = bad ? KMIP_ERR_BAD_OFFSETS : KMIP_OK;
        if (tid == (int)(offsetof(StatusBlock, detail) / 4)) v = bad ? 1 : 0;
        if (tid == (int)(offsetof(StatusBlock, route) / 4)) v = bad ? 0 : kRouteSmall;
        reinterpret_cast<int*>(sb)[tid] = v;
    }
    if (bad) return;

    extern __shared__ __align__(16) unsigned char smem[];
    T* sQ = reinterpret_cast<T*>(smem);                                      // [R][D]
    cand_t* sList = reinterpret_cast<cand_t*>(smem + R * D * sizeof(T));     // [warps][32]: each warp's best, sorted
    cand_t* sBest = sList + R * WR * 32;                                     // [R][32]: the rows' answers
    unsigned char* sStage = reinterpret_cast<unsigned char*>(sBest + R * 32);  // [warps] key rows, then candidates
    float* sScore = reinterpret_cast<float*>(sStage + R * WR * kOneStage);  // [R][pitch]
    const int pitch = one_graph_pitch(N);

    for (int x = tid; x < R * P; x += threads) {
        const int r = x / P, v = x % P, i = min(row0 + r, N - 1);
        reinterpret_cast<uint4*>(sQ)[x] = __ldg(reinterpret_cast<const uint4*>(Q + ((size_t)i * H + h) * D) + v);
    }
    for (int x = tid; x < R * 32; x += threads) sBest[x] = 0ull;
    __syncthreads();
    {
        // 32 keys a warp, part by part; the next part's copies (kPieces neighbouring lanes to a row, so that an instruction
        // touches few cache lines) run under the arithmetic of this one
        constexpr int kParts = D / Part::kElems, PP = Part::kPieces;
        unsigned char* stage = sStage + warp * kOneStage;
        auto fetch = [&](int j0, int c) {
            if (j0 < N) {
#pragma unroll
                for (int u = 0; u < PP; ++u) {
                    const int row = u * (32 / PP) + lane / PP, v = lane % PP;
                    ptx::cp_async_16(stage + row * kOneStageRow + v * 16,
                                     reinterpret_cast<const unsigned char*>(K + ((size_t)min(j0 + row, N - 1) * H + h) * D + c * Part::kElems) + v * 16);
                }
            }
            ptx::cp_async_commit();
        };
        int j0 = warp * 32;
        fetch(j0, 0);
        for (; j0 < N; j0 += threads) {
            float s[R];
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = 0.0f;
#pragma unroll
            for (int c = 0; c < kParts; ++c) {
                ptx::cp_async_wait<0>();
                __syncwarp();
                Part key;
                key.load(stage + lane * kOneStageRow);
                __syncwarp();
                if (c + 1 < kParts) fetch(j0, c + 1); else fetch(j0 + threads, 0);
#pragma unroll
                for (int r = 0; r < R; ++r) s[r] = key.add(sQ + r * D + c * Part::kElems, s[r]);
            }
            const int j = j0 + lane;
#pragma unroll
            for (int r = 0; r < R; ++r) sScore[r * pitch + j] = j < N ? s[r] : -CUDART_INF_F;
        }
        ptx::cp_async_wait<0>();
    }
    __syncthreads();

    // Warp `part` of row x selects from the row's scores 32 * part + lane, then 32 * WR further on, ...  The k-th largest of
    // its 32 lane maxima is a lower bound of its k-th best score, so only the few that reach it (about 32 ln 2 at k = 16, however
    // many there are) are sorted.
    const int x = warp / WR, part = warp % WR;
    const float* scores = sScore + x * pitch + lane;
    cand_t* pend = reinterpret_cast<cand_t*>(sStage + warp * kOneStage);
    cand_t best = 0ull;
    float top = -CUDART_INF_F;
#pragma unroll 4
    for (int c0 = part * 32; c0 < N; c0 += WR * 32) top = fmaxf(top, scores[c0]);
    const unsigned at = __ballot_sync(FULL, lane_rank(order_bits(top), lane) == k - 1);
    const float bound = __shfl_sync(FULL, top, __ffs(at) - 1);
    int cnt = 0;
    bool sorted = true;  // `best` holds nothing yet
#pragma unroll 4
    for (int c0 = part * 32; c0 < N; c0 += WR * 32) {
        const float s = scores[c0];
        // a score of -infinity (or a NaN) is nobody's choice, as in the other kernels
        const bool pass = s >= bound && s > -CUDART_INF_F;
        const unsigned m = __ballot_sync(FULL, pass);
        if (m) {
            if (cnt > kOnePend - 32) {  // ties
                __syncwarp();
                for (int p0 = 0; p0 < cnt; p0 += 32) best = merge_sorted(best, p0 + lane < cnt ? pend[p0 + lane] : 0ull, k, lane);
                __syncwarp();
                cnt = 0;
                sorted = false;
            }
            if (pass) pend[cnt + __popc(m & ((1u << lane) - 1u))] = make_cand(s, c0 + lane);
            cnt += __popc(m);
        }
    }
    __syncwarp();
    if (sorted && cnt <= 32) {
        // the usual case: at most a warp of candidates, listed by key, so a candidate's place is the number of larger
        // scores and of equal ones before it
        const cand_t c = lane < cnt ? pend[lane] : 0ull;
        const int place = lane_rank((uint32_t)(c >> 32), lane);
        __syncwarp();
        if (lane < cnt) pend[place] = c;
        __syncwarp();
        best = lane < cnt ? pend[lane] : 0ull;
    } else {
        for (int p0 = 0; p0 < cnt; p0 += 32) best = merge_sorted(best, p0 + lane < cnt ? pend[p0 + lane] : 0ull, k, lane);
    }
    if (lane >= k) best = 0ull;
    if constexpr (WR > 1) {
        // an entry's place in the row's answer: its place in its own list and the larger entries of the others
        sList[warp * 32 + lane] = best;
        __syncthreads();
        int place = lane;
#pragma unroll
        for (int o = 1; o < WR; ++o) {
            const cand_t* other = sList + (x * WR + (part + o) % WR) * 32;
            int n = 0;  // entries of `other` (descending) above `best`
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (other[n + step - 1] > best) n += step;
            if (n == 31 && other[31] > best) n = 32;
            place += n;
        }
        if (best && place < k) sBest[x * 32 + place] = best;
        __syncthreads();
    } else {
        sBest[x * 32 + lane] = best;
        __syncthreads();
    }
    // softmax over the kept scores and the weighted sum of their V rows
    const int i = row0 + warp;
    if (warp >= R || i >= N) return;
    best = sBest[warp * 32 + lane];
    const size_t r = (size_t)i * H + h;
    finish_row<T, D>(best, V, H, h, k, lane, r, scale, drop_p, seed, out, topk_idx, topk_score);
}

template <typename T, int D>
cudaError_t launch_d(const FwdArgs& a) {
    const long long rows = a.N * a.H;
    // one wave of rows per warp where they are few, eight rows per warp (and one load of the keys) where there are many
    const int rows_per_warp = (int)std::max<long long>(1, std::min<long long>(kMaxRowsPerWarp, rows / ((long long)sm_count() * 4 * kWarps)));
    auto bytes = [](int rows_each) { return (size_t)kChunk * row_stride<T, D>() + ((size_t)kWarps * rows_each * 32 + (size_t)kWarps * kPend) * sizeof(cand_t); };
    const size_t smem = bytes(rows_per_warp);
    auto kern = small_forward_kernel<T, D>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(kMaxRowsPerWarp));
    if (err != cudaSuccess) return err;
    const dim3 grid((unsigned)((a.N + kWarps * rows_per_warp - 1) / (kWarps * rows_per_warp)), (unsigned)std::min(a.H, 65535));
    return launch_next(a, kern, grid, kWarps * 32, smem, static_cast<const T*>(a.Q), static_cast<const T*>(a.K), static_cast<const T*>(a.V),
                                                a.graph_offsets, a.G, (int)a.N, a.H, a.k, rows_per_warp, 1.0f / sqrtf((float)a.d), a.drop_p,
                                                a.seed, static_cast<T*>(a.out), a.topk_idx, a.topk_score, reinterpret_cast<StatusBlock*>(a.ws));
}

template <typename T, int D, int R, int WR>
cudaError_t launch_one(const FwdArgs& a) {
    const size_t smem = one_graph_smem((int)a.N, D * (int)sizeof(T), R, R * WR);
    auto kern = one_graph_forward_kernel<T, D, R, WR>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (err != cudaSuccess) return err;
    return launch_next(a, kern, dim3((unsigned)((a.N + R - 1) / R), (unsigned)a.H), R * WR * 32, smem, static_cast<const T*>(a.Q),
                       static_cast<const T*>(a.K), static_cast<const T*>(a.V), a.graph_offsets, (int)a.N, a.H, a.k, 1.0f / sqrtf((float)a.d),
                       a.drop_p, a.seed, static_cast<T*>(a.out), a.topk_idx, a.topk_score, reinterpret_cast<StatusBlock*>(a.ws));
}

// Rows of a block and warps of a row: no more warps than there are keys for (100 nodes, d 16, H 1: 4.0 us with 8, 7.0 with
// 32); half as many rows per block where that still is one wave of blocks (512 nodes, H 4: 12.3 us in two waves, 9.6 in one).
struct OneGraphShape { int rows, warps; };
OneGraphShape one_graph_shape(int64_t N, int32_t H, int row_bytes) {
    if (N <= 256) return {8, 1};
    const bool few = ((N + 7) / 8) * H <= sm_count();
    if (few && N <= 512) return {8, 2};
    if (few || one_graph_smem((int)N, row_bytes, 16, 32) > kMaxSmem) return {8, 4};
    return {16, 2};
}

template <typename T, int D>
cudaError_t launch_shape(const FwdArgs& a, bool one_graph) {
    if (!one_graph) return launch_d<T, D>(a);
    const OneGraphShape s = one_graph_shape(a.N, a.H, D * (int)sizeof(T));
    if (s.rows == 16) return launch_one<T, D, 16, 2>(a);
    return s.warps == 1 ? launch_one<T, D, 8, 1>(a) : s.warps == 2 ? launch_one<T, D, 8, 2>(a) : launch_one<T, D, 8, 4>(a);
}

template <typename T>
cudaError_t launch_t(const FwdArgs& a, bool one_graph) {
    switch (a.d) {
        case 16: return launch_shape<T, 16>(a, one_graph);
        case 32: return launch_shape<T, 32>(a, one_graph);
        case 64: return launch_shape<T, 64>(a, one_graph);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Batches: where one warp per row against all keys beats the filter (measured, us for the forward pass, here against the
// filter).
//   batches of small graphs  22 400 rows x 4 heads, n = 175, d 16, k 8: 139 / 249, k 24: 196 / 412; n = 156, d 64: 215 / 358;
//                            but n = 500, d 16, one head: 125 / 119
// What it takes grows with the sum of the squared graph sizes, so n is that sum / N (one graph of 20 000 nodes among 255 of
// 60, 4 heads, d 16, has a mean size of 138: 5755 us here, 915 behind the filter).  The host knows the mean alone, which is
// never above n: where that decides nothing, the plan kernel applies the rule and both routes are launched.  Smaller batches
// then have the fp32-accumulate or the tiled sweep behind them (plan_forward, api.cu), which at d = 16 meet this kernel on
// the same line (100 graphs of 460: 120 / 124 us bf16, 131 / 153 fp32), wider heads later: 100 of 300, d 32 182 / 306 bf16
// and 254 / 409 fp32, 100 of 185, d 64 105 / 161 and 151 / 267.
int small_graphs_use(int64_t N, int32_t G, int32_t H, int32_t d, int32_t k) {
    if (k > 32 || d > 64) return kSmallNever;
    if (small_graphs_preferred((double)N * N, N, H, d)) return kSmallAlways;
    return small_graphs_preferred((double)N * N / std::max(G, 1), N, H, d) ? kSmallDecide : kSmallNever;
}

cudaError_t launch_small_graphs(const FwdArgs& a) {
    return a.mode == KMIP_FP32_EXACT ? launch_t<float>(a, false) : launch_t<__nv_bfloat16>(a, false);
}

// Where that beats what the call takes without it, the kernel for batches or the filter.  Its work grows with N^2 H d, the
// filter's mostly with its launches and its rows, and its blocks of up to 32 warps want to come in one wave: from the second
// on a warp per row fills the chip as well, without a block's barriers, unless key rows of 128 bytes and more are dear to
// read a row at a time.  From k = 30 on most of its time is selection (each warp keeps more candidates); fp32 has no filter below k = 4.  Measured (us, CUDA graph,
// here / batch kernel / filter), up to one wave: fp32 d 16 H 1 n 2048 17 / 36 / 47, d 32 H 1 1184 16 / 26 / 48; 1.2 to 5 waves:
// bf16 d 16 H 8 n 351 k 16 17 / 14 / 38, 702 31 / 28 / 44, k 32 51 / 38 / 56, H 4 n 1368 k 4 35 / 45 / 40, k 32 65 / 59 / 58; fp32
// d 32 H 32 n 360 k 16 52 / 60 / 83; d 64 H 1 n 2048 39 / 83 / 76; more: bf16 d 16 H 16 n 1104 k 16 94 / 112 / 67, H 64 n 398 k 16
// 91 / 69 / 85, d 32 H 64 n 624 k 4 165 / 154 / 92; fp32 d 64 H 32 n 360 k 24 81 / 98 / 175.  Geometric means of here /
// the better of the others, d 16 and 32, k 24 / 28 / 30 / 32: rows below 128 bytes, n > 1000, two waves 0.77 0.80 0.85 0.97,
// four 0.97 1.00 1.06 1.21; 512 nodes, two to four waves, k <= 28 1.06, 620 nodes 0.97; wider rows, three waves 0.81 0.83 0.86
// 0.95.  Of 2808 such sizes and k inside the first line, 95 % are within 5 % of the better side, the worst 1.3 times it; with
// that line alone 81 %, and with H up to 64 twice.
bool one_graph_preferred(int64_t N, int32_t H, int32_t d, int32_t k, int mode) {
    if ((double)N * N * H * (d + 32) > 4.2e8 + 3.0e4 * (double)N * H) return false;
    const bool fp32 = mode == KMIP_FP32_EXACT;
    if (N <= 256 || (d == 64 && (fp32 || k >= 8))) return true;
    const int row_bytes = d * (fp32 ? 4 : 2);
    const bool wide = row_bytes >= 128;
    const int waves = k >= 30 ? (wide ? 3 : N > 1000 ? 2 : 1) : wide || (fp32 && k < 4 && N > 440) ? 6 : N > 600 ? 4 : 1;
    const OneGraphShape s = one_graph_shape(N, H, row_bytes);
    return (N + s.rows - 1) / s.rows * H <= (int64_t)waves * sm_count();  // more than 256 nodes: a block per SM
}

bool one_graph_supported(int64_t N, int32_t G, int32_t H, int32_t d, int32_t k, int mode) {
    return G == 1 && k <= 32 && d <= 64 && H <= 65535 && N <= (1 << 16) &&
           one_graph_smem((int)N, d * (mode == KMIP_FP32_EXACT ? 4 : 2), 8, 32) <= kMaxSmem;
}

cudaError_t launch_one_graph(const FwdArgs& a) {
    return a.mode == KMIP_FP32_EXACT ? launch_t<float>(a, true) : launch_t<__nv_bfloat16>(a, true);
}

}  // namespace kmip
