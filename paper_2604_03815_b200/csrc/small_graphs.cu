// Forward pass for small graphs in one kernel (Algorithm 1 lines 2-6): scores, selection, softmax and weighted sum of a
// (query, head) row by one warp, against the graph's keys in shared memory.
//
// On graphs of a few hundred nodes the filter of score_select_f16.cu saves nothing: its rescoring alone takes about 900
// instructions a row, and it needs seven launches.  Here a lane scores kU keys of a 256-key chunk (the same chains of
// fused multiply-adds in index order as every other kernel); the k-th largest of the 32 lane maxima is a lower bound of
// the row's k-th best score (k <= 32), so only the few scores that reach it are sorted, as (score, key) words.  Graphs of
// any size work, 256 keys at a time against the running list; small_graphs_preferred() has the line where the filter
// takes over.  Bound by instruction issue (about 1000 a row at n = 175, d = 16, k = 8; 0.72 of the issue slots).
// A block owns up to 8 * rows_per_warp consecutive rows of the batch and one head; rows of several graphs may meet in it.
#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"
#include "rowops.cuh"
#include "topk_buffer.cuh"

namespace kmip {

namespace {

constexpr int kWarps = 8;
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
                        for (int p0 = 0; p0 < cnt; p0 += 32) {
                            cand_t v[1] = {p0 + lane < cnt ? pend[p0 + lane] : 0ull};
                            warp_sort_desc<1>(v, lane);
                            const cand_t rev = __shfl_sync(FULL, v[0], 31 - lane);
                            cand_t m = cmax(lane < k ? best : 0ull, rev);
#pragma unroll
                            for (int j = 16; j > 0; j >>= 1) {
                                const cand_t o = __shfl_xor_sync(FULL, m, j);
                                m = ((lane & j) == 0) ? cmax(m, o) : cmin(m, o);
                            }
                            best = m;
                        }
                    }
                    if (lane >= k) best = 0ull;
                    if (!last_chunk) {
                        if (lane < k) list[lane] = best;
                        continue;
                    }
                    // softmax over the kept scores and the weighted sum of their V rows
                    int jj[1];
                    float p[1];
                    jj[0] = best ? cand_index(best) : -1;
                    const float sc = best ? cand_score(best) : -CUDART_INF_F;
                    const float mx = __shfl_sync(FULL, sc, 0);
                    p[0] = best ? __expf((sc - mx) * scale) : 0.0f;
                    const float z = warp_sum(p[0]);
                    p[0] *= z > 0.0f ? 1.0f / z : 0.0f;
                    if (lane < k) {
                        topk_idx[r * k + lane] = jj[0];
                        topk_score[r * k + lane] = sc;
                    }
                    if (drop_p > 0.0f) {
                        float f[1];
                        dropout_factors((long long)r, k, lane, drop_p, seed, f);
                        p[0] *= f[0];
                    }
                    gather_weighted_sum<T, D>(V, H, h, k, lane, jj, p, out + r * D);
                }
            }
            i0 = i1;
        }
    }
}

template <typename T, int D>
cudaError_t launch_d(const FwdArgs& a) {
    const long long rows = a.N * a.H;
    // one wave of rows per warp where they are few, eight rows per warp (and one load of the keys) where there are many
    const int rows_per_warp = (int)std::max<long long>(1, std::min<long long>(8, rows / ((long long)sm_count() * 4 * kWarps)));
    const size_t smem = (size_t)kChunk * row_stride<T, D>() + ((size_t)kWarps * rows_per_warp * 32 + (size_t)kWarps * kPend) * sizeof(cand_t);
    auto kern = small_forward_kernel<T, D>;
    if (smem > 48 * 1024) {  // what a kernel may have unasked
        cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err != cudaSuccess) return err;
    }
    const dim3 grid((unsigned)((a.N + kWarps * rows_per_warp - 1) / (kWarps * rows_per_warp)), (unsigned)std::min(a.H, 65535));
    return launch_next(a, kern, grid, kWarps * 32, smem, static_cast<const T*>(a.Q), static_cast<const T*>(a.K), static_cast<const T*>(a.V),
                                                a.graph_offsets, a.G, (int)a.N, a.H, a.k, rows_per_warp, 1.0f / sqrtf((float)a.d), a.drop_p,
                                                a.seed, static_cast<T*>(a.out), a.topk_idx, a.topk_score, reinterpret_cast<StatusBlock*>(a.ws));
}

template <typename T>
cudaError_t launch_t(const FwdArgs& a) {
    switch (a.d) {
        case 16: return launch_d<T, 16>(a);
        case 32: return launch_d<T, 32>(a);
        case 64: return launch_d<T, 64>(a);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Where one warp per row against all keys beats the filter (measured, us for the forward pass, here against the filter;
// fp32 below 1536 rows: against one warp per row reading the keys from global memory).
//   batches of small graphs  22 400 rows x 4 heads, n = 175, d 16, k 8: 139 / 249, k 24: 196 / 412; n = 156, d 64: 215 / 358;
//                            but n = 500, d 16, one head: 125 / 119
//   few rows                 one graph of 500: 33 / 61, 1024: 40 / 68, 2000: 60 / 83, 4000: 152 / 99; 2000 x 4 heads: 112 / 93
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
    return a.mode == KMIP_FP32_EXACT ? launch_t<float>(a) : launch_t<__nv_bfloat16>(a);
}

}  // namespace kmip
