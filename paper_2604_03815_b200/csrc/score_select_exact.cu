// CUDA-core score + running top-k kernel (Algorithm 1 lines 2-3), one warp per (query, head).
//
// This is the KMIP_FP32_EXACT path: every score is d fused multiply-adds in fp32, in index
// order c = 0..d-1.  It also serves bf16 storage for (d, k) combinations the tensor-core
// kernel does not cover.  The N x N score matrix is never stored: each lane scores one key
// per step and the warp appends the survivors of the threshold test to the row's buffer.
#include <algorithm>

#include "common.cuh"
#include "topk_buffer.cuh"

namespace kmip {

namespace {

constexpr int kWarpsPerBlock = 8;

// Graph range of row i: binary search for the last offset <= i, skipping empty graphs.
__device__ inline void graph_range(const int32_t* offs, int G, int N, int i, int& lo, int& hi) {
    if (offs == nullptr) { lo = 0; hi = N; return; }
    int a = 0, b = G;  // invariant: offs[a] <= i, answer in [a, b)
    while (b - a > 1) {
        const int m = (a + b) >> 1;
        if (__ldg(offs + m) <= i) a = m; else b = m;
    }
    lo = max(0, min(N, __ldg(offs + a)));
    hi = max(lo, min(N, __ldg(offs + a + 1)));
}

template <typename T, int D, int E>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
score_select_exact_kernel(const T* __restrict__ Q, const T* __restrict__ K,
                          const int32_t* __restrict__ offs, int G, int N, int H, int k,
                          int32_t* __restrict__ topk_idx, float* __restrict__ topk_score,
                          const StatusBlock* __restrict__ sb) {
    if (sweep_off(sb)) return;  // the plan kernel rejected the offsets
    constexpr int CAP = 32 * E;
    constexpr int VEC = Elem<T>::kVec;
    __shared__ cand_t s_rows[kWarpsPerBlock][CAP];
    __shared__ float s_q[kWarpsPerBlock][D];

    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    cand_t* row = s_rows[wib];
    float* q = s_q[wib];
    const long long n_rows = (long long)N * H;
    const int room = CAP - k;  // pending slots

    for (long long r = (long long)blockIdx.x * kWarpsPerBlock + wib; r < n_rows;
         r += (long long)gridDim.x * kWarpsPerBlock) {
        const int i = (int)(r / H), h = (int)(r % H);
        int lo, hi;
        graph_range(offs, G, N, i, lo, hi);

        __syncwarp();
        for (int c = lane; c < D; c += 32) q[c] = Elem<T>::load(Q + ((size_t)i * H + h) * D + c);
        for (int t = lane; t < k; t += 32) row[t] = 0ull;
        __syncwarp();

        float tau = -CUDART_INF_F;
        int cnt = 0;
        for (int j0 = lo; j0 < hi; j0 += 32) {
            const int j = j0 + lane;
            const bool valid = j < hi;
            float s = 0.0f;
            if (valid) {
                const T* kr = K + ((size_t)j * H + h) * D;
#pragma unroll
                for (int c0 = 0; c0 < D; c0 += VEC) {
                    float kv[VEC];
                    Elem<T>::load_vec(kr + c0, kv);
#pragma unroll
                    for (int c = 0; c < VEC; ++c) s = fmaf(q[c0 + c], kv[c], s);
                }
            }
            const bool pass = valid && (s > tau);
            const unsigned m = __ballot_sync(0xFFFFFFFFu, pass);
            if (m) {
                if (pass) row[k + cnt + __popc(m & ((1u << lane) - 1u))] = make_cand(s, j);
                cnt += __popc(m);
                if (cnt > room - 32) {
                    tau = warp_compact_row<E>(row, k, cnt, lane);
                    cnt = 0;
                }
            }
        }
        warp_compact_row<E>(row, k, cnt, lane);
        warp_store_row(row, k, lane, topk_idx + (size_t)r * k, topk_score + (size_t)r * k);
    }
}

// The rows that the rescoring kernel of the half-precision prefilter listed, from all keys of their graph.  Their number
// is known on the device only, and it decides how the grid is shared out (block-uniform):
//   few rows    a listed row is one long scan over its graph (one row of a 500k-node graph took a single warp 15.7 ms,
//               a block of 16 warps 1.2 ms), so up to kRedoSplitMax rows are cut into parts, one block each, until the
//               grid is full: 0.10 ms.  The last block of a row to finish merges the parts' lists, which wait in
//               `scratch` (the call's `out` array: the softmax stage that writes it comes later);
//   more rows   a block per row;
//   many rows   (ties everywhere) a warp per row: no merging.
// Scores are the same chains of fused multiply-adds in index order as everywhere, and lists compare whole
// (score, key) words, so the result does not depend on how the keys were shared out.
constexpr int kRedoWarps = 8;
constexpr int kRedoBlocksPerSm = 4;

// Merges `n` lists of k keys (list l at src + l * stride) into the warp's sorted list row[0, k).  Only keys that beat the
// k-th best so far are taken, so most lists cost one pass of loads and no sorting.
template <int E>
__device__ __forceinline__ void merge_into_row(cand_t* row, int k, const cand_t* src, int n, size_t stride, int lane) {
    const int room = 32 * E - k;
    int cnt = 0;
    cand_t kth = row[k - 1];
    for (int l = 0; l < n; ++l) {
        for (int t0 = 0; t0 < k; t0 += 32) {
            const cand_t v = t0 + lane < k ? src[l * stride + t0 + lane] : 0ull;
            const bool pass = v > kth;
            const unsigned m = __ballot_sync(0xFFFFFFFFu, pass);
            if (!m) continue;
            if (pass) row[k + cnt + __popc(m & ((1u << lane) - 1u))] = v;
            cnt += __popc(m);
            if (cnt > room - 32) {
                compact_row_outlined<E>(row, k, cnt);
                kth = row[k - 1];
                cnt = 0;
            }
        }
    }
    compact_row_outlined<E>(row, k, cnt);
}

template <typename T, int D, int E>
__global__ void __launch_bounds__(kRedoWarps * 32)
score_select_redo_kernel(const T* __restrict__ Q, const T* __restrict__ K, const int32_t* __restrict__ offs, int G, int N, int H,
                         int k, int32_t* __restrict__ topk_idx, float* __restrict__ topk_score, StatusBlock* __restrict__ sb,
                         const int* __restrict__ redo_list, cand_t* scratch, long long scratch_lists, int limit) {
    if (sweep_off(sb)) return;
    const int n_rows = sb->n_redo;
    if (n_rows == 0 || n_rows > limit) return;  // too many: all rows are swept again (api.cu)
    constexpr int CAP = 32 * E, VEC = Elem<T>::kVec, U = 2;
    __shared__ cand_t s_rows[kRedoWarps][CAP];
    __shared__ float s_q[kRedoWarps][D];
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    cand_t* row = s_rows[wib];
    float* q = s_q[wib];
    const int room = CAP - k;
    const bool by_warp = n_rows > 2 * (int)gridDim.x;
    int parts = 1;
    if (n_rows <= kRedoSplitMax) parts = (int)max(1ll, min((long long)((int)gridDim.x / n_rows), scratch_lists / n_rows));
    const int first = by_warp ? (int)blockIdx.x * kRedoWarps + wib : (int)blockIdx.x;
    const int stride = by_warp ? (int)gridDim.x * kRedoWarps : (int)gridDim.x;
    const int n_units = n_rows * parts;  // parts > 1 only for few rows

    for (int x = first; x < n_units; x += stride) {
        const int li = x / parts, part = x % parts;
        const long long r = __ldg(redo_list + li);
        const int i = (int)(r / H), h = (int)(r % H);
        int lo, hi;
        graph_range(offs, G, N, i, lo, hi);
        __syncwarp();
        for (int c = lane; c < D; c += 32) q[c] = Elem<T>::load(Q + ((size_t)i * H + h) * D + c);
        for (int t = lane; t < k; t += 32) row[t] = 0ull;
        __syncwarp();
        const int step0 = by_warp ? 0 : part * kRedoWarps + wib, n_steps = by_warp ? 1 : parts * kRedoWarps;
        float tau = -CUDART_INF_F;
        int cnt = 0;
        for (long long j0 = lo + (long long)step0 * 32 * U; j0 < hi; j0 += (long long)n_steps * 32 * U) {
            float s[U];
#pragma unroll
            for (int u = 0; u < U; ++u) s[u] = 0.0f;
#pragma unroll
            for (int c0 = 0; c0 < D; c0 += VEC) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = (int)min(j0 + u * 32 + lane, (long long)hi - 1);
                    float kv[VEC];
                    Elem<T>::load_vec(K + ((size_t)j * H + h) * D + c0, kv);
#pragma unroll
                    for (int c = 0; c < VEC; ++c) s[u] = fmaf(q[c0 + c], kv[c], s[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long long j = j0 + u * 32 + lane;
                const bool pass = j < hi && s[u] > tau;
                const unsigned m = __ballot_sync(0xFFFFFFFFu, pass);
                if (m) {
                    if (pass) row[k + cnt + __popc(m & ((1u << lane) - 1u))] = make_cand(s[u], (int)j);
                    cnt += __popc(m);
                    if (cnt > room - 32) {
                        tau = compact_row_outlined<E>(row, k, cnt);
                        cnt = 0;
                    }
                }
            }
        }
        compact_row_outlined<E>(row, k, cnt);
        if (by_warp) {
            warp_store_row(row, k, lane, topk_idx + (size_t)r * k, topk_score + (size_t)r * k);
            continue;
        }
        auto merge_block = [&] {  // the block's lists, pairwise, into warp 0's
            for (int o = kRedoWarps / 2; o > 0; o >>= 1) {
                __syncthreads();
                if (wib < o) merge_into_row<E>(row, k, s_rows[wib + o], 1, 0, lane);
            }
            __syncwarp();
        };
        merge_block();
        if (parts > 1) {
            cand_t* mine = scratch + (size_t)x * k;
            if (wib == 0) {
                for (int t = lane; t < k; t += 32) mine[t] = row[t];
                __threadfence();
                __syncwarp();
                if (lane == 0) s_last = atomicAdd(&sb->redo_done[li], 1) == parts - 1;
            }
            __syncthreads();
            if (!s_last) continue;  // block-uniform
            __threadfence();
            for (int t = lane; t < k; t += 32) row[t] = 0ull;
            __syncwarp();
            // plain loads of what other blocks wrote before their counter moved; warp w takes every kRedoWarps-th part
            const int n_mine = (parts - wib + kRedoWarps - 1) / kRedoWarps;
            if (n_mine > 0)
                merge_into_row<E>(row, k, scratch + ((size_t)li * parts + wib) * k, n_mine, (size_t)kRedoWarps * k, lane);
            merge_block();
        }
        if (wib == 0) warp_store_row(row, k, lane, topk_idx + (size_t)r * k, topk_score + (size_t)r * k);
        __syncthreads();  // s_rows is rewritten by the next row
    }
}

template <typename T, int D>
cudaError_t launch_d(const FwdArgs& a) {
    const long long n_rows = (long long)a.N * a.H;
    const int blocks = (int)std::min<long long>((n_rows + kWarpsPerBlock - 1) / kWarpsPerBlock, (long long)sm_count() * (a.maybe_small ? 8 : 64));
    const T* Q = static_cast<const T*>(a.Q);
    const T* K = static_cast<const T*>(a.K);
    // pending room CAP-k must hold one 32-key step beyond the compaction trigger
#define KMIP_LAUNCH_EXACT(E_) \
    return launch_next(a, score_select_exact_kernel<T, D, E_>, dim3(blocks), kWarpsPerBlock * 32, 0, \
        Q, K, a.graph_offsets, a.G, (int)a.N, a.H, a.k, a.topk_idx, a.topk_score, \
        reinterpret_cast<const StatusBlock*>(a.ws))
    if (a.k <= 16) KMIP_LAUNCH_EXACT(2);
    else if (a.k <= 96) KMIP_LAUNCH_EXACT(4);
    else KMIP_LAUNCH_EXACT(8);
#undef KMIP_LAUNCH_EXACT
}

template <typename T>
cudaError_t launch_t(const FwdArgs& a) {
    switch (a.d) {
        case 16: return launch_d<T, 16>(a);
        case 32: return launch_d<T, 32>(a);
        case 64: return launch_d<T, 64>(a);
        case 128: return launch_d<T, 128>(a);
        default: return cudaErrorInvalidValue;
    }
}


template <typename T, int D>
cudaError_t launch_redo_d(const FwdArgs& a, const F16Buffers& b) {
    const int blocks = sm_count() * (a.maybe_small ? 1 : kRedoBlocksPerSm);
    const long long lists = b.scratch_words / a.k;
#define KMIP_LAUNCH_REDO(E_) \
    return launch_next(a, score_select_redo_kernel<T, D, E_>, dim3(blocks), kRedoWarps * 32, 0, \
        static_cast<const T*>(a.Q), static_cast<const T*>(a.K), a.graph_offsets, a.G, (int)a.N, a.H, a.k, \
        a.topk_idx, a.topk_score, reinterpret_cast<StatusBlock*>(a.ws), b.redo, static_cast<cand_t*>(b.scratch), lists, a.redo_limit)
    if (a.k <= 16) KMIP_LAUNCH_REDO(2);
    else if (a.k <= 96) KMIP_LAUNCH_REDO(4);
    else KMIP_LAUNCH_REDO(8);
#undef KMIP_LAUNCH_REDO
}

template <typename T>
cudaError_t launch_redo_t(const FwdArgs& a, const F16Buffers& b) {
    switch (a.d) {
        case 16: return launch_redo_d<T, 16>(a, b);
        case 32: return launch_redo_d<T, 32>(a, b);
        case 64: return launch_redo_d<T, 64>(a, b);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_score_select_exact(const FwdArgs& a) {
    return a.mode == KMIP_FP32_EXACT ? launch_t<float>(a) : launch_t<__nv_bfloat16>(a);
}

// The rows the half-precision prefilter could not decide, again from all keys of their graph; overwrites
// their topk_idx / topk_score.
cudaError_t launch_score_select_exact_redo(const FwdArgs& a, const FwdWorkspace& w) {
    const F16Buffers b = f16_buffers(a, w);
    return a.mode == KMIP_FP32_EXACT ? launch_redo_t<float>(a, b) : launch_redo_t<__nv_bfloat16>(a, b);
}

}  // namespace kmip
