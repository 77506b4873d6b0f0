// Softmax over the k kept scores fused with the gather-V weighted sum (Algorithm 1 lines 4-6).
// One warp per (query, head) row; the N x k x d tensor V_topk of line 4 is never materialised.
#include <algorithm>

#include "common.cuh"
#include "rowops.cuh"

namespace kmip {

namespace {

constexpr int kWarpsPerBlock = 8;

template <typename T, int D, int E, int W>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, W == 32 ? 0 : 8)
softmax_gather_kernel(const T* __restrict__ V, const int32_t* __restrict__ topk_idx,
                      const float* __restrict__ topk_score, int N, int H, int k, float scale,
                      float drop_p, unsigned long long seed, T* __restrict__ out,
                      const StatusBlock* __restrict__ sb) {
    if (sweep_off(sb)) return;  // an earlier stage failed: topk_idx was not written
    constexpr int kRows = 32 / W;  // rows of a warp
    const int lane = threadIdx.x % W, sub = (threadIdx.x & 31) / W;
    const unsigned n_rows = (unsigned)N * (unsigned)H, step = gridDim.x * kWarpsPerBlock * kRows;  // below 2^31
    unsigned r0 = (blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5)) * kRows;
    RowWalk walk(r0 + sub, step, H);
    for (; r0 < n_rows; r0 += step, walk.next()) {
        const bool live = r0 + sub < n_rows;
        const unsigned r = live ? r0 + sub : r0;  // a half without a row runs along with its neighbour's
        const int h0 = W == 32 ? walk.h : __shfl_sync(0xFFFFFFFFu, walk.h, 0), h = live ? walk.h : h0;
        int j[E];
        float p[E];
        load_row_softmax<E, W>(topk_idx + (size_t)r * k, topk_score + (size_t)r * k, k, N, scale, lane, j, p);
        if (drop_p > 0.0f) {  // training only: the weights go through dropout before the weighted sum
            float f[E];
            dropout_factors<E, W>(r, k, lane, drop_p, seed, f);
#pragma unroll
            for (int e = 0; e < E; ++e) p[e] *= f[e];
        }
        gather_weighted_sum<T, D, E, W>(V, H, h, k, lane, j, p, out + (size_t)r * D, live);
    }
}

template <typename T, int D>
cudaError_t launch_d(const FwdArgs& a) {
    const long long n_rows = (long long)a.N * a.H;
    const bool half = a.k <= kHalfWarp && half_warp_rows<T, D>();
    const long long warps = half ? (n_rows + 1) / 2 : n_rows;
    const int blocks = grid_blocks(a, (warps + kWarpsPerBlock - 1) / kWarpsPerBlock, 8);
    auto kern = a.k <= 32 ? softmax_gather_kernel<T, D, 1, 32> : a.k <= 64 ? softmax_gather_kernel<T, D, 2, 32> : softmax_gather_kernel<T, D, kMaxEntriesPerLane, 32>;
    if constexpr (half_warp_rows<T, D>()) {
        if (half) kern = softmax_gather_kernel<T, D, 1, kHalfWarp>;
    }
    return launch_next(a, kern, dim3(blocks), kWarpsPerBlock * 32, 0,
        static_cast<const T*>(a.V), a.topk_idx, a.topk_score, (int)a.N, a.H, a.k,
        1.0f / sqrtf((float)a.d), a.drop_p, a.seed, static_cast<T*>(a.out), reinterpret_cast<const StatusBlock*>(a.ws));
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

}  // namespace

cudaError_t launch_softmax_gather(const FwdArgs& a) {
    return a.mode == KMIP_FP32_EXACT ? launch_t<float>(a) : launch_t<__nv_bfloat16>(a);
}

}  // namespace kmip
