// Warp-level building blocks for the gather stages (Algorithm 1 lines 4-6 and their backward):
// softmax over the k kept scores of one (query, head) row, and the weighted sum of gathered rows
// with 16-byte vector loads.
// The kernels made of them are bound by instruction issue more than by their gathers.  With sums by halves instead of
// butterflies, one entry per lane where k <= 32 and no 64-bit division per row (us, before / after): softmax_gather 100k
// nodes H 4 d 32 k 16 160 / 114, 4 x 200k nodes H 8 d 16 k 16 2201 / 1423; bwd_rows 309 / 232, 3901 / 2702; bwd_segments
// 4 x 200k nodes 1888 / 1061; then two rows per warp, below.
#pragma once

#include "common.cuh"
#include <math_constants.h>

namespace kmip {

constexpr int kMaxEntriesPerLane = 4;  // k <= 128; kernels come with E = 1 (k <= 32), 2 (k <= 64) and 4 entries per lane

// Lanes per row, W: a whole warp, or half of one for k <= 16, so that a warp does two rows at a time (the two halves run the
// same instructions and must be converged).  Entry t of a row lives in lane t % W of its W lanes, register t / W.  Measured
// (us, a warp per row / two rows per warp): softmax_gather 100k nodes H 4 d 32 k 16 119 / 83, 4 x 40k nodes H 8 d 16 k 16
// 295 / 177; bwd_rows 236 / 170, 545 / 333.  The second partial sum of a lane would cost the kernels of two rows a step of
// occupancy (softmax_gather 40 registers instead of 32, bwd_rows 48 and more instead of 40: 100k nodes H 4 d 32 k 16 94 and
// 206 us), so their launch bounds hold them to it.
constexpr int kHalfWarp = 16;
// Whether a gathered row is as wide as the vector loads of half a warp, or narrower.
template <typename T, int D> __host__ __device__ constexpr bool half_warp_rows() { return D / Elem<T>::kVec <= kHalfWarp; }

template <int W = 32>
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
template <int W = 32>
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// The (query, head) rows first, first + step, ... of a warp: row = i * H + h, without a 64-bit division per row.
struct RowWalk {
    int i, h;
    int H, di, dh;
    __device__ __forceinline__ RowWalk(unsigned first, unsigned step, int H_)
        : i((int)(first / (unsigned)H_)), h((int)(first % (unsigned)H_)), H(H_), di((int)(step / (unsigned)H_)), dh((int)(step % (unsigned)H_)) {}
    __device__ __forceinline__ void next() {
        i += di;
        h += dh;
        if (h >= H) { h -= H; ++i; }
    }
};

// Column sums over the W / LPR lane groups of a row's lanes.  Before: lane l holds N partial sums for part l % LPR.  A step
// exchanges halves, so N + N / 2 + ... values move instead of N per step (the additions are those of a butterfly, bit for
// bit).  After: v[0 .. kLeft) of lane l are the full sums of columns col .. col + kLeft of its part (`col` returned), and
// the lanes below kWriters hold every column once.
template <int N, int LPR, int W = 32>
struct ColumnSums {
    static constexpr int kGroups = W / LPR;
    static constexpr int kLeft = N > kGroups ? N / kGroups : 1;
    static constexpr int kWriters = N > kGroups ? W : LPR * N;
};
template <int N, int LPR, int W = 32>
__device__ __forceinline__ int column_sums(float (&v)[N], int lane) {
    int col = 0, w = N;
#pragma unroll
    for (int o = LPR; o < W; o <<= 1) {
        if (w > 1) {
            const int half = w / 2;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int c = 0; c < N / 2; ++c) {
                if (c < half) {
                    const float send = up ? v[c] : v[c + half], keep = up ? v[c + half] : v[c];
                    v[c] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
                }
            }
            col += up ? half : 0;
            w = half;
        } else {
            v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
        }
    }
    return col;
}

// n values to consecutive columns, n times the element size aligned.
template <int n>
__device__ __forceinline__ void store_columns(float* p, const float* v) {
    if constexpr (n == 1) *p = v[0];
    else if constexpr (n == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    else *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <int n>
__device__ __forceinline__ void store_columns(__nv_bfloat16* p, const float* v) {
    if constexpr (n == 1) {
        *p = __float2bfloat16_rn(v[0]);
    } else {
        uint32_t w[n / 2];
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<const uint32_t*>(&b);
        }
        if constexpr (n == 2) *reinterpret_cast<uint32_t*>(p) = w[0];
        else if constexpr (n == 4) *reinterpret_cast<uint2*>(p) = make_uint2(w[0], w[1]);
        else *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Loads the row's indices and scores and
// turns the scores into softmax weights p_t = exp((s_t - max)/sqrt(d)) / sum (Algorithm 1 line 5).
// Empty slots (index < 0) and indices outside [0, N) get weight 0.
template <int E, int W = 32>
__device__ __forceinline__ void load_row_softmax(const int32_t* idx_row, const float* score_row, int k, int N,
                                                 float scale, int lane,
                                                 int (&j)[E], float (&p)[E]) {
    float m = -CUDART_INF_F;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int t = e * W + lane;
        j[e] = -1;
        p[e] = -CUDART_INF_F;
        if (t < k) {
            j[e] = __ldg(idx_row + t);
            if (j[e] >= N) j[e] = -1;  // never follow an index outside the batch
            const float s = __ldg(score_row + t);
            if (j[e] >= 0) p[e] = s;
        }
        m = fmaxf(m, p[e]);
    }
    m = warp_max<W>(m);
    float z = 0.0f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        p[e] = (j[e] >= 0) ? __expf((p[e] - m) * scale) : 0.0f;
        z += p[e];
    }
    z = warp_sum<W>(z);
    const float inv = z > 0.0f ? 1.0f / z : 0.0f;
#pragma unroll
    for (int e = 0; e < E; ++e) p[e] *= inv;
}

// Attention dropout on the k weights of row r (= query * H + head): factor 1/(1-drop) when the slot's
// counter-based uniform is >= drop, else 0.  The draw of slot t is the (r*k + t + 1)-th SplitMix64
// output for `seed`, top 24 bits / 2^24.  f[e] belongs to entry t = e * W + lane.
template <int E, int W = 32>
__device__ __forceinline__ void dropout_factors(long long r, int k, int lane, float drop, unsigned long long seed,
                                                float (&f)[E]) {
    const float keep_scale = 1.0f / (1.0f - drop);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const unsigned long long pair = (unsigned long long)r * (unsigned long long)k + (unsigned long long)(e * W + lane);
        unsigned long long z = seed + (pair + 1ull) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z = z ^ (z >> 31);
        const float u = (float)(unsigned)(z >> 40) * (1.0f / 16777216.0f);  // 24 bits: exact in fp32
        f[e] = (u >= drop) ? keep_scale : 0.0f;
    }
}

// out_row[0, D) = sum_t w_t * X[j_t, h, :].
// LPR = D/VEC lanes share one gathered row (one 16-byte load each), W/LPR rows per round.  `lane`: among the row's W lanes.
// The order of the additions is that of 32 lanes whatever W is, so that every kernel gives the same bits: entry t goes to
// partial sum t % (32 / LPR), and these are added as a tree of neighbours.  With half a warp a lane keeps two neighbours, so
// the first step of the tree stays in the lane; up to W / LPR entries take one partial sum each, the other half are 0.
// MIN_K: a k that the caller knows to be reached; rounds below it are not asked for.
template <typename T, int D, int E, int W = 32, int MIN_K = 1>
__device__ __forceinline__ void gather_weighted_sum(const T* __restrict__ X, int H, int h, int k, int lane,
                                                    const int (&j)[E], const float (&w)[E], T* __restrict__ out_row, bool live = true) {
    constexpr int VEC = Elem<T>::kVec;
    constexpr int LPR = D / VEC;
    constexpr int EPW = W / LPR;
    constexpr int SETS = 32 / W;
    static_assert(LPR >= 1 && LPR <= W, "row width");
    const int part = lane % LPR, sub = lane / LPR;
    float acc[SETS][VEC];
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
        for (int c = 0; c < VEC; ++c) acc[s][c] = 0.0f;
    auto add = [&](int e, int src, float (&a)[VEC]) {
        const int jj = __shfl_sync(0xFFFFFFFFu, j[e], src, W);
        const float ww = __shfl_sync(0xFFFFFFFFu, w[e], src, W);
        if (jj >= 0) {
            float v[VEC];
            Elem<T>::load_vec(X + ((size_t)jj * H + h) * D + part * VEC, v);
#pragma unroll
            for (int c = 0; c < VEC; ++c) a[c] = fmaf(ww, v[c], a[c]);
        }
    };
    if (SETS == 2 && k <= EPW) {
        add(0, sub, acc[0]);
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e * W < k) {
#pragma unroll
                for (int base = 0; base < W; base += SETS * EPW) {
                    if (e * W + base >= MIN_K && e * W + base >= k) break;
#pragma unroll
                    for (int s = 0; s < SETS; ++s) add(e, base + SETS * sub + s, acc[s]);
                }
            }
        }
        if constexpr (SETS == 2) {
#pragma unroll
            for (int c = 0; c < VEC; ++c) acc[0][c] += acc[1][c];
        }
    }
    using Sums = ColumnSums<VEC, LPR, W>;
    const int col = column_sums<VEC, LPR, W>(acc[0], lane);
    if (live && lane < Sums::kWriters) store_columns<Sums::kLeft>(out_row + part * VEC + col, acc[0]);
}

// dots[e] of lane l = g . X[j[e] of lane l, h, :] for the row's entries, with
// the same lane layout as gather_weighted_sum: LPR lanes share one gathered row, one 16-byte load each, so a load
// instruction touches 32 / LPR rows instead of 32; the partial sums of a row are added across its lanes and handed
// to the entry's own lane.  g is the row-major vector of D elements at `g_row`.
template <typename T, int D, int E, int W = 32>
__device__ __forceinline__ void gather_dot(const T* __restrict__ X, int H, int h, int k, int lane, const T* __restrict__ g_row,
                                           const int (&j)[E], float (&dots)[E]) {
    constexpr int VEC = Elem<T>::kVec;
    constexpr int LPR = D / VEC;
    constexpr int EPW = W / LPR;
    const int part = lane % LPR, sub = lane / LPR;
    float gv[VEC];
    Elem<T>::load_vec(g_row + part * VEC, gv);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        dots[e] = 0.0f;
        if (e * W < k) {
#pragma unroll
            for (int base = 0; base < W; base += EPW) {
                if (e * W + base >= k) break;
                const int jj = __shfl_sync(0xFFFFFFFFu, j[e], base + sub, W);
                float s = 0.0f;
                if (jj >= 0) {
                    float v[VEC];
                    Elem<T>::load_vec(X + ((size_t)jj * H + h) * D + part * VEC, v);
#pragma unroll
                    for (int c = 0; c < VEC; ++c) s = fmaf(gv[c], v[c], s);
                }
#pragma unroll
                for (int o = 1; o < LPR; o <<= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
                // the entry of lane l was gathered by the lanes (l % EPW) * LPR ... in the round base = l - l % EPW
                const float t = __shfl_sync(0xFFFFFFFFu, s, (lane % EPW) * LPR, W);
                if (lane - lane % EPW == base) dots[e] = t;
            }
        }
    }
}

}  // namespace kmip
