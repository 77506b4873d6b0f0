// Dense products of the full attention layer (Eq. 2; Algorithm 1 "Require" line and line 8), bf16 operands with fp32
// accumulation on the 5th-generation tensor cores: TMA -> shared-memory ring (128-byte swizzle) -> tcgen05.mma
// (M 128 x N 128 x K 16, accumulators in tensor memory) -> four epilogue warps.
//   C_z[M, N] = A_z[M, K] B_z[N, K]^T
// Either operand may lie in memory with K as its row axis instead ("MN-major": A stored [K, M], B stored [K, N]); TMA
// then brings boxes of 64 columns x 64 rows and the matrix descriptors say so, which is why no activation or weight is
// ever transposed (ten transposes cost 203 us of a 114 001-node training step).  Three uses of a launch:
//   batched   up to four (A, B, C) triples, one grid layer each (the Q, K and V projections of X);
//   summed    C = sum_i A_i B_i^T over up to three K segments (dX = dQ W_Q + dK W_K + dV W_V);
//   split     the K axis of every product is cut into parts, one grid layer each, that store fp32 partial sums
//             [product][part][M][N] (weight gradients, whose K axis is the node axis: with one CTA per output tile
//             the four products of a 114 001-node graph took 3.6 ms on four SMs); launch_reduce_partials adds them up
//             in a fixed order.
// One CTA per 128 x 128 output tile and part; ragged edges are zero-filled by TMA on the way in and masked on the way
// out.  Products with at most two K blocks take two ring stages instead of four: three CTAs then share an SM and hide
// each other's latencies.  Every wait is bounded (status word KMIP_ERR_TIMEOUT, clean return).
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "ptx.cuh"

namespace kmip {

namespace {

constexpr int GM = 128, GN = 128, GK = 64;
constexpr int kTileBytes = 128 * GK * 2;  // one operand tile: 128 x 64 elements
constexpr int kGemmThreads = 192;         // warp 0: TMA producer, warp 1: MMA issuer (owns TMEM), warps 2-5: epilogue
constexpr unsigned FULL = 0xFFFFFFFFu;

// 128-byte swizzle, 8-row groups 1024 bytes apart.  K-major: the rows are M or N, 64 K values each.  MN-major: the rows
// are K, 64 M or N values each, and the two 64-wide halves of a tile are 8192 bytes apart (leading offset).
__device__ __forceinline__ uint64_t gemm_desc(uint32_t saddr, bool mn_major) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(mn_major ? (kTileBytes / 2) >> 4 : 1) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// fp32 accumulate, bf16 A and B, M = 128, N = 128; bits 15 and 16: A, B are MN-major
constexpr uint32_t kGemmIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GN >> 3) << 17) | ((uint32_t)(GM >> 4) << 24);

struct GemmParams {
    CUtensorMap a[4], b[4];
    void* C[4];
    int M, N, K;
    int ldc;          // elements between output rows
    int a_mn, b_mn;   // operand is MN-major
    int out_f32;      // 1: fp32 output, 0: bf16
    int n_batch;      // products; the grid has n_batch * n_split layers
    int n_kseg;       // summed mode: K segments (1 otherwise)
    int kb_per_split; // K blocks per part
    StatusBlock* sb;
    const StatusBlock* merge_from;  // status of the attention call before this launch, copied into sb (may be null)
    long long wait_limit;
};

// One operand tile: rows (or columns) r0 .. r0+127 of the M / N axis, K values k0 .. k0+63.
__device__ __forceinline__ void load_tile(uint32_t dst, const CUtensorMap* tm, bool mn_major, int r0, int k0, uint32_t bar) {
    if (mn_major) {
        ptx::tma_load_2d(dst, tm, r0, k0, bar);
        ptx::tma_load_2d(dst + kTileBytes / 2, tm, r0 + 64, k0, bar);
    } else {
        ptx::tma_load_2d(dst, tm, k0, r0, bar);
    }
}

template <int GS>
__global__ void __launch_bounds__(kGemmThreads)
gemm_tn_kernel(const __grid_constant__ GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = smem + GS * kTileBytes;
    uint64_t* sBars = reinterpret_cast<uint64_t*>(sB + GS * kTileBytes);
    uint32_t* sTmem = reinterpret_cast<uint32_t*>(sBars + 2 * GS + 1);
    volatile int* sAbort = reinterpret_cast<volatile int*>(sTmem + 1);
    const uint32_t bar0 = ptx::smem_u32(sBars);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto empty = [&](int s) { return bar0 + 8u * (GS + s); };
    const uint32_t acc_full = bar0 + 8u * (2 * GS);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * GM, n0 = blockIdx.y * GN;
    const int z = blockIdx.z % p.n_batch, split = blockIdx.z / p.n_batch;
    const int nk_seg = (p.K + GK - 1) / GK;  // K blocks per segment
    const int kb_lo = split * p.kb_per_split, kb_hi = min(nk_seg * p.n_kseg, kb_lo + p.kb_per_split);

    if (threadIdx.x == 0) {
        for (int s = 0; s < GS; ++s) { ptx::mbar_init(full(s), 1); ptx::mbar_init(empty(s), 1); }
        ptx::mbar_init(acc_full, 1);
        *sAbort = 0;
        ptx::fence_barrier_init();
        ptx::fence_proxy_async();
        if (p.merge_from && blockIdx.x + blockIdx.y + blockIdx.z == 0 && p.merge_from->status != KMIP_OK)
            record_status(p.sb, p.merge_from->status, p.merge_from->detail);
    }
    if (warp == 1) { ptx::tmem_alloc(ptx::smem_u32(sTmem), GN); ptx::tmem_relinquish(); }
    if (warp == 0 && lane == 0) { ptx::prefetch_tensormap(&p.a[z]); ptx::prefetch_tensormap(&p.b[z]); }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = *sTmem;
    bool ok = true;

    if (warp == 0) {
        if (lane == 0) {
            for (int kb = kb_lo; kb < kb_hi; ++kb) {
                const int x = kb - kb_lo, s = x % GS;
                if (!(ok = ptx::mbar_wait_bounded<0>(empty(s), ((x / GS) & 1) ^ 1, sAbort, p.wait_limit))) break;
                const int seg = kb / nk_seg, kk = (kb - seg * nk_seg) * GK;
                const int op = p.n_kseg > 1 ? seg : z;
                ptx::mbar_arrive_expect_tx(full(s), 2 * kTileBytes);
                load_tile(ptx::smem_u32(sA + s * kTileBytes), &p.a[op], p.a_mn, m0, kk, full(s));
                load_tile(ptx::smem_u32(sB + s * kTileBytes), &p.b[op], p.b_mn, n0, kk, full(s));
            }
            if (!ok) record_status(p.sb, KMIP_ERR_TIMEOUT, 21);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = kGemmIdesc | (p.a_mn ? 1u << 15 : 0u) | (p.b_mn ? 1u << 16 : 0u);
            // 16 K values further: 32 bytes along a row, or 16 rows of 128 bytes
            const uint64_t step_a = p.a_mn ? 2048 >> 4 : 2, step_b = p.b_mn ? 2048 >> 4 : 2;
            for (int kb = kb_lo; kb < kb_hi; ++kb) {
                const int x = kb - kb_lo, s = x % GS;
                if (!(ok = ptx::mbar_wait_bounded<0>(full(s), (x / GS) & 1, sAbort, p.wait_limit))) break;
                ptx::tc_fence_after();
                const uint64_t da = gemm_desc(ptx::smem_u32(sA + s * kTileBytes), p.a_mn);
                const uint64_t db = gemm_desc(ptx::smem_u32(sB + s * kTileBytes), p.b_mn);
#pragma unroll
                for (int ks = 0; ks < GK / 16; ++ks)
                    ptx::mma_bf16_ss(tmem, da + ks * step_a, db + ks * step_b, idesc, (x > 0 || ks > 0) ? 1u : 0u);
                ptx::mma_commit(empty(s));  // the stage is free once these MMAs have read it
            }
            if (ok) ptx::mma_commit(acc_full);
            else record_status(p.sb, KMIP_ERR_TIMEOUT, 22);
        }
    } else {
        // epilogue: warp w reads the TMEM lanes of its sub-partition, 32 rows x 32 columns at a time
        const int quarter = warp & 3;
        ok = ptx::mbar_wait_bounded<0>(acc_full, 0, sAbort, p.wait_limit);
        ok = __all_sync(FULL, ok);
        if (ok) {
            ptx::tc_fence_after();
            const int row = m0 + quarter * 32 + lane;
            // 16-byte stores where the rows allow them
            const bool vec = ((size_t)p.ldc * (p.out_f32 ? 4 : 2)) % 16 == 0;
            const size_t part = (size_t)split * p.M;  // split mode: parts of a product follow each other
#pragma unroll 1
            for (int c0 = 0; c0 < GN && n0 + c0 < p.N; c0 += 32) {
                uint32_t v[32];
                ptx::tmem_ld_32x32_sync(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
                if (row < p.M) {
                    const size_t o = (part + row) * p.ldc + n0 + c0;
                    const int left = p.N - n0 - c0;
                    if (p.out_f32) {
                        float* c = static_cast<float*>(p.C[z]) + o;
#pragma unroll
                        for (int x = 0; x < 32; x += 4) {
                            if (vec && x + 4 <= left) {
                                *reinterpret_cast<uint4*>(c + x) = make_uint4(v[x], v[x + 1], v[x + 2], v[x + 3]);
                            } else {
#pragma unroll
                                for (int y = 0; y < 4; ++y)
                                    if (x + y < left) c[x + y] = __uint_as_float(v[x + y]);
                            }
                        }
                    } else {
                        __nv_bfloat16* c = static_cast<__nv_bfloat16*>(p.C[z]) + o;
#pragma unroll
                        for (int x = 0; x < 32; x += 8) {
                            float f[8];
#pragma unroll
                            for (int y = 0; y < 8; ++y) f[y] = __uint_as_float(v[x + y]);
                            if (vec && x + 8 <= left) {
                                Elem<__nv_bfloat16>::store_vec(c + x, f);
                            } else {
#pragma unroll
                                for (int y = 0; y < 8; ++y)
                                    if (x + y < left) c[x + y] = __float2bfloat16_rn(f[y]);
                            }
                        }
                    }
                }
                __syncwarp();
            }
        } else if (lane == 0) {
            record_status(p.sb, KMIP_ERR_TIMEOUT, 23);
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) { ptx::tc_fence_after(); ptx::tmem_dealloc(tmem, GN); }
}

// dst_z = scale_z * sum over the parts of partial[z][part][M][N], in part order, as bf16, without the zero padding of the
// heads: index i of the padded M axis is kept iff i % pad < real and lands at (i / pad) * real + i % pad.  transposed_z:
// dst_z is [N, M'] instead of [M', N].
__global__ void reduce_partials_kernel(const float* __restrict__ partial, int n_split, int M, int N, int pad, int real,
                                       const ReduceOut out) {
    const int z = blockIdx.y;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)M * N) return;
    const int m = (int)(i / N), n = (int)(i % N);
    if (m % pad >= real) return;
    const float* src = partial + (size_t)z * n_split * M * N + i;
    float acc = 0.0f;
#pragma unroll 8
    for (int s = 0; s < n_split; ++s) acc += __ldg(src + (size_t)s * M * N);
    const int om = (m / pad) * real + m % pad, om_n = M / pad * real;
    __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(out.dst[z]);
    dst[out.transposed[z] ? (size_t)n * om_n + om : (size_t)om * N + n] = __float2bfloat16_rn(acc * out.scale[z]);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn gemm_encode_fn() {
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

// bf16 matrix [rows, cols] with `ld` elements between rows; a box is `box_rows` rows x 64 columns, out-of-range parts read as 0
bool gemm_tensor_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    EncodeTiledFn enc = gemm_encode_fn();
    if (!enc) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int GS>
cudaError_t launch_gs(const GemmParams& p, dim3 grid, cudaStream_t stream) {
    constexpr size_t smem = 1024 + 2 * GS * kTileBytes + (2 * GS + 1) * 8 + 64;
    cudaError_t err = cudaFuncSetAttribute(gemm_tn_kernel<GS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    gemm_tn_kernel<GS><<<grid, kGemmThreads, smem, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace

// Leading dimensions in elements, multiples of 8; bases 16-byte aligned.  n_kseg > 1 needs n_batch = 1 and n_split = 1;
// n_split > 1 needs fp32 outputs with room for n_split * M rows each.
cudaError_t launch_gemm(const GemmCall& g, StatusBlock* sb, cudaStream_t stream) {
    if (g.M <= 0 || g.N <= 0 || g.K <= 0) return cudaSuccess;
    const int n_op = g.n_kseg > 1 ? g.n_kseg : g.n_batch;
    if (g.n_batch < 1 || g.n_batch > 4 || g.n_kseg < 1 || g.n_kseg > 3 || g.n_split < 1 || (g.n_batch > 1 && g.n_kseg > 1) ||
        (g.n_split > 1 && (g.n_kseg > 1 || !g.out_f32)) || (g.lda & 7) || (g.ldb & 7) || !sb)
        return cudaErrorInvalidValue;
    GemmParams p;
    for (int z = 0; z < 4; ++z) {
        const int zo = z < n_op ? z : 0;
        const bool ok_a = g.a_mn ? gemm_tensor_map(&p.a[z], g.A[zo], g.K, g.M, g.lda, GK) : gemm_tensor_map(&p.a[z], g.A[zo], g.M, g.K, g.lda, GM);
        const bool ok_b = g.b_mn ? gemm_tensor_map(&p.b[z], g.B[zo], g.K, g.N, g.ldb, GK) : gemm_tensor_map(&p.b[z], g.B[zo], g.N, g.K, g.ldb, GN);
        if (!ok_a || !ok_b) return cudaErrorInvalidValue;
        p.C[z] = g.C[z < g.n_batch ? z : 0];
    }
    const int nk = (g.K + GK - 1) / GK * g.n_kseg;
    p.M = g.M; p.N = g.N; p.K = g.K;
    p.ldc = g.ldc;
    p.a_mn = g.a_mn; p.b_mn = g.b_mn;
    p.out_f32 = g.out_f32;
    p.n_batch = g.n_batch;
    p.n_kseg = g.n_kseg;
    p.kb_per_split = (nk + g.n_split - 1) / g.n_split;
    p.sb = sb;
    p.merge_from = g.merge_from;
    p.wait_limit = kDefaultWaitLimitCycles;
    const dim3 grid((g.M + GM - 1) / GM, (g.N + GN - 1) / GN, g.n_batch * g.n_split);
    return p.kb_per_split <= 2 ? launch_gs<2>(p, grid, stream) : launch_gs<4>(p, grid, stream);
}

int gemm_splits(int M, int N, int K, int n_batch, size_t partial_bytes) {
    const int nk = (K + GK - 1) / GK, tiles = ((M + GM - 1) / GM) * ((N + GN - 1) / GN) * n_batch;
    // one wave of CTAs, at least four K blocks each (their reduction costs 64 KB of traffic a tile and part)
    int s = std::max(1, std::min(sm_count() / tiles, nk / 4));
    s = (int)std::min<long long>(s, (long long)(partial_bytes / ((size_t)n_batch * M * N * 4)));
    if (s < 1) return 1;
    const int per = (nk + s - 1) / s;
    return (nk + per - 1) / per;  // no empty parts
}

cudaError_t launch_reduce_partials(const float* partial, int n_split, int M, int N, int pad, int real, int n_batch, const ReduceOut& out,
                                   cudaStream_t stream) {
    const dim3 grid((unsigned)(((long long)M * N + 255) / 256), (unsigned)n_batch);
    reduce_partials_kernel<<<grid, 256, 0, stream>>>(partial, n_split, M, N, pad, real, out);
    return cudaGetLastError();
}

}  // namespace kmip
