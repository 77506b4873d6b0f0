// The full multi-head k-MIP self-attention layer of Eq. 2 (Algorithm 1 with its "Require" line and
// line 8), bf16: Q^h = X W_Q^h, K^h = X W_K^h, V^h = X W_V^h, O^h = kMIP-Attn(Q^h, K^h, V^h) inside each
// graph, Y = sum_h O^h W_O^h, and its backward pass with the selection held constant (Sec. 3.1).
//
// Every dense product runs in gemm_tn.cu, which reads either operand with the contraction along its rows or along its
// columns, so nothing is transposed.  A head width that the attention kernels do not take (the paper's own study uses
// d_K = 10) is zero-padded to 16, 32, 64 or 128 in copies of the weights (zero ROWS of W_Q, W_K, W_V, zero COLUMNS of
// W_O), which leaves every inner product unchanged; the softmax still divides by sqrt(d_head) because the Q projection
// is scaled by sqrt(d_pad / d_head).  Widths that need no padding use the weights where they are.
//   forward   [Q | K | V] = X [W_Q; W_K; W_V]^T   one launch, three output layers, X read once
//             attention core (kmip_attn_forward)
//             Y = O W_O^T
//   backward  dO = dY W_O;  attention backward (dQ, dK, dV);
//             dX = dQ W_Q + dK W_K + dV W_V       one launch, three K segments
//             dW_Q = dQ^T X, dW_K = dK^T X, dW_V = dV^T X, dW_O^T = O^T dY   one launch, the node axis cut into parts,
//             and one that adds the parts up
#include "common.cuh"

namespace kmip {

namespace {

// dst[r, c] = scale * src[map(r), c] for r < rows_pad: rows with r % pad >= real are zero (head padding of W_Q, W_K, W_V)
__global__ void pad_rows_kernel(const __nv_bfloat16* __restrict__ src, __nv_bfloat16* __restrict__ dst, int rows_pad, int cols,
                                int pad, int real, float scale) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)rows_pad * cols) return;
    const int r = (int)(i / cols), c = (int)(i % cols), rr = r % pad;
    dst[i] = rr < real ? __float2bfloat16_rn(__bfloat162float(src[(size_t)((r / pad) * real + rr) * cols + c]) * scale)
                       : __float2bfloat16_rn(0.0f);
}
// dst[r, c] = src[r, map(c)] for c < cols_pad: columns with c % pad >= real are zero (head padding of W_O)
__global__ void pad_cols_kernel(const __nv_bfloat16* __restrict__ src, __nv_bfloat16* __restrict__ dst, int rows, int cols_pad,
                                int pad, int real) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)rows * cols_pad) return;
    const int r = (int)(i / cols_pad), c = (int)(i % cols_pad), cc = c % pad;
    const int cols = cols_pad / pad * real;
    dst[i] = cc < real ? src[(size_t)r * cols + (c / pad) * real + cc] : __float2bfloat16_rn(0.0f);
}

}  // namespace

int layer_pad_width(int d_head) { return d_head <= 16 ? 16 : d_head <= 32 ? 32 : d_head <= 64 ? 64 : 128; }

LayerWorkspace plan_layer_workspace(int64_t N, int32_t G, int32_t d_model, int32_t H, int32_t d_head, int32_t k, int pass) {
    LayerWorkspace w;
    const int d_pad = layer_pad_width(d_head);
    const size_t hp = (size_t)H * d_pad, wbytes = hp * d_model * 2;
    size_t o = kStatusBytes;
    auto take = [&o](size_t bytes) { const size_t at = o; o = align_up(o + bytes); return at; };
    w.wq_pad = take(wbytes); w.wk_pad = take(wbytes); w.wv_pad = take(wbytes); w.wo_pad = take(wbytes);
    if (pass == KMIP_PASS_FORWARD) {
        w.attn = take(0);
        w.attn_bytes = plan_fwd_workspace(N, G > 0 ? G : 1, H, d_pad, k, KMIP_BF16_TC).total;
        o = align_up(o + w.attn_bytes);
    } else {
        // dO, dQ, dK, dV [N, H*d_pad]; the partial sums of the weight gradients get as much as the six activations they
        // are computed from (X, dY, O, dQ, dK, dV) take, and at least one part of every product
        w.d_o = take((size_t)N * hp * 2); w.d_q = take((size_t)N * hp * 2); w.d_k = take((size_t)N * hp * 2);
        w.d_v = take((size_t)N * hp * 2);
        const size_t one = 4 * 4 * hp * (size_t)d_model, room = (size_t)N * 2 * (2 * (size_t)d_model + 4 * hp);
        w.partial_bytes = room > one ? room : one;
        w.partial = take(w.partial_bytes);
        w.attn = take(0);
        w.attn_bytes = plan_bwd_workspace(N, H, k).total;
        o = align_up(o + w.attn_bytes);
    }
    w.total = o;
    return w;
}

// The weights as the products read them: padded copies (W_Q scaled, W_K, W_V with zero rows, W_O with zero columns), or
// the caller's own when the head width needs no padding.
struct Weights {
    const void *q, *k, *v, *o;
};
static cudaError_t padded_weights(const LayerArgs& a, const LayerWorkspace& w, int d_pad, float q_scale, Weights& out) {
    if (d_pad == a.d_head) {
        out = {a.w_q, a.w_k, a.w_v, a.w_o};
        return cudaSuccess;
    }
    const int hp = a.H * d_pad;
    const long long n = (long long)hp * a.d_model;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    auto P = [&](size_t off) { return reinterpret_cast<__nv_bfloat16*>(a.ws + off); };
    auto S = [](const void* p) { return static_cast<const __nv_bfloat16*>(p); };
    pad_rows_kernel<<<blocks, 256, 0, a.stream>>>(S(a.w_q), P(w.wq_pad), hp, a.d_model, d_pad, a.d_head, q_scale);
    pad_rows_kernel<<<blocks, 256, 0, a.stream>>>(S(a.w_k), P(w.wk_pad), hp, a.d_model, d_pad, a.d_head, 1.0f);
    pad_rows_kernel<<<blocks, 256, 0, a.stream>>>(S(a.w_v), P(w.wv_pad), hp, a.d_model, d_pad, a.d_head, 1.0f);
    pad_cols_kernel<<<blocks, 256, 0, a.stream>>>(S(a.w_o), P(w.wo_pad), a.d_model, hp, d_pad, a.d_head);
    out = {P(w.wq_pad), P(w.wk_pad), P(w.wv_pad), P(w.wo_pad)};
    return cudaGetLastError();
}

// Returns a kmip_status_t.
int layer_forward(const LayerArgs& a) {
    const int d_pad = layer_pad_width(a.d_head), hp = a.H * d_pad;
    const LayerWorkspace w = plan_layer_workspace(a.N, a.G, a.d_model, a.H, a.d_head, a.k, KMIP_PASS_FORWARD);
    StatusBlock* sb = reinterpret_cast<StatusBlock*>(a.ws);
    if (cudaMemsetAsync(a.ws, 0, kStatusBytes, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    // the Q projection carries sqrt(d_pad / d_head): the core divides by sqrt(d_pad), Eq. 1 by sqrt(d_head)
    Weights wt;
    if (padded_weights(a, w, d_pad, sqrtf((float)d_pad / (float)a.d_head), wt) != cudaSuccess) return KMIP_ERR_CUDA;
    GemmCall proj{};
    proj.A[0] = proj.A[1] = proj.A[2] = a.x;
    proj.B[0] = wt.q; proj.B[1] = wt.k; proj.B[2] = wt.v;
    proj.C[0] = a.q; proj.C[1] = a.k_proj; proj.C[2] = a.v;
    proj.M = (int)a.N; proj.N = hp; proj.K = a.d_model;
    proj.lda = proj.ldb = a.d_model; proj.ldc = hp;
    proj.n_batch = 3;
    if (launch_gemm(proj, sb, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    const int rc = kmip_attn_forward(a.q, a.k_proj, a.v, a.graph_offsets, a.G, a.N, a.H, d_pad, a.k, KMIP_BF16_TC, a.o,
                                     a.topk_idx, a.topk_score, a.ws + w.attn, w.attn_bytes, a.stream);
    if (rc != KMIP_OK) return rc;
    GemmCall last{};
    last.A[0] = a.o; last.B[0] = wt.o; last.C[0] = a.y;
    last.M = (int)a.N; last.N = a.d_model; last.K = hp;
    last.lda = last.ldb = hp; last.ldc = a.d_model;
    last.merge_from = reinterpret_cast<const StatusBlock*>(a.ws + w.attn);
    if (launch_gemm(last, sb, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    return KMIP_OK;
}

int layer_backward(const LayerArgs& a) {
    const int d_pad = layer_pad_width(a.d_head), hp = a.H * d_pad, N = (int)a.N;
    const LayerWorkspace w = plan_layer_workspace(a.N, a.G, a.d_model, a.H, a.d_head, a.k, KMIP_PASS_BACKWARD);
    StatusBlock* sb = reinterpret_cast<StatusBlock*>(a.ws);
    if (cudaMemsetAsync(a.ws, 0, kStatusBytes, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    const float q_scale = sqrtf((float)d_pad / (float)a.d_head);
    Weights wt;
    if (padded_weights(a, w, d_pad, q_scale, wt) != cudaSuccess) return KMIP_ERR_CUDA;
    auto P = [&](size_t off) { return static_cast<void*>(a.ws + off); };
    // dO = dY W_O (padded columns come out zero); W_O is [d_model, H*d_pad]: the contraction runs along its rows
    GemmCall g_o{};
    g_o.A[0] = a.d_y; g_o.B[0] = wt.o; g_o.C[0] = P(w.d_o);
    g_o.M = N; g_o.N = hp; g_o.K = a.d_model;
    g_o.lda = a.d_model; g_o.ldb = hp; g_o.ldc = hp;
    g_o.b_mn = true;
    if (launch_gemm(g_o, sb, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    const int rc = kmip_attn_backward(a.q, a.k_proj, a.v, a.graph_offsets, a.G, a.N, a.H, d_pad, a.k, KMIP_BF16_TC, a.o, P(w.d_o),
                                      a.topk_idx, a.topk_score, P(w.d_q), P(w.d_k), P(w.d_v), a.ws + w.attn, w.attn_bytes,
                                      a.stream);
    if (rc != KMIP_OK) return rc;
    // dX = dQ' W_Q' + dK W_K + dV W_V with the scaled, padded W_Q' (its scale is the chain rule of Q' = s Q)
    GemmCall g_x{};
    g_x.A[0] = P(w.d_q); g_x.A[1] = P(w.d_k); g_x.A[2] = P(w.d_v);
    g_x.B[0] = wt.q; g_x.B[1] = wt.k; g_x.B[2] = wt.v;
    g_x.C[0] = a.d_x;
    g_x.M = N; g_x.N = a.d_model; g_x.K = hp;
    g_x.lda = hp; g_x.ldb = a.d_model; g_x.ldc = a.d_model;
    g_x.b_mn = true;
    g_x.n_kseg = 3;
    g_x.merge_from = reinterpret_cast<const StatusBlock*>(a.ws + w.attn);
    if (launch_gemm(g_x, sb, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    // weight gradients: dW_Q = s dQ'^T X (rows of the padding dropped), dW_K, dW_V alike, dW_O = (O^T dY)^T
    GemmCall g_w{};
    g_w.A[0] = P(w.d_q); g_w.A[1] = P(w.d_k); g_w.A[2] = P(w.d_v); g_w.A[3] = a.o;
    g_w.B[0] = g_w.B[1] = g_w.B[2] = a.x; g_w.B[3] = a.d_y;
    g_w.M = hp; g_w.N = a.d_model; g_w.K = N;
    g_w.lda = hp; g_w.ldb = a.d_model; g_w.ldc = a.d_model;
    g_w.a_mn = g_w.b_mn = true;
    g_w.out_f32 = true;
    g_w.n_batch = 4;
    g_w.n_split = gemm_splits(hp, a.d_model, N, 4, w.partial_bytes);
    float* partial = static_cast<float*>(P(w.partial));
    for (int z = 0; z < 4; ++z) g_w.C[z] = partial + (size_t)z * g_w.n_split * hp * a.d_model;
    if (launch_gemm(g_w, sb, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    const ReduceOut out{{a.dw_q, a.dw_k, a.dw_v, a.dw_o}, {q_scale, 1.0f, 1.0f, 1.0f}, {0, 0, 0, 1}};
    if (launch_reduce_partials(partial, g_w.n_split, hp, a.d_model, d_pad, a.d_head, 4, out, a.stream) != cudaSuccess) return KMIP_ERR_CUDA;
    return KMIP_OK;
}

}  // namespace kmip
