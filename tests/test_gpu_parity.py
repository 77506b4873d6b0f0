"""GPU parity tests: the CUDA path, called through the C ABI, against the CPU oracle."""
import numpy as np
import pytest
import torch

from paper_2604_03815_b200 import workloads as wl

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2604_03815_b200 import binding as kb
    from tests import parity_util as pu


# which kernels a call runs (kmip_test.h): 0 = the library's choice, the small-graph kernel, the prefilter, the fp32-accumulate sweep
SMALL, FILTER, TENSOR_CORE = 1, 2, 3
MODE_AND_ROUTE = [(wl.MODE_BF16_TC, SMALL), (wl.MODE_BF16_TC, FILTER), (wl.MODE_BF16_TC, TENSOR_CORE), (wl.MODE_FP32_EXACT, SMALL),
                  (wl.MODE_FP32_EXACT, FILTER), (wl.MODE_FP32_EXACT, 0)]


def _fwd_bwd(w, rows=None, backward=True, fp32_path=0, route=0):
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev, fp32_path=fp32_path, route=route)
    st = pu.check_forward(w, fb, rows)
    if backward:
        bb = pu.run_backward(w, fb, dev)
        st.update(pu.check_backward(w, fb, bb))
    return st


# ------------------------------------------------------------------ tensor-core contraction alone
@pytest.mark.parametrize("d", [16, 32, 64, 128])
def test_tc_dense_scores_match_fp64(d):
    N, H = 300, 2                      # three key tiles with a ragged tail, two 128-row query tiles + tail
    w = wl.iid_workload("s", 40 + d, [N], H, d, 4, wl.MODE_BF16_TC)
    Q, K, V, dO, offs = pu.to_device(w)
    S = torch.full((H, N, N), float("nan"), dtype=torch.float32, device="cuda")
    ws = torch.empty(kb.kmip_attn_workspace_bytes(N, 1, H, d, 1, kb.KMIP_BF16_TC, kb.PASS_FORWARD),
                     dtype=torch.uint8, device="cuda")
    assert kb.kmip_test_tc_scores(Q, K, S, ws) == kb.KMIP_OK
    assert kb.kmip_last_status(ws) == kb.KMIP_OK
    ref = np.einsum("ihc,jhc->hij", w.Q.astype(np.float64), w.K.astype(np.float64))
    got = S.cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    np.testing.assert_allclose(got, ref, rtol=2e-5, atol=1e-5 * np.sqrt(d))


# ------------------------------------------------------------------ small cases, every element
def test_config1_fp32_exact():
    w = wl.make_config(1)
    st = _fwd_bwd(w, backward=False)
    assert st["identical_rows"] == 1.0 and st["min_gap"] > pu.FP32_SCORE_ERR   # bit-exact indices, no near-tie
    assert st["undecided_set_rows"] == 0 and st["excused_rows"] == 0            # no row is excused


def test_config1_fp32_backward_too():
    w = wl.make_config(1)
    _fwd_bwd(w, backward=True)


def test_config2_batched_small_graphs():
    w = wl.make_config(2)
    st = _fwd_bwd(w)
    assert st["identical_rows"] > 0.99


@pytest.mark.parametrize("d,k,H,N", [(32, 16, 4, 3000), (16, 8, 3, 2500), (64, 32, 2, 1500), (128, 20, 1, 1100),
                                     (32, 1, 2, 700), (32, 32, 1, 257), (16, 48, 2, 900), (64, 96, 1, 700),
                                     (128, 64, 1, 600), (32, 128, 1, 600)])
def test_small_single_graph_bf16(d, k, H, N):
    w = wl.iid_workload("s", 1000 + d + k, [N], H, d, k, wl.MODE_BF16_TC, input_scale=1.0 / np.sqrt(d))
    st = _fwd_bwd(w)
    assert st["identical_rows"] > 0.98


@pytest.mark.parametrize("d,k", [(16, 5), (32, 16), (64, 40), (128, 100)])
def test_small_fp32_mode(d, k):
    w = wl.iid_workload("s", 2000 + d, [500, 300], 2, d, k, wl.MODE_FP32_EXACT, input_scale=1.0 / np.sqrt(d))
    st = _fwd_bwd(w)
    assert st["identical_rows"] == 1.0
    assert st["excused_rows"] == 0


def test_small_pointcloud_mixture():
    w = wl.make_config(4, N=4000)
    _fwd_bwd(w)


def test_small_hub_batch():
    w = wl.make_config(5, n_per_graph=1500)
    _fwd_bwd(w)


# ------------------------------------------------------------------ edge cases
@pytest.mark.parametrize("mode,route", MODE_AND_ROUTE)
def test_ragged_batch_with_tiny_and_empty_graphs(mode, route):
    sizes = [1, 0, 3, 129, 0, 7, 256, 2, 385, 16, 31, 33]
    w = wl.iid_workload("s", 77, sizes, 2, 32, 16, mode)
    st = _fwd_bwd(w, route=route)
    assert st["rows"] == sum(sizes)


@pytest.mark.parametrize("route", [FILTER, TENSOR_CORE])
def test_item_and_ring_boundaries(route):
    """Graphs around the work-item sizes of the sweeps (128, 256 and 384 rows): one to three active query
    tiles, several items, a short last key tile, and enough key tiles per item for the accumulator buffers and their
    barrier phases to wrap several times."""
    sizes = [383, 384, 385, 511, 512, 513, 769, 1025, 1153, 2000, 127, 128, 129]
    for d, k in ((32, 32), (16, 16)):
        w = wl.iid_workload("s", 90 + d, sizes, 2, d, k, wl.MODE_BF16_TC, input_scale=1.0 / np.sqrt(d))
        st = _fwd_bwd(w, route=route)
        assert st["rows"] == sum(sizes)


@pytest.mark.parametrize("mode,route", MODE_AND_ROUTE)
def test_padded_head_width_of_the_paper_sweep(mode, route):
    """d_K = 10 stored zero-padded to 16 columns, k = 10, one head (the shape of the paper's size
    sweep): same parity bar as every other shape, and the padded output and gradient columns stay zero."""
    w = wl.padded_workload("s", 91, 3000, 1, 10, 16, 10, mode)
    _fwd_bwd(w, route=route)


def test_single_node():
    w = wl.iid_workload("s", 78, [1], 2, 16, 4, wl.MODE_BF16_TC)
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev)
    assert fb.topk_idx.cpu().numpy()[0, :, 0].tolist() == [0, 0]
    assert np.all(fb.topk_idx.cpu().numpy()[0, :, 1:] == -1)
    np.testing.assert_allclose(fb.out.float().cpu().numpy(), w.V, rtol=1e-2)
    pu.check_forward(w, fb)


@pytest.mark.parametrize("mode,route", MODE_AND_ROUTE)
def test_identical_keys_tie_break_by_index(mode, route):
    w = wl.iid_workload("s", 79, [200, 90], 2, 32, 8, mode)
    w.K[:] = w.K[5]
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev, route=route)
    idx = fb.topk_idx.cpu().numpy()
    assert np.all(idx[:200] == np.arange(8)) and np.all(idx[200:] == 200 + np.arange(8))
    pu.check_forward(w, fb)


# fp32 problems with at least 48 blocks of 128 rows x heads have the tiled CUDA-core sweep and the
# fp32 rescoring kernel behind the prefilter; here the two run by themselves
@pytest.mark.parametrize("d,k", [(16, 10), (32, 32), (64, 17)])
def test_fp32_tiled_sweep(d, k):
    sizes = [3000, 129, 5000, 1, 2000, 383, 0, 64]
    w = wl.iid_workload("s", 3000 + d, sizes, 4, d, k, wl.MODE_FP32_EXACT, input_scale=1.0 / np.sqrt(d))
    st = _fwd_bwd(w, fp32_path=2)
    assert st["identical_rows"] > 0.999   # all but rows where two neighbouring scores tie within fp32 rounding
    # of ~42 000 (row, head) pairs the rule could excuse up to 714 (oracle neighbours closer than the fp32
    # error bound); the pairs that really differ, and are let through, stay a handful
    assert st["undecided_order_rows"] <= 800 and st["excused_rows"] <= 8


def test_fp32_tiled_sweep_tie_break_by_index():
    """Identical keys inside each graph: every score of a row ties, so the answer is the k lowest
    key indices of the graph, and equal group maxima must be ordered by their first key."""
    w = wl.iid_workload("s", 3100, [6000, 4500], 4, 16, 12, wl.MODE_FP32_EXACT)
    w.K[:] = w.K[7]
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev, fp32_path=2)
    idx = fb.topk_idx.cpu().numpy()
    assert np.all(idx[:6000] == np.arange(12)) and np.all(idx[6000:] == 6000 + np.arange(12))
    pu.check_forward(w, fb)


@pytest.mark.parametrize("d,k", [(16, 5), (32, 16), (64, 32)])
def test_fp32_sweeps_agree_bit_for_bit(d, k):
    """The two fp32-mode sweeps (one warp per row; tiled, thread per row) run the same fp32 FMAs in
    the same order and the same (score desc, key asc) rule: identical outputs on ragged batches
    with tiny and empty graphs, whichever the library would pick by size."""
    sizes = [1, 0, 3, 129, 0, 7, 256, 2, 385, 16, 31, 33, 700]
    w = wl.iid_workload("s", 3200 + d, sizes, 2, d, k, wl.MODE_FP32_EXACT, input_scale=1.0 / np.sqrt(d))
    dev = pu.to_device(w)
    res = []
    for path in (1, 2):
        fb = pu.run_forward(w, dev, fp32_path=path)
        torch.cuda.synchronize()
        res.append((fb.topk_idx.cpu().numpy().copy(), fb.topk_score.cpu().numpy().copy(), fb.out.cpu().numpy().copy()))
    for a, b in zip(res[0], res[1]):
        assert np.array_equal(a, b)
    pu.check_forward(w, fb)


@pytest.mark.parametrize("route", [SMALL, FILTER, TENSOR_CORE])
def test_null_offsets_means_one_graph(route):
    w = wl.iid_workload("s", 80, [600], 2, 32, 8, wl.MODE_BF16_TC)
    Q, K, V, dO, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, w.k, w.mode, route=route)
    b = kb.forward(Q, K, V, None, w.k, w.mode, route=route)
    torch.cuda.synchronize()
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.out, b.out)


def test_forward_is_deterministic():
    w = wl.make_config(5, n_per_graph=1200)
    dev = pu.to_device(w)
    a = pu.run_forward(w, dev)
    b = pu.run_forward(w, dev)
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score) and torch.equal(a.out, b.out)


def test_bad_offsets_are_reported_by_the_device():
    w = wl.iid_workload("s", 81, [300, 300], 1, 32, 8, wl.MODE_BF16_TC)
    Q, K, V, dO, offs = pu.to_device(w)
    bad = torch.tensor([0, 400, 300, 600], dtype=torch.int32, device="cuda")
    b = kb.ForwardBuffers(600, 3, 1, 32, 8, w.mode)
    assert kb.kmip_attn_forward(Q, K, V, bad, 8, w.mode, b.out, b.topk_idx, b.topk_score, b.workspace) == kb.KMIP_OK
    assert kb.kmip_last_status(b.workspace) == kb.KMIP_ERR_BAD_OFFSETS
    # the context is still usable afterwards
    pu.check_forward(w, pu.run_forward(w, (Q, K, V, dO, offs)))


def test_bounded_wait_runs_out_and_is_reported():
    """Failure detection without a GPU fault: a per-call test option (kmip_test.h) leaves one key tile of
    CTA 0 unloaded, so the waits on it can never be satisfied.  They must run out (limit shortened to
    ~0.2 s of SM clocks), the kernel must return normally with KMIP_ERR_TIMEOUT in the status word, and
    the context must stay usable for the next call."""
    w = wl.iid_workload("s", 83, [2000], 1, 32, 8, wl.MODE_BF16_TC)
    dev = pu.to_device(w)
    Q, K, V, dO, offs = dev
    b = kb.ForwardBuffers(w.N, 1, w.H, w.d, w.k, w.mode)
    assert kb.kmip_test_attn_forward(Q, K, V, offs, w.k, w.mode, b.out, b.topk_idx, b.topk_score, b.workspace,
                                     wait_limit_cycles=400_000_000, drop_first_tile=1) == kb.KMIP_OK
    assert kb.kmip_last_status(b.workspace) == kb.KMIP_ERR_TIMEOUT
    torch.cuda.synchronize()
    pu.check_forward(w, pu.run_forward(w, dev))


@pytest.mark.parametrize("route", [0, SMALL, FILTER, TENSOR_CORE])
def test_forward_and_backward_replay_from_a_cuda_graph(route):
    """Both calls only enqueue work on the caller's stream (no allocation, no synchronisation), so a
    forward + backward pair can be captured once and replayed on new input values."""
    w = wl.make_config(2)
    Q, K, V, dO, offs = pu.to_device(w)
    G = len(w.graph_offsets) - 1
    fb = kb.ForwardBuffers(w.N, G, w.H, w.d, w.k, w.mode)
    bb = kb.BackwardBuffers(w.N, G, w.H, w.d, w.k, w.mode)

    def step():
        if route:
            assert kb.kmip_test_attn_forward(Q, K, V, offs, w.k, w.mode, fb.out, fb.topk_idx, fb.topk_score, fb.workspace,
                                             route=route) == kb.KMIP_OK
        else:
            assert kb.kmip_attn_forward(Q, K, V, offs, w.k, w.mode, fb.out, fb.topk_idx, fb.topk_score, fb.workspace) == kb.KMIP_OK
        assert kb.kmip_attn_backward(Q, K, V, offs, w.k, w.mode, fb.out, dO, fb.topk_idx, fb.topk_score, bb.dQ, bb.dK,
                                     bb.dV, bb.workspace) == kb.KMIP_OK

    step()  # first call outside the capture (driver entry points, kernel attributes)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    # new values in the same buffers: rows reversed inside the batch would change graphs, so scale instead
    Q.mul_(-1.0)
    dO.mul_(0.5)
    graph.replay()
    torch.cuda.synchronize()
    assert kb.kmip_last_status(fb.workspace) == kb.KMIP_OK and kb.kmip_last_status(bb.workspace) == kb.KMIP_OK
    got = [t.clone() for t in (fb.out, fb.topk_idx, fb.topk_score, bb.dQ, bb.dK, bb.dV)]
    step()  # eager, same inputs
    torch.cuda.synchronize()
    for a, b in zip(got[:3], (fb.out, fb.topk_idx, fb.topk_score)):
        assert torch.equal(a, b)
    for a, b in zip(got[3:], (bb.dQ, bb.dK, bb.dV)):   # hit lists are filled with atomics: equal up to summation order
        assert torch.allclose(a.float(), b.float(), rtol=2e-2, atol=2e-3)
    w2 = wl.make_config(2)
    w2.Q *= -1.0
    w2.dOut *= 0.5
    pu.check_forward(w2, fb)
    pu.check_backward(w2, fb, bb)


def test_workspace_too_small_is_refused():
    w = wl.iid_workload("s", 82, [300], 1, 32, 8, wl.MODE_BF16_TC)
    Q, K, V, dO, offs = pu.to_device(w)
    b = kb.ForwardBuffers(300, 1, 1, 32, 8, w.mode)
    small = torch.empty(64, dtype=torch.uint8, device="cuda")
    assert kb.kmip_attn_forward(Q, K, V, offs, 8, w.mode, b.out, b.topk_idx, b.topk_score, small) == kb.KMIP_ERR_WORKSPACE


def test_workspace_is_linear_in_n():
    a = kb.kmip_attn_workspace_bytes(100_000, 1, 4, 32, 16, kb.KMIP_BF16_TC, kb.PASS_BACKWARD)
    b = kb.kmip_attn_workspace_bytes(1_000_000, 1, 4, 32, 16, kb.KMIP_BF16_TC, kb.PASS_BACKWARD)
    assert b < 10.5 * a and b < 1_000_000 * 4 * (10 * 16 + 4) * 4 + (160 << 20)   # 40 bytes per selected pair + per-row arrays + digit table (at most 4096 digits x 7104 warps x 4 bytes)
    # forward: 2-byte copies of K (regrouped) and Q (sweep order), the prefilter's 24 groups of 6 bytes and a redo
    # slot per (node, head), 6 bytes per node, work items
    rows = 1_000_000 * 4
    assert kb.kmip_attn_workspace_bytes(1_000_000, 1, 4, 32, 16, kb.KMIP_BF16_TC, kb.PASS_FORWARD) < 2 * rows * 32 * 2 + rows * (24 * 6 + 4) + 8 * 1_000_000


@pytest.mark.parametrize("route", [SMALL, FILTER, TENSOR_CORE])
@pytest.mark.parametrize("d", [64, 32])
def test_kth_score_near_zero_keeps_k_keys(d, route):
    """Rows whose k-th best score is a tiny remainder of large cancelling terms: the tensor-core score and
    the fp32 rescoring of the same key differ by far more than any margin RELATIVE to that score, and the
    key that defines the k-th place must still come back (Algorithm 1 line 3 returns k keys whenever the
    graph has k nodes): no padded slot, and the usual acceptance rule on every row."""
    k, H, n = 8, 2, 600
    w = wl.iid_workload("s", 6100 + d, [n, n], H, d, k, wl.MODE_BF16_TC)
    rng = np.random.default_rng(61)
    u = np.full(d, 0.125, dtype=np.float32)
    alt = np.where(np.arange(d) % 2 == 0, 1.0, -1.0).astype(np.float32)
    w.Q[:] = wl.round_to_bf16(u[None, None, :] + 0.01 * rng.standard_normal(w.Q.shape).astype(np.float32))
    K = -u[None, None, :] * rng.uniform(0.5, 1.5, size=(w.N, H, 1)).astype(np.float32)          # clearly negative scores
    for g0 in (0, n):
        K[g0 + 3:g0 + 3 + (k - 1)] = 2.0 * u                                                      # k-1 clearly positive keys
        near = g0 + 50 + 9 * np.arange(24)                                                         # 24 keys that score about zero
        K[near] = 4.0 * (u * alt)[None, None, :] + 2.0 ** -13 * rng.standard_normal((24, H, d)).astype(np.float32)
    w.K[:] = wl.round_to_bf16(K)
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev, route=route)
    idx = fb.topk_idx.cpu().numpy()
    assert np.all(idx >= 0), f"{int((idx < 0).sum())} padded slots although every graph has more than k nodes"
    pu.check_forward(w, fb)


@pytest.mark.parametrize("sizes,H,d,k,mode", [([1, 2, 0, 33, 31], 2, 16, 32, wl.MODE_BF16_TC), ([255, 256, 257, 64, 1], 1, 32, 7, wl.MODE_BF16_TC),
                                              ([511, 513, 40], 3, 64, 31, wl.MODE_BF16_TC), ([1500], 1, 16, 1, wl.MODE_BF16_TC),
                                              ([255, 256, 257, 3], 2, 16, 9, wl.MODE_FP32_EXACT), ([700, 0, 5], 1, 64, 32, wl.MODE_FP32_EXACT),
                                              ([1030], 1, 32, 16, wl.MODE_FP32_EXACT)])
def test_small_graphs_in_one_kernel(sizes, H, d, k, mode):
    """Batches whose forward pass is one kernel: chunk edges (256 keys), graphs smaller than k and than a warp, several
    graphs in a block, several chunks against the running list; with ties, which the list order must break by key."""
    w = wl.iid_workload("s", 6300 + sum(sizes) + k, sizes, H, d, k, mode, backward=False)
    pu.check_forward(w, pu.run_forward(w))
    w.K[::2] = w.K[1]                                    # half of the keys tie
    Q, K, V, dO, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, k, w.mode)
    # one warp per row in fp32: of bf16 values the same exact products and the same order of sums
    b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score)


@pytest.mark.parametrize("n,H,d,k,mode", [(1, 1, 16, 3, "bf16"), (31, 2, 32, 32, "fp32"), (33, 1, 64, 7, "bf16"), (256, 3, 16, 32, "fp32"),
                                          (257, 1, 64, 1, "fp32"), (512, 2, 32, 20, "bf16"), (513, 1, 16, 31, "bf16"), (300, 4, 64, 9, "fp32"),
                                          (1184, 1, 32, 16, "fp32"), (1185, 1, 32, 16, "bf16"), (2047, 1, 64, 24, "fp32"), (2100, 1, 16, 5, "bf16")])
def test_one_graph_in_one_kernel(n, H, d, k, mode):
    """One graph without a plan kernel: one, two and four warps per row, 8 and 16 rows per block, partial blocks and partial groups
    of 32 keys; then with a few hundred equal scores per row, more than a warp keeps unsorted, which go by key."""
    m = {"bf16": wl.MODE_BF16_TC, "fp32": wl.MODE_FP32_EXACT}[mode]
    w = wl.iid_workload("s", 6500 + n + k, [n], H, d, k, m, backward=False)
    fb = pu.run_forward(w, route=kb.ROUTE_SMALL)
    assert kb.kmip_test_route(fb.workspace) == kb.ROUTE_SMALL
    pu.check_forward(w, fb)
    w.K[::2] = w.K[n // 2]
    Q, K, V, dO, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, k, w.mode, route=kb.ROUTE_SMALL)
    b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score)


@pytest.mark.parametrize("n,H,d,k,mode,route", [
    (1024, 1, 32, 16, "fp32", SMALL), (2048, 1, 64, 16, "fp32", SMALL), (200, 64, 16, 32, "bf16", SMALL),
    (351, 8, 16, 16, "bf16", SMALL), (430, 32, 16, 32, "fp32", SMALL), (398, 64, 16, 7, "bf16", SMALL),   # a warp per row
    (1104, 16, 16, 16, "bf16", FILTER), (788, 64, 16, 24, "fp32", FILTER), (1389, 8, 16, 32, "bf16", FILTER),
    (2400, 1, 16, 8, "bf16", SMALL), (2700, 1, 16, 17, "fp32", SMALL)])                   # 16 rows of scores no longer fit a block
def test_a_lone_graph_with_many_heads_does_not_queue_for_whole_blocks(n, H, d, k, mode, route):
    """Where the one-graph kernel's blocks come in many waves, or selection is most of their work, a warp per row or the filter
    takes the call (H 64, 788 nodes, d 16, k 32: 375 us in the one-graph kernel, 214 in the filter)."""
    m = {"bf16": wl.MODE_BF16_TC, "fp32": wl.MODE_FP32_EXACT}[mode]
    w = wl.iid_workload("s", 6550 + n + k, [n], H, d, k, m, backward=False)
    Q, K, V, dO, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, k, w.mode)
    assert kb.kmip_test_route(a.workspace) == route
    pu.check_forward(w, a)
    b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert torch.equal(a.topk_score, b.topk_score) and (route != SMALL or torch.equal(a.topk_idx, b.topk_idx))


def test_one_graph_with_bad_offsets_is_reported():
    w = wl.iid_workload("s", 6600, [200], 1, 16, 4, wl.MODE_BF16_TC, backward=False)
    Q, K, V, dO, offs = pu.to_device(w)
    for bad in ([1, 200], [0, 199]):
        fb = kb.ForwardBuffers(200, 1, 1, 16, 4, w.mode, Q.device)
        assert kb.kmip_attn_forward(Q, K, V, torch.tensor(bad, dtype=torch.int32, device="cuda"), 4, w.mode, fb.out, fb.topk_idx,
                                    fb.topk_score, fb.workspace) == kb.KMIP_OK
        assert kb.kmip_last_status(fb.workspace) == kb.KMIP_ERR_BAD_OFFSETS


@pytest.mark.parametrize("n,H,d,k,mode", [(1, 1, 16, 1, "bf16"), (301, 1, 32, 16, "bf16"), (301, 3, 64, 16, "fp32"), (77, 1, 128, 15, "bf16"),
                                          (77, 1, 128, 16, "fp32"), (301, 1, 16, 17, "bf16"), (301, 1, 32, 64, "bf16"), (301, 1, 32, 65, "bf16"),
                                          (603, 1, 16, 7, "bf16")])
def test_rows_and_lists_by_half_warps(n, H, d, k, mode):
    """Softmax, weighted sum and backward pass with two rows (k <= 16) and two hit lists per warp: odd numbers of rows, k on both sides
    of half a warp, rows too wide for it; three keys that every query takes give lists that half a warp does not take (301 hits) and, at 603
    nodes, that a block reduces."""
    m = {"bf16": wl.MODE_BF16_TC, "fp32": wl.MODE_FP32_EXACT}[mode]
    w = wl.iid_workload("s", 6700 + n + k, [n], H, d, k, m, backward=True)
    if k >= 4:
        w.K[: 3] = wl.round_to_bf16(np.sign(w.Q.mean(axis=0, keepdims=True)) * 8.0)
        w.Q[:] = wl.round_to_bf16(np.abs(w.Q) * np.sign(w.Q.mean(axis=0, keepdims=True)))
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev)
    pu.check_forward(w, fb)
    pu.check_backward(w, fb, pu.run_backward(w, fb, dev))


@pytest.mark.parametrize("sizes", [[8192, 8191, 24385], [100, 9000, 0, 1, 7, 16384, 40, 8200, 1], [33000]])
def test_sweep_order_of_large_graphs(sizes):
    """The rows of a graph of at least 8192 rows are grouped by query (equal queries lie together), all others stay in order."""
    N, H, d, k = sum(sizes), 1, 16, 8
    g = torch.Generator().manual_seed(N)
    kind = torch.randint(0, 60, (N,), generator=g)
    Q = torch.randn(60, H, d, generator=g)[kind].bfloat16().cuda()
    K = torch.randn(N, H, d, generator=g).bfloat16().cuda()
    offs = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), dtype=torch.int32, device="cuda")
    fb = kb.forward(Q, K, K, offs, k, kb.KMIP_BF16_TC)
    order, _ = kb.kmip_test_sweep_order(fb.workspace, N, len(sizes), H, d, k, kb.KMIP_BF16_TC)
    order = np.asarray(order)
    lo = 0
    for n in sizes:
        part = order[lo:lo + n]
        if n < 8192:
            assert (part == np.arange(lo, lo + n)).all()
        else:
            assert (np.sort(part) == np.arange(lo, lo + n)).all()
            kinds = kind.numpy()[part]
            assert (kinds[1:] != kinds[:-1]).sum() < 60 * 60  # kinds that share a bucket may mix
            assert (kinds[1:] != kinds[:-1]).mean() < 0.25    # unsorted: 59 of 60 neighbours differ
        lo += n


@pytest.mark.parametrize("over", ["Q", "K", "both, shifted"])
@pytest.mark.parametrize("sizes,H,d,k,mode", [([3100], 1, 32, 16, wl.MODE_FP32_EXACT), ([200, 1, 300], 2, 16, 8, wl.MODE_FP32_EXACT),
                                              ([7000], 1, 16, 8, wl.MODE_FP32_EXACT), ([2900], 2, 64, 9, wl.MODE_BF16_TC),
                                              ([3000], 1, 32, 45, wl.MODE_BF16_TC), ([3100], 1, 32, 16, wl.MODE_BF16_TC),
                                              ([200, 1, 300], 2, 16, 8, wl.MODE_BF16_TC), ([33000], 1, 16, 8, "pruned")])
def test_out_may_lie_over_the_queries_or_keys(sizes, H, d, k, mode, over):
    """An in-place call: the same keys and outputs as a call with an array of its own, on every sweep, with a few rows that
    the filter cannot decide."""
    w = wl.iid_workload("p", 6400 + sum(sizes) + k, sizes, H, d, k, wl.MODE_BF16_TC if mode == "pruned" else mode, backward=False)
    if mode == "pruned":
        w.mode = kb.KMIP_BF16_TC_PRUNED
    w.Q[3] = 0.0
    Q, K, V, dO, offs = pu.to_device(w)
    ref = kb.forward(Q, K, V, offs, k, w.mode)
    fb = kb.ForwardBuffers(w.N, w.G, H, d, k, w.mode)
    n, gap = Q.numel(), 64                     # 64 elements: 16-byte aligned, not a row of every shape
    mem = torch.empty(2 * n + gap, dtype=Q.dtype, device="cuda")
    q_at, k_at = (gap, n + gap) if over != "K" else (n + gap, gap)
    qv, kv = (mem[at:at + n].view(Q.shape) for at in (q_at, k_at))
    qv.copy_(Q); kv.copy_(K)
    fb.out = mem[:n].view(Q.shape) if over == "both, shifted" else qv if over == "Q" else kv
    kb.forward(qv, kv, V, offs, k, w.mode, buffers=fb)
    if mode == wl.MODE_FP32_EXACT:
        assert torch.equal(fb.topk_idx, ref.topk_idx) and torch.equal(fb.topk_score, ref.topk_score) and torch.equal(fb.out, ref.out)
    pu.check_forward(w, fb, None if w.N < 10000 else wl.sample_rows(w, 256))


@pytest.mark.parametrize("n,d,k", [(40, 16, 32), (300, 32, 32), (700, 64, 5)])
def test_small_graphs_with_scores_that_overflow(n, d, k):
    """Scores of -infinity keep their slots empty, those of +infinity come first: what one warp per row does."""
    g = torch.Generator().manual_seed(n)
    Q, K, V = (torch.randn(n, 1, d, generator=g).cuda() for _ in range(3))
    Q[::3] = 1e20
    Q[::6] = -1e20
    K[1::2] = 1e20
    K[2, 0, 0] = float("nan")
    a = kb.forward(Q, K, V, None, k, kb.KMIP_FP32_EXACT)
    b = kb.forward(Q, K, V, None, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert n > 40 or bool((b.topk_idx[::6, 0, -1] < 0).all())
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score)
    assert torch.equal(a.out.nan_to_num(nan=7.0), b.out.nan_to_num(nan=7.0))


@pytest.mark.parametrize("sizes,H,d,k,mode,small", [
    ([60] * 255 + [20000], 1, 16, 8, "bf16", False), ([20000] + [60] * 255, 2, 16, 8, "fp32", False), ([60] * 100 + [9000] + [60] * 100, 1, 64, 8, "bf16", False),
    ([60] * 100 + [9000] + [60] * 100, 1, 64, 2, "bf16", False), ([60] * 255 + [9000], 1, 32, 2, "fp32", False), ([3000] * 5 + [0] * 1000, 2, 16, 8, "bf16", False),
    ([100] * 400 + [12000], 1, 32, 16, "bf16", False), ([100] * 400 + [12000], 1, 32, 16, "pruned", False),
    ([175] * 128, 4, 16, 8, "bf16", True), ([175] * 300, 1, 32, 8, "pruned", True), ([100] * 200 + [0, 1, 1500], 2, 16, 24, "fp32", True),
    ([468] * 60, 2, 16, 9, "bf16", True), ([469] * 60, 2, 16, 9, "bf16", False)])
def test_batches_of_unequal_graphs(sizes, H, d, k, mode, small):
    """The small-graph kernel takes a batch by the sum of the squared graph sizes, which the device alone knows, not by the mean
    size: a large graph among many tiny (or empty) ones goes to the sweep.  Either way the answer is that of one warp per
    row in fp32 (at k < 4 the tensor-core sweep's: the same keys up to scores within its rounding)."""
    m = {"bf16": kb.KMIP_BF16_TC, "fp32": kb.KMIP_FP32_EXACT, "pruned": kb.KMIP_BF16_TC_PRUNED}[mode]
    w = wl.iid_workload("u", 6500 + len(sizes) + d + k, sizes, H, d, k, wl.MODE_FP32_EXACT if mode == "fp32" else wl.MODE_BF16_TC, backward=False)
    w.mode = m
    Q, K, V, _, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, k, m)
    assert (kb.kmip_test_route(a.workspace) == kb.ROUTE_SMALL) == small
    if mode != "pruned" and k >= 4 or small:
        b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
        assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score)
    pu.check_forward(w, a, wl.sample_rows(w, 200))
    order, rows = kb.kmip_test_sweep_order(a.workspace, w.N, w.G, H, d, k, m)
    assert rows % 128 == 0 and (np.sort(order) == np.arange(w.N)).all()


@pytest.mark.parametrize("mode,sizes,d,k", [("fp32", [3300, 40, 3000], 64, 16), ("fp32", [2000], 16, 32), ("fp32", [1500], 32, 5),
                                            ("bf16", [3000], 128, 16)])
def test_lower_key_wins_among_thousands_of_ties(mode, sizes, d, k):
    """Keys that are copies of 50 vectors through the sweeps that rank groups of keys: the groups of a row are rescored in
    list order, and a key that ties with the k-th best must still displace one with a larger number."""
    fp32 = mode == "fp32"
    w = wl.iid_workload("t", 6600 + sum(sizes) + k, sizes, 2, d, k, wl.MODE_FP32_EXACT if fp32 else wl.MODE_BF16_TC, backward=False)
    w.K[:] = w.K[np.random.default_rng(5).integers(0, 50, w.N)]
    Q, K, V, _, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, k, w.mode, fp32_path=2 if fp32 else 0)
    b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    same = (a.topk_idx == b.topk_idx).all(-1)
    assert bool(same.all()) if fp32 else float(same.float().mean()) > 0.999   # bf16: sums in another order
