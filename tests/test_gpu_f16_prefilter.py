"""The half-precision prefilter of the tensor-core mode (head widths 16 and 32, k <= 32): the fp16
tensor-core scores stay inside the error bound the rescoring kernel relies on, and inputs built to
defeat a 11-bit filter - floods of near-ties, huge and tiny magnitudes, mixed scales per head - still
give the oracle's answer (rows the filter cannot decide are recomputed by the exact kernel)."""
import numpy as np
import pytest
import torch

from paper_2604_03815_b200 import workloads as wl

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2604_03815_b200 import binding as kb
    from tests import parity_util as pu


def _scale(n2max):
    """Power of two that puts sqrt(n2max) into [32, 64), as the conversion kernel chooses it."""
    if not n2max > 0:
        return 1.0
    m, e = np.frexp(np.sqrt(np.float32(n2max)))
    return float(np.ldexp(1.0, 6 - int(e)))


@pytest.mark.parametrize("d,spread", [(16, 1.0), (32, 1.0), (32, 300.0), (16, 1e-3)])
def test_fp16_scores_stay_inside_the_error_bound(d, spread):
    N, H = 700, 2
    w = wl.iid_workload("s", 5100 + d, [N], H, d, 4, wl.MODE_BF16_TC, input_scale=spread)
    w.K[::7] = wl.round_to_bf16(w.K[::7] * np.float32(4.0))          # a few heavy keys
    w.Q[5] = wl.round_to_bf16(w.Q[5] * np.float32(1e-3))             # a query far below the others
    Q, K, V, dO, offs = pu.to_device(w)
    S = torch.full((H, N, N), float("nan"), dtype=torch.float32, device="cuda")
    stats = torch.zeros((H, 4), dtype=torch.float32, device="cuda")
    ws = torch.empty(kb.kmip_attn_workspace_bytes(N, 1, H, d, 1, kb.KMIP_BF16_TC, kb.PASS_FORWARD),
                     dtype=torch.uint8, device="cuda")
    assert kb.kmip_test_f16_scores(Q, K, S, stats, ws) == kb.KMIP_OK
    assert kb.kmip_last_status(ws) == kb.KMIP_OK
    got = S.cpu().numpy().astype(np.float64)
    st = stats.cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    q64, k64 = w.Q.astype(np.float64), w.K.astype(np.float64)
    for h in range(H):
        qn2, kn2, ka2 = (q64[:, h] ** 2).sum(1), (k64[:, h] ** 2).sum(1), (k64[:, h, :16] ** 2).sum(1)
        # the statistics are upper bounds of the true maxima, and tight ones
        assert qn2.max() <= st[h, 0] <= qn2.max() * 1.001 and kn2.max() <= st[h, 1] <= kn2.max() * 1.001
        assert ka2.max() <= st[h, 2] <= ka2.max() * 1.001
        sq, sk = _scale(st[h, 0]), _scale(st[h, 1])
        exact = (q64[:, h] @ k64[:, h].T) * sq * sk
        nq, nqa = np.sqrt(qn2) * sq, np.sqrt((q64[:, h, :16] ** 2).sum(1)) * sq
        nk, nka = np.sqrt(st[h, 1]) * sk, np.sqrt(st[h, 2]) * sk
        r = 2.0 ** -11 * (1 + 2.0 ** -9)
        a = (r * nqa * nka if d == 32 else 0.0) + 2.0 ** -18 * nq * nk + 2.5e-5
        err = np.abs(got[h] - exact)
        bound = a[:, None] + r * np.abs(got[h])
        assert np.all(err <= bound), f"head {h}: fp16 score off by {(err - bound).max():.3e} beyond the bound"
        assert 32 <= np.sqrt(st[h, 1]) * sk < 64.1


def _check(w, min_identical=0.98):
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev, route=kb.ROUTE_FILTER)
    st = pu.check_forward(w, fb)
    st["redo"] = kb.kmip_attn_sweep_counters(fb.workspace)[4]
    if w.backward:
        st.update(pu.check_backward(w, fb, pu.run_backward(w, fb, dev)))
    assert st["identical_rows"] >= min_identical
    return st


@pytest.mark.parametrize("d,k", [(32, 32), (16, 16), (32, 8)])
def test_flood_of_near_ties_is_recomputed_exactly(d, k):
    """Keys are copies of a handful of vectors with perturbations far below fp16 resolution: hundreds of
    groups tie within the filter's error bound, the list of k + slack groups cannot hold them, and the
    rows must come back from the exact kernel with the oracle's answer (lowest key among equals)."""
    N, H = 3000, 2
    w = wl.iid_workload("s", 5200 + d + k, [N], H, d, k, wl.MODE_BF16_TC)
    base = w.K[:5].copy()
    w.K[:] = base[np.arange(N) % 5]
    w.K[::3, :, 0] = wl.round_to_bf16(w.K[::3, :, 0] * np.float32(1.0078125))   # one bf16 ulp on one element
    st = _check(w, 0.9)
    assert st["redo"] > 0      # the redo path really ran


def test_well_separated_scores_need_no_redo():
    st = _check(wl.make_config(3, N=6000))
    assert st["redo"] == 0


@pytest.mark.parametrize("scale_q,scale_k", [(1e-4, 1.0), (300.0, 200.0), (1e-3, 1e3), (3e-5, 3e-5)])
def test_extreme_magnitudes(scale_q, scale_k):
    """Values far outside fp16's range in both directions (bf16 holds them): the per-head scaling of the
    fp16 copies has to absorb them without overflow, and what underflows only loosens the filter."""
    w = wl.iid_workload("s", 5300, [2500, 40, 700], 2, 32, 16, wl.MODE_BF16_TC)
    w.Q[:] = wl.round_to_bf16(w.Q * np.float32(scale_q))
    w.K[:] = wl.round_to_bf16(w.K * np.float32(scale_k))
    w.K[:, 1] = wl.round_to_bf16(w.K[:, 1] * np.float32(64.0))       # heads on different scales
    dev = pu.to_device(w)
    fb = pu.run_forward(w, dev, route=kb.ROUTE_FILTER)
    # scores of this size are outside the absolute tolerances of check_forward: compare selections directly
    from oracle import kmip_oracle as oracle
    ref = oracle.forward(w.Q, w.K, w.V, w.graph_offsets, w.k)
    idx = fb.topk_idx.cpu().numpy()
    same = np.all(np.sort(idx, -1) == np.sort(ref["idx"], -1), axis=-1)
    assert same.mean() > 0.97
    _, exact = oracle.forward_given_idx(w.Q, w.K, w.V, idx)
    offs = w.graph_offsets.astype(np.int64)
    g = np.searchsorted(offs, np.arange(w.N), side="right") - 1
    keff = np.minimum(w.k, offs[g + 1] - offs[g])
    valid = np.arange(w.k)[None, None, :] < keff[:, None, None]
    kth = np.take_along_axis(ref["score"], np.maximum(keff - 1, 0)[:, None, None].repeat(w.H, 1), axis=2)[..., 0]
    worst = np.where(valid, exact, np.inf).min(axis=-1)
    assert np.all(worst >= kth - 1e-2 * np.abs(kth))
    assert np.all((idx == -1) == ~np.broadcast_to(valid, idx.shape))


def test_rows_with_one_dominant_and_many_tiny_queries():
    """One query row a million times larger than the rest sets the head's scale; the other rows' scaled
    scores sink towards fp16's subnormals, where the filter is loose but must stay correct."""
    w = wl.iid_workload("s", 5400, [4000], 2, 32, 16, wl.MODE_BF16_TC, input_scale=1.0 / np.sqrt(32.0))
    w.Q[17] = wl.round_to_bf16(w.Q[17] * np.float32(1e6))
    _check(w, 0.95)


@pytest.mark.parametrize("n_tied,k", [(1, 32), (5, 8), (48, 16), (60, 32), (1300, 16)])
def test_few_undecidable_rows(n_tied, k):
    """`n_tied` queries score equally on hundreds of keys (zero vectors: every score is 0), the others do not: from one
    row that the whole grid shares, over the most rows that are cut into parts, to a block and to a warp per row."""
    N, H, d = 2900, 1, 32
    w = wl.iid_workload("s", 5500 + n_tied + k, [N], H, d, k, wl.MODE_BF16_TC, input_scale=1.0 / np.sqrt(32.0))
    rows = (np.arange(n_tied) * 2) % N
    w.Q[rows] = 0.0
    st = _check(w, 0.98)
    assert st["redo"] == n_tied


@pytest.mark.parametrize("sizes,H,d,k", [([1536], 1, 16, 4), ([1537, 3, 0, 700], 1, 32, 5), ([2500], 2, 16, 12), ([127, 129, 2000], 2, 64, 9),
                                         ([5000], 1, 64, 32), ([3000], 1, 32, 17), ([9001], 1, 32, 31), ([40, 1, 700] * 3, 1, 16, 8),
                                         ([7000, 0, 130, 4000], 1, 16, 4), ([300, 2500, 17] * 2, 2, 64, 5)])
def test_fp32_through_the_filter_is_the_same_bit_for_bit(sizes, H, d, k):
    """fp32 storage, values that fp16 cannot hold exactly: the filter path (operand copies and lists in the output arrays)
    against the one-warp-per-row kernel, which scores every key in fp32 - the same keys in the same order and the same
    scores, bit for bit."""
    N = sum(sizes)
    g = torch.Generator().manual_seed(N + d + k)
    Q, K, V = (torch.randn(N, H, d, generator=g).cuda() for _ in range(3))
    Q[N // 2] *= 1e-3
    offs = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), dtype=torch.int32, device="cuda")
    a = kb.forward(Q, K, V, offs, k, kb.KMIP_FP32_EXACT, route=kb.ROUTE_FILTER)
    assert kb.kmip_test_route(a.workspace) == kb.ROUTE_FILTER
    b = kb.forward(Q, K, V, offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score) and torch.equal(a.out, b.out)


def test_fp32_near_ties_beyond_half_precision():
    """Keys that differ by a few fp32 ulps only: no fp16 score can tell them apart, the rows go to the exact kernel."""
    g = torch.Generator().manual_seed(5)
    N, d, k = 3000, 32, 16
    Q = torch.randn(N, 1, d, generator=g)
    K = torch.randn(5, 1, d, generator=g)[torch.arange(N) % 5] * (1 + 1e-6 * torch.randn(N, 1, 1, generator=g))
    Q, K, V = Q.cuda(), K.cuda(), torch.randn(N, 1, d, generator=g).cuda()
    a = kb.forward(Q, K, V, None, k, kb.KMIP_FP32_EXACT)
    assert kb.kmip_attn_sweep_counters(a.workspace)[4] > 0
    b = kb.forward(Q, K, V, None, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score) and torch.equal(a.out, b.out)


def test_graph_of_several_segments():
    """More than 2^19 keys: the entries of a row number their groups inside a segment, the kept ones carry its number along.
    Against dense fp32 scores of sampled rows; the best keys of every row are planted in the first and the last segment."""
    N, d, k = (1 << 19) + 70_001, 16, 6
    g = torch.Generator(device="cuda").manual_seed(11)
    Q, K, V = (torch.randn(N, 1, d, device="cuda", generator=g).to(torch.bfloat16) for _ in range(3))
    for j in (3, (1 << 19) - 1, 1 << 19, N - 1):
        K[j] = K[j] * 4
    fb = kb.forward(Q, K, V, None, k, kb.KMIP_BF16_TC)
    rows = torch.randint(0, N, (256,), device="cuda", generator=g)
    dense = Q[rows, 0].float() @ K[:, 0].float().T
    best = dense.topk(k, dim=1).values
    got = dense.gather(1, fb.topk_idx[rows, 0].long())
    assert torch.all((got - best).abs() <= 1e-4 * best.abs() + 1e-4)
    assert all(len(set(r)) == k for r in fb.topk_idx[rows, 0].tolist())


@pytest.mark.parametrize("sizes,H,d,k,mode", [([2048], 1, 16, 33, wl.MODE_BF16_TC), ([2049, 3, 0, 700], 1, 32, 45, wl.MODE_BF16_TC),
                                              ([1500, 1200], 2, 16, 64, wl.MODE_BF16_TC), ([127, 129, 2000], 1, 32, 72, wl.MODE_BF16_TC),
                                              ([40, 2500], 1, 16, 103, wl.MODE_BF16_TC), ([1024], 2, 32, 65, wl.MODE_FP32_EXACT),
                                              ([33000], 1, 16, 80, wl.MODE_BF16_TC)])
def test_long_lists_through_the_filter(sizes, H, d, k, mode):
    """32 < k <= 103: three and two query tiles per block, lists of more than one entry per lane, rows with fewer keys than
    k, rows in locality order; then half of the keys tied, so that every row is undecidable.  Both must be what one warp
    per row finds in fp32 (of bf16 values the same exact products in the same order)."""
    w = wl.iid_workload("l", 7100 + sum(sizes) + k, sizes, H, d, k, mode, backward=False)
    for tied in (False, True):
        if tied:
            w.K[::2] = w.K[1]
        Q, K, V, _, offs = pu.to_device(w)
        a = kb.forward(Q, K, V, offs, k, w.mode)
        assert kb.kmip_test_route(a.workspace) == kb.ROUTE_FILTER or (tied and w.N >= 33000)   # there all are swept again
        b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
        assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score)


@pytest.mark.parametrize("mode,d,k", [("fp32", 16, 12), ("fp32", 64, 8), ("bf16", 64, 20), ("bf16", 32, 45), ("bf16", 16, 16)])
@pytest.mark.parametrize("what", ["key", "key_inf", "key_nan", "query", "query_nan"])
def test_rows_beyond_the_range_of_the_copies(mode, d, k, what):
    """A key or query whose squared norm overflows has no half-precision copy under the scale that suits the others; its
    scores are finite all the same (or infinite, or not numbers), and the answer is what one warp per row finds in fp32."""
    N, H = 4000, 2
    g = torch.Generator().manual_seed(d + k)
    Q, K, V = (torch.randn(N, H, d, generator=g).to(torch.bfloat16).cuda() for _ in range(3))
    if what == "key": K[1234, 0] *= 1e20
    if what == "key_inf": K[1234, 0, 3] = float("inf")
    if what == "key_nan": K[1234, 0, 3] = float("nan")
    if what == "query": Q[77, 1] *= 1e20
    if what == "query_nan": Q[77, 1, 5] = float("nan")
    m = kb.KMIP_FP32_EXACT if mode == "fp32" else kb.KMIP_BF16_TC
    a = kb.forward(*(t.to(kb.storage_dtype(m)) for t in (Q, K, V)), None, k, m)
    redo = kb.kmip_attn_sweep_counters(a.workspace)[4]
    assert redo >= {"key": N, "key_inf": N, "query": 1}.get(what, 0) and redo < N + 100
    b = kb.forward(Q.float(), K.float(), V.float(), None, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    assert torch.equal(a.topk_idx, b.topk_idx) and torch.equal(a.topk_score, b.topk_score)
    if what == "key":
        assert int((a.topk_idx[:, 0, 0] == 1234).sum()) > N // 4


@pytest.mark.parametrize("sizes,H,d,k,mode,route", [
    ([7000], 1, 16, 12, "fp32", "ROUTE_TILED"), ([3300, 40, 3000], 2, 64, 16, "fp32", "ROUTE_TILED"), ([6500], 1, 64, 20, "bf16", "ROUTE_TENSOR_CORE"),
    ([3300, 40, 3000], 2, 32, 45, "bf16", "ROUTE_TENSOR_CORE"), ([6400], 1, 32, 100, "bf16", "ROUTE_TENSOR_CORE"), ([33000], 1, 64, 8, "bf16", "ROUTE_TENSOR_CORE"),
    ([6200], 1, 32, 80, "fp32", "ROUTE_FILTER"), ([5000], 1, 64, 20, "bf16", "ROUTE_FILTER")])
@pytest.mark.parametrize("what", ["ties", "heavy"])
def test_many_undecidable_rows_are_swept_again(sizes, H, d, k, mode, route, what):
    """Keys that are copies of 50 vectors, or one key a thousand times the others' size: the filter decides next to no row.
    From 48 blocks of rows on the sweep that scores everything takes over; smaller calls and those without such a sweep
    stay with the exact pass.  Equal scores go to the lower key in all of them."""
    fp32 = mode == "fp32"
    w = wl.iid_workload("t", 5600 + sum(sizes) + k, sizes, H, d, k, wl.MODE_FP32_EXACT if fp32 else wl.MODE_BF16_TC, backward=False)
    if fp32:                       # values that fp16 cannot hold exactly
        w.Q[:], w.K[:] = w.Q * np.float32(1.1), w.K * np.float32(1.1)
    if what == "ties":
        w.K[:] = w.K[np.random.default_rng(5).integers(0, 50, w.N)]
    else:
        w.K[w.N // 2] = w.K[w.N // 2] * 1024
    Q, K, V, _, offs = pu.to_device(w)
    a = kb.forward(Q, K, V, offs, k, w.mode)
    assert kb.kmip_attn_sweep_counters(a.workspace)[4] > w.N * H // 4
    assert kb.kmip_test_route(a.workspace) == getattr(kb, route)
    b = kb.forward(Q.float(), K.float(), V.float(), offs, k, kb.KMIP_FP32_EXACT, fp32_path=1)
    same = (a.topk_idx == b.topk_idx).all(-1)
    if route == "ROUTE_TENSOR_CORE":   # scores summed in another order: a tie within their rounding may go the other way
        assert float(same.float().mean()) > 0.999 and torch.allclose(a.topk_score, b.topk_score, rtol=1e-5, atol=1e-5)
    else:
        assert bool(same.all()) and torch.equal(a.topk_score, b.topk_score)
    if w.N < 10000:
        pu.check_forward(w, a, wl.sample_rows(w, 200))
