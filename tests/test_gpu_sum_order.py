"""The order in which a row's weighted sum and a key's hit list are added is a matter of the head width and the storage type
alone: term t goes to partial sum t mod g, g = 32 lanes / (lanes that share a row's 16-byte loads), each partial sum runs in
order, and the partial sums are added as a tree of neighbours.  Every kernel keeps to it, whichever route a call takes, however
many rows a warp does at a time and whatever list lies beside it, so a graph's results are the same bits in every batch.

With Q = 0 every score is 0 and every weight 1 / k exactly, so the sums can be repeated here in fp32, bit for bit: the product of
a power of two is exact and each addition rounds once."""
import numpy as np
import pytest
import torch

from paper_2604_03815_b200 import binding as kb
from paper_2604_03815_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def tree(part):
    while part.shape[0] > 1:
        part = part[0::2] + part[1::2]
    return part[0]


def ordered_sums(terms, groups):
    """terms [n, ..., D] float32 -> [..., D], in the documented order; a term of 0 leaves a partial sum as it is."""
    part = np.zeros((groups,) + terms.shape[1:], dtype=np.float32)
    for t in range(terms.shape[0]):
        part[t % groups] += terms[t]
    return tree(part)


CASES = [  # sizes of graphs below k are powers of two, so that their weights are exact too
    (1, 16, 8, [8, 9, 31, 300, 1, 64, 8, 8, 201, 17, 2, 33], "bf16"),      # two rows and two lists per warp, long beside short
    (1, 16, 16, [16, 33, 8, 128, 511], "fp32"),
    (3, 16, 4, [5, 70, 1, 12], "fp32"),
    (1, 32, 16, [16, 17, 300, 1, 129, 16, 16, 45], "bf16"),
    (1, 32, 8, [101, 8, 9, 64, 15], "fp32"),
    (1, 32, 32, [32, 100, 33], "bf16"),                                    # a row per warp
    (3, 64, 2, [3, 40, 7, 120], "fp32"),                                   # two rows per warp, one group of lanes each
    (1, 64, 16, [16, 90, 1, 31], "bf16"),
    (1, 128, 2, [3, 9, 40, 7], "bf16"),
    (1, 128, 16, [16, 50, 33], "fp32"),                                    # rows as wide as a warp's loads
    (1, 32, 16, [16] * 9400 + [300, 17], "bf16"),                          # more than 150 000 lists
    (1, 16, 64, [64, 65, 200, 64], "bf16"),
]


def problem(H, d, k, sizes, mode):
    """Q = 0, random K, V and dOut; the weight of a row's entries; the partial sums of a row or list."""
    m = {"bf16": wl.MODE_BF16_TC, "fp32": wl.MODE_FP32_EXACT}[mode]
    dt = kb.storage_dtype(m)
    N = sum(sizes)
    rng = np.random.default_rng(8100 + N + d)
    V, K, dO = (torch.from_numpy(rng.standard_normal((N, H, d)).astype(np.float32)).to("cuda", dt) for _ in range(3))
    offs = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)).cuda()
    weight = np.repeat((1.0 / np.minimum(sizes, k)).astype(np.float32), sizes)
    return torch.zeros_like(K), K, V, dO, offs, m, weight, 32 // (d // (16 // V.element_size()))


@pytest.mark.parametrize("H,d,k,sizes,mode", CASES)
def test_weighted_sums_run_in_one_order(H, d, k, sizes, mode):
    Q, K, V, dO, offs, m, weight, groups = problem(H, d, k, sizes, mode)
    routes = [{}]
    if mode == "fp32":
        routes.append({"fp32_path": 1})
    elif k <= 32:
        routes.append({"route": kb.ROUTE_TENSOR_CORE})
    v = V.float().cpu().numpy()
    for route in routes:
        fb = kb.forward(Q, K, V, offs, k, m, **route)
        idx = fb.topk_idx.cpu().numpy().transpose(2, 0, 1)                  # [k, N, H]
        w = np.where(idx >= 0, weight[:, None], np.float32(0))
        out = ordered_sums(w[..., None] * v[np.maximum(idx, 0), np.arange(H)], groups)
        assert torch.equal(fb.out, torch.from_numpy(out).to("cuda", V.dtype)), route


@pytest.mark.parametrize("H,d,k,sizes,mode", CASES)
def test_hit_lists_are_added_in_one_order(H, d, k, sizes, mode):
    """dV of a key: its hits in the order of the queries."""
    Q, K, V, dO, offs, m, weight, groups = problem(H, d, k, sizes, mode)
    N = sum(sizes)
    fb = kb.forward(Q, K, V, offs, k, m)
    bb = kb.backward(Q, K, V, offs, k, m, fb, dO)
    g, idx = dO.float().cpu().numpy(), fb.topk_idx.cpu().numpy()
    q, h, t = np.nonzero(idx >= 0)
    seg = idx[q, h, t].astype(np.int64) * H + h
    by = np.argsort(seg, kind="stable")
    q, h, seg = q[by], h[by], seg[by]
    count = np.bincount(seg, minlength=N * H)
    assert count.max() <= 512                                               # a longer list is a block's
    rank = np.arange(len(seg)) - np.repeat(np.cumsum(count) - count, count)
    part = np.zeros((groups, N * H, d), dtype=np.float32)
    for r in range(count.max()):
        at = rank == r
        part[r % groups, seg[at]] += weight[q[at], None] * g[q[at], h[at]]
    assert torch.equal(bb.dV, torch.from_numpy(tree(part).reshape(N, H, d)).to("cuda", V.dtype))
