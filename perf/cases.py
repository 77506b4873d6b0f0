"""Performance cases of the k-MIP attention library: what its users run, through its public calls.

A case is a dict of plain values:

  kind   "core"   kmip_attn_forward (and kmip_attn_backward when train) on Q, K, V that are already there
         "layer"  KMIPSelfAttention, the whole layer of Eq. 2, with autograd when train
  mode   "bf16", "fp32" or "pruned" (the tensor-core mode with exact tile skipping)
  data   "iid"      Q, K, V iid N(0, 1)
         "cluster"  Q and K from a mixture of 64 Gaussian clusters (std 0.2), a point cloud's skewed scores
         "hubs"     iid, with 1 % of the keys of each graph scaled by 5 (heavily shared keys)
  graphs, lo, hi    number of graphs of the batch; node counts uniform in [lo, hi]
  H, d, k           heads, head width, keys kept per query
  d_model, drop     "layer" only: width of the node features, attention dropout
  train             forward and backward, or inference
"""
import math

import torch

from paper_2604_03815_b200 import binding as kb
from paper_2604_03815_b200.layer import KMIPSelfAttention

_MODES = {"bf16": kb.KMIP_BF16_TC, "fp32": kb.KMIP_FP32_EXACT, "pruned": kb.KMIP_BF16_TC_PRUNED}


def _core(name, mode, data, graphs, lo, hi, H, d, k, train):
    return {"name": name, "kind": "core", "mode": mode, "data": data, "graphs": graphs, "lo": lo, "hi": hi, "H": H, "d": d,
            "k": k, "train": train}


def _layer(name, mode, graphs, lo, hi, d_model, H, d, k, drop, train):
    return {"name": name, "kind": "layer", "mode": mode, "data": "iid", "graphs": graphs, "lo": lo, "hi": hi, "d_model": d_model,
            "H": H, "d": d, "k": k, "drop": drop, "train": train}


def listed():
    return [
        # one small graph in the reference precision (bit-exact selection): the smallest call, latency and launches
        _core("small_graph_fp32", "fp32", "iid", 1, 1024, 1024, 1, 32, 16, False),
        # a training step's attention on a mini-batch of molecule-sized graphs
        _core("minibatch_train", "bf16", "iid", 128, 50, 300, 4, 16, 8, True),
        # the whole layer on such a mini-batch with the attention dropout that graph-level tasks train with
        _layer("minibatch_layer_dropout", "bf16", 128, 50, 300, 64, 4, 16, 8, 0.5, True),
        # one point of the size study (one head, k = 10, the narrow head padded to 16): inference
        _core("study_31623_infer", "bf16", "iid", 1, 31623, 31623, 1, 16, 10, False),
        # the same study in fp32, where every score is an fp32 sum on the CUDA cores: training
        _core("study_100k_fp32_train", "fp32", "iid", 1, 100000, 100000, 1, 16, 10, True),
        # its runs with many keys kept
        _core("study_100k_k45_train", "bf16", "iid", 1, 100000, 100000, 1, 16, 45, True),
        # wider heads, an odd node count
        _core("wide_heads_train", "bf16", "iid", 1, 50001, 50001, 4, 64, 20, True),
        # a city-scale road network, attention only
        _core("city_100k_train", "bf16", "iid", 1, 100000, 100000, 4, 32, 16, True),
        # the whole layer on another city graph: projections, attention, output projection and their gradients
        _layer("city_layer_114001_train", "bf16", 1, 114001, 114001, 128, 4, 32, 15, 0.0, True),
        # a large point cloud, with the full search and with the exact tile skipping
        _core("pointcloud_500k_train", "bf16", "cluster", 1, 500000, 500000, 4, 32, 32, True),
        _core("pointcloud_500k_pruned_train", "pruned", "cluster", 1, 500000, 500000, 4, 32, 32, True),
        # a batch of four large graphs whose hub keys are selected by many queries: contention in dK and dV
        _core("hub_batch_train", "bf16", "hubs", 4, 200000, 200000, 8, 16, 16, True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# The most that a drawn case computes: score multiply-adds on the tensor cores, and on the CUDA cores.
_MOST_TC, _MOST_FP32, _MOST_LONG_LIST = 1.6e13, 1.6e11, 6.0e12


def _nodes(rng, lo, hi, H, d, most):
    return _log_int(rng, lo, min(hi, int(math.sqrt(most / (H * max(d, 16))))))


def draw(rng):
    what = rng.choice(["small", "minibatch", "minibatch_layer", "fp32", "long_list", "wide", "city", "city_layer", "cloud", "hubs"])
    train = rng.random() < 0.7
    if what == "small":
        n, H, d, k = _log_int(rng, 100, 6000), rng.choice([1, 2, 4]), rng.choice([16, 32, 64]), rng.randint(4, 32)
        c = _core("", rng.choice(["bf16", "fp32"]), "iid", 1, n, n, H, d, k, train)
    elif what == "minibatch":
        lo = rng.randint(10, 100)
        c = _core("", "bf16", "iid", rng.randint(16, 256), lo, lo + rng.randint(20, 400), rng.choice([1, 2, 4, 8]),
                  rng.choice([16, 32, 64]), rng.randint(3, 24), train)
    elif what == "minibatch_layer":
        lo = rng.randint(10, 100)
        c = _layer("", rng.choice(["bf16", "bf16", "fp32"]), rng.randint(16, 256), lo, lo + rng.randint(20, 400),
                   rng.choice([48, 64, 96, 128]), 4, rng.choice([10, 16, 24, 32]), rng.randint(3, 20), rng.choice([0.0, 0.5]), train)
    elif what == "fp32":
        H, d, k = rng.choice([1, 1, 2, 4]), rng.choice([16, 32, 64]), rng.randint(5, 32)
        n = _nodes(rng, 6000, 100000, H, d, _MOST_FP32)
        c = _core("", "fp32", "iid", 1, n, n, H, d, k, train)
    elif what == "long_list":
        H, d, k = rng.choice([1, 1, 2, 4]), rng.choice([16, 32]), rng.randint(33, 100)
        n = _nodes(rng, 10000, 300000, H, d, _MOST_LONG_LIST)
        c = _core("", "bf16", "iid", 1, n, n, H, d, k, train)
    elif what == "wide":
        H, d, k = rng.choice([1, 2, 4]), rng.choice([64, 128]), rng.randint(5, 32)
        n = _nodes(rng, 5000, 200000, H, d, _MOST_TC)
        c = _core("", "bf16", "iid", 1, n, n, H, d, k, train)
    elif what == "city":
        H, d, k = rng.choice([1, 2, 4, 8]), rng.choice([16, 32]), rng.randint(5, 32)
        n = _nodes(rng, 6000, 600000, H, d, _MOST_TC)
        c = _core("", "bf16", "iid", 1, n, n, H, d, k, train)
    elif what == "city_layer":
        d, k = rng.choice([10, 16, 32]), rng.randint(5, 20)
        n = _nodes(rng, 6000, 300000, 4, 32, _MOST_TC)
        c = _layer("", "bf16", 1, n, n, rng.choice([64, 128, 256]), 4, d, k, rng.choice([0.0, 0.0, 0.5]), train)
    elif what == "cloud":
        H, d, k = rng.choice([1, 2, 4]), rng.choice([16, 32]), rng.randint(10, 32)
        n = _nodes(rng, 33000, 500000, H, d, _MOST_TC)
        c = _core("", rng.choice(["bf16", "pruned"]), "cluster", 1, n, n, H, d, k, train)
    else:
        G, H, k = rng.randint(2, 6), rng.choice([4, 8]), rng.randint(8, 20)
        n = _nodes(rng, 5000, 150000, G * H, 16, _MOST_TC)
        c = _core("", "bf16", "hubs", G, max(1, n - n // 8), n, H, 16, k, train)
    c.pop("name")
    return c


def _sizes(case, gen_cpu):
    """Node counts of the batch: the same set for every seed of a case, in an order that the seed draws."""
    sizes = torch.randint(case["lo"], case["hi"] + 1, (case["graphs"],), generator=torch.Generator().manual_seed(case["graphs"]))
    return sizes[torch.randperm(case["graphs"], generator=gen_cpu)]


def _mean_square(case):
    """Expected square of a graph's node count."""
    lo, hi = case["lo"], case["hi"]
    n = hi - lo + 1
    return ((lo + hi) / 2) ** 2 + (n * n - 1) / 12


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen_cpu = torch.Generator().manual_seed(seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    sizes = _sizes(case, gen_cpu)
    offs_cpu = torch.zeros(case["graphs"] + 1, dtype=torch.int64)
    offs_cpu[1:] = torch.cumsum(sizes, 0)
    N, G, H, d, k = int(offs_cpu[-1]), case["graphs"], case["H"], case["d"], case["k"]
    offs = offs_cpu.to(torch.int32).to(dev)
    mode = _MODES[case["mode"]]
    dt = kb.storage_dtype(mode)

    def normal(*shape):
        return torch.randn(*shape, device=dev, generator=gen)

    if case["kind"] == "layer":
        layer = KMIPSelfAttention(case["d_model"], H, d, k, dtype=dt, device=dev, attn_dropout=case["drop"])
        with torch.no_grad():
            for lin in (layer.w_q, layer.w_k, layer.w_v, layer.w_o):
                lin.weight.copy_(normal(*lin.weight.shape) / math.sqrt(lin.in_features))
        layer.train(case["train"])
        x = normal(N, case["d_model"]).to(dt).requires_grad_(case["train"])
        d_y = normal(N, case["d_model"]).to(dt) if case["train"] else None
        return {"case": case, "layer": layer, "x": x, "d_y": d_y, "offs": offs, "seed": seed}

    if case["data"] == "cluster":
        centres = normal(64, H, d)
        at = centres[torch.randint(0, 64, (N,), device=dev, generator=gen)]
        Q, K = at + 0.2 * normal(N, H, d), at + 0.2 * normal(N, H, d)
    else:
        Q, K = normal(N, H, d), normal(N, H, d)
    if case["data"] == "hubs":
        for g in range(G):
            lo, n = int(offs_cpu[g]), int(sizes[g])
            K[lo + torch.randperm(n, device=dev, generator=gen)[:max(1, n // 100)]] *= 5.0
    Q, K, V = Q.to(torch.bfloat16).to(dt), K.to(torch.bfloat16).to(dt), normal(N, H, d).to(torch.bfloat16).to(dt)
    s = {"case": case, "Q": Q, "K": K, "V": V, "offs": offs, "k": k, "mode": mode, "fwd": kb.ForwardBuffers(N, G, H, d, k, mode, dev)}
    if case["train"]:
        s["d_out"] = normal(N, H, d).to(dt)
        s["bwd"] = kb.BackwardBuffers(N, G, H, d, k, mode, dev)
    return s


def _ok(rc):
    if rc != kb.KMIP_OK:
        raise kb.KmipError(rc, "kmip_attn")


def run(s):
    if s["case"]["kind"] == "layer":
        layer, x = s["layer"], s["x"]
        if not s["case"]["train"]:
            with torch.no_grad():
                return {"y": layer(x, s["offs"])}
        torch.default_generator.manual_seed(s["seed"])   # the dropout's draws: the same for the same inputs
        layer.zero_grad(set_to_none=True)
        x.grad = None
        y = layer(x, s["offs"])
        y.backward(s["d_y"])
        return {"y": y, "dx": x.grad, "dw_q": layer.w_q.weight.grad, "dw_k": layer.w_k.weight.grad,
                "dw_v": layer.w_v.weight.grad, "dw_o": layer.w_o.weight.grad}
    f = s["fwd"]
    _ok(kb.kmip_attn_forward(s["Q"], s["K"], s["V"], s["offs"], s["k"], s["mode"], f.out, f.topk_idx, f.topk_score, f.workspace))
    r = {"out": f.out, "topk_idx": f.topk_idx, "topk_score": f.topk_score}
    if s["case"]["train"]:
        b = s["bwd"]
        _ok(kb.kmip_attn_backward(s["Q"], s["K"], s["V"], s["offs"], s["k"], s["mode"], f.out, s["d_out"], f.topk_idx, f.topk_score,
                                  b.dQ, b.dK, b.dV, b.workspace))
        r.update(dQ=b.dQ, dK=b.dK, dV=b.dV)
    return r


def work(case):
    """Bytes of inputs read once and outputs written once; flops of the scores (2 d each), of the weighted sums
    (2 d per selected pair) and, when training, of dP, dQ, dK, dV (8 d per selected pair).  How many scores the pruned
    mode has to compute depends on the data, so there only the selected pairs count."""
    N = case["graphs"] * (case["lo"] + case["hi"]) / 2
    scores = case["graphs"] * case["H"] * _mean_square(case)
    H, d, k, train = case["H"], case["d"], case["k"], case["train"]
    e = 4 if case["mode"] == "fp32" else 2
    pairs = N * H * k
    flops = (0 if case["mode"] == "pruned" else 2 * d * scores) + 2 * d * pairs + (8 * d * pairs if train else 0)
    if case["kind"] == "layer":
        dm, inner = case["d_model"], H * d
        weights = 4 * dm * inner
        # x, y and the weights; with gradients also d_y, d_x, and the weights' gradients
        nbytes = e * (2 * N * dm + weights) * (2 if train else 1)
        flops += 2 * N * weights * (3 if train else 1)
    else:
        # Q, K, V, out, topk_idx, topk_score; with gradients also d_out, dQ, dK, dV
        nbytes = e * N * H * d * (8 if train else 4) + 8 * pairs
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what the library differs from itself by when the columns of the heads (and of x) are permuted, which puts
    every sum into another order.  That moves a few keys across the k-th place where two scores are within rounding of each
    other: such a row keeps another, equally good key, so single elements may be off by as much as they are large."""
    if case["mode"] == "fp32":
        return {"rel": 1e-5, "max": 3e-4, "differ": 1e-5}
    return {"rel": 1e-2, "max": 0.99, "differ": 4e-4}
