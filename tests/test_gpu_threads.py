"""Calls of different sizes from two host threads, each with a stream and buffers of its own.  What a kernel may use of shared
memory is state of the kernel, not of the call: a call that set it to its own size would take it from a larger one in
another thread, between that one's setting and its launch."""
import threading

import pytest
import torch

from paper_2604_03815_b200 import binding as kb

pytestmark = pytest.mark.gpu


def _calls(sizes, H, d, k, mode, backward):
    """A function that enqueues one forward (and backward) pass and returns the library's status codes."""
    N, dt = sum(sizes), kb.storage_dtype(mode)
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q, K, V, dO = (torch.randn(N, H, d, device="cuda", generator=gen).to(dt) for _ in range(4))
    offs = torch.tensor([0] + torch.tensor(sizes).cumsum(0).tolist(), dtype=torch.int32, device="cuda")
    fb, bb = kb.ForwardBuffers(N, len(sizes), H, d, k, mode), kb.BackwardBuffers(N, len(sizes), H, d, k, mode)

    def call(stream):
        rc = [kb.kmip_attn_forward(Q, K, V, offs, k, mode, fb.out, fb.topk_idx, fb.topk_score, fb.workspace, stream)]
        if backward:
            rc.append(kb.kmip_attn_backward(Q, K, V, offs, k, mode, fb.out, dO, fb.topk_idx, fb.topk_score, bb.dQ, bb.dK, bb.dV,
                                            bb.workspace, stream))
        return rc
    return call


@pytest.mark.parametrize("large,small,backward", [
    (([1184], 1, 64, 16, kb.KMIP_FP32_EXACT), ([600], 1, 64, 16, kb.KMIP_FP32_EXACT), False),              # one graph
    (([300] * 200, 4, 64, 8, kb.KMIP_FP32_EXACT), ([100] * 4, 4, 64, 8, kb.KMIP_FP32_EXACT), True),              # batches, hit lists
    (([9000], 8, 32, 8, kb.KMIP_BF16_TC_PRUNED), ([9000], 1, 16, 8, kb.KMIP_BF16_TC_PRUNED), False),       # pivots
], ids=["one_graph", "batch", "pruned"])
def test_calls_of_two_sizes_from_two_threads(large, small, backward):
    calls = [_calls(*large, backward), _calls(*small, backward)]
    seen = [set(), set()]
    gate = threading.Barrier(2)

    def work(t):
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.default_stream())
        gate.wait(timeout=60)
        for i in range(400):
            seen[t].update(calls[t](stream))
            if i % 50 == 49:
                stream.synchronize()
        stream.synchronize()

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert seen == [{kb.KMIP_OK}, {kb.KMIP_OK}]
