"""Batches of single-tile segments are bound by the first-tile kernels' latency per item: the achieved bytes per second against
a copy in the same process."""
import pytest

pytestmark = pytest.mark.gpu


def _best_ms(torch, f, n=5, rounds=6):
    best = 1e9
    f()
    for _ in range(rounds):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        for _ in range(n):
            f()
        end.record()
        torch.cuda.synchronize()
        best = min(best, start.elapsed_time(end) / n)
    return best


def test_backward_of_one_head_per_item():
    """1,024 segments of 128 tokens, a KV head per q head: 5.4 GB in 1.38 ms, 0.60 of the copy rate. Where the LSE loads of an
    item followed one another it was 1.64 ms, 0.50."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import workloads as W
    from paper_2609_22755_b200.api import NspAttention

    w = W.custom([128] * 1024, 16, 16)
    e = NspAttention(w)
    for t in (e.q, e.k, e.v, e.do):
        t.normal_()
    e.forward()
    a = torch.empty(1 << 30, dtype=torch.uint8, device="cuda")
    b = torch.empty_like(a)
    copy = 2 * a.numel() / _best_ms(torch, lambda: b.copy_(a))
    q, kv = w.q_elems(), w.kv_elems()
    # q, k, v, o, dO in, dQ out in bf16, dK and dV out in fp32, the LSE
    moved = 2 * (4 * q + 2 * kv) + 2 * 4 * kv + 4 * w.lse_elems()
    rate = moved / _best_ms(torch, e.backward)
    assert e.status()[0] == 0
    assert rate >= 0.55 * copy, (rate / copy, copy / 1e9)
