"""Plan construction beside work that is still running: it returns before that work has finished."""
import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import binding as B
    from paper_2609_22755_b200 import workloads as W

    return torch, B, W


def test_destroyed_plans_of_another_stream_are_not_waited_for(env):
    torch, B, W = env
    from paper_2609_22755_b200.api import NspAttention

    w = W.custom([700, 300], 8, 2, seed=81)
    e = NspAttention(w)
    e.load(W.make_tensors(w))
    e.forward()
    torch.cuda.synchronize()
    want = e.o.clone()
    B.nsp_trim()
    slow = torch.ones(1 << 28, device="cuda")
    a = torch.cuda.Stream()
    a.wait_stream(torch.cuda.current_stream())
    plans = [B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv) for _ in range(4)]
    with torch.cuda.stream(a):
        for _ in range(600):  # ~200 ms
            slow.mul_(1.0)
        running = torch.cuda.Event()
        running.record()
        for p in plans:
            B.nsp_attn_fwd(p, e.q, e.k, e.v, e.o, e.lse, e.scale)
    del p
    plans.clear()  # destroyed behind the slow work
    seen = []

    def construct():
        with torch.cuda.stream(torch.cuda.Stream()):
            seen.append((B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv), running.query()))

    t = threading.Thread(target=construct)
    t.start()
    t.join()
    assert not seen[0][1]
    e.o.fill_(0.0)
    torch.cuda.synchronize()
    e.plan = seen[0][0]
    e.forward()
    assert e.status()[0] == 0 and torch.equal(e.o, want)
