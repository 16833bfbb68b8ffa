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


@pytest.mark.parametrize("lengths,head_dim", [
    ([16384] * 4, 64),    # no registers left on an SM
    ([16384] * 4, 128),   # no shared memory left
    ([128] * 4096, 128),  # the first-tile kernel
])
@pytest.mark.parametrize("captured", [False, True])
def test_construction_under_a_backward_pass(env, lengths, head_dim, captured):
    """The call returns while the pass still runs, and the first calls on the plan, plain or captured, find its lists."""
    torch, B, W = env
    from paper_2609_22755_b200.api import NspAttention

    names = ("o", "lse", "dk", "dv")
    w = W.custom([700, 300, 64, 5], 8, 2, seed=82)
    e = NspAttention(w)
    e.load(W.make_tensors(w))
    e.step_device()
    torch.cuda.synchronize()
    want = {n: getattr(e, n).clone() for n in names}
    big = NspAttention(W.custom(lengths, 32, 4, head_dim=head_dim))
    for t in (big.q, big.k, big.v, big.do):
        t.normal_()
    big.step_device()
    for n in names:
        getattr(e, n).fill_(float("nan"))
    busy = torch.cuda.Stream()
    busy.wait_stream(torch.cuda.current_stream())
    e.plan = None
    plans = [B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv) for _ in range(8)]  # leave memory for those below: no allocation there
    plans.clear()
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):
        for _ in range(3):
            big.backward()
        running = torch.cuda.Event()
        running.record()
    plans = [B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv) for _ in range(8)]  # some of them meet a kernel that leaves no room
    assert not running.query()
    graphs = []
    for p in plans:
        e.plan = p
        if captured:
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[-1]):
                e.step_device()
        else:
            e.step_device()
    for i, p in enumerate(plans):
        if captured:
            for n in names:
                getattr(e, n).fill_(float("nan"))
            graphs[i].replay()
        torch.cuda.synchronize()
        assert B.nsp_device_status(p) == (0, 0, 0, 0)
        for n in names:
            assert torch.equal(getattr(e, n), want[n]), n
    assert big.status()[0] == 0


def test_lists_read_while_they_are_being_built(env):
    torch, B, W = env
    import oracle
    from paper_2609_22755_b200.api import NspAttention

    big = NspAttention(W.custom([16384] * 4, 32, 4, head_dim=64))
    for t in (big.q, big.k, big.v, big.do):
        t.normal_()
    big.forward()
    torch.cuda.synchronize()
    busy = torch.cuda.Stream()
    with torch.cuda.stream(busy):
        big.backward()
    w = W.custom([700, 300, 64, 5], 8, 2)
    for _ in range(4):
        plan = B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv)
        for p in (0, 1, 2):
            assert (B.nsp_plan_get(plan, p) == oracle.plan_tiles(w.cu_seqlens, w.hq, w.hkv, 128, 128, p)).all()
    torch.cuda.synchronize()


def test_captured_plan_destroyed_before_others(env):
    """The memory of a plan that took part in a capture is not handed to later plans."""
    torch, B, W = env
    from paper_2609_22755_b200.api import NspAttention

    w = W.custom([700, 300, 64, 5], 8, 2, seed=83)
    e = NspAttention(w)
    e.load(W.make_tensors(w))
    e.step_device()
    torch.cuda.synchronize()
    names = ("o", "lse", "dk", "dv")
    want = {n: getattr(e, n).clone() for n in names}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        e.step_device()
    for _ in range(3):
        for n in names:
            getattr(e, n).fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert e.status()[0] == 0
        for n in names:
            assert torch.equal(getattr(e, n), want[n]), n
    del graph
    e.plan.destroy()
    e.plan = None
    plans = [B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv) for _ in range(4)]
    for p in plans:
        for n in names:
            getattr(e, n).fill_(float("nan"))
        e.plan = p
        e.step_device()
        torch.cuda.synchronize()
        assert e.status()[0] == 0
        for n in names:
            assert torch.equal(getattr(e, n), want[n]), n


@pytest.mark.parametrize("lengths,hq,hkv", [
    ([1] * 8192, [4] * 8192, [2] * 8192),  # 2^26 terms: positions summed on the device
    ([1] * 8193, [4] * 8193, [2] * 8193),  # counted on the host from here on
    ([130, 0, 260, 5] * 1800, [6] * 3600 + [4] * 3600, [2] * 7200),  # groups of 3 and 2, equal costs across them
    ([1] * 65535, [32] * 65535, [4] * 65535),  # memory that is not kept, its image not pinned
    ([129, 257] * 2600, [2] * 5200, [2] * 2600 + [1] * 2600),        # one head per group, and pairs of heads
])
def test_lists_of_many_segments(env, lengths, hq, hkv):
    torch, B, W = env
    import oracle
    import parity_util as P

    w = W.custom(lengths, hq, hkv, seed=84)
    plan = B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv)
    for p in (0, 1, 2):
        assert (B.nsp_plan_get(plan, p) == oracle.plan_tiles(w.cu_seqlens, w.hq, w.hkv, 128, 128, p)).all()
    run = P.GpuRun(w)  # the list of forward pairs, which nobody can read: through the results
    run.forward()
    assert run.status()[0] == 0
    res, bits = run.results(), {n: W.bf16_bits(run.host[n]) for n in ("q", "k", "v")}
    o, lse = oracle.attn_fwd(bits["q"], bits["k"], bits["v"], w.cu_seqlens, w.hq, w.hkv, w.head_dim, w.softmax_scale)
    P.check("o", res["o"], o)
    assert abs(res["lse"] - lse).max() <= P.LSE_ABS_TOL
