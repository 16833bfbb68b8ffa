"""Plans built and dropped while their kernels still run: the memory of a destroyed plan goes to later plans, never while
the device still uses it. And the lists of plans at the edges of the list construction (many segments, ties of cost and
length, several group sizes, empty segments) against the oracle, built while other work is queued."""
import threading

import numpy as np
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


@pytest.mark.parametrize("lengths,hq,hkv", [
    ([16] * 8192, [8] * 8192, [2] * 8192),
    ([1] * 33 + [0] * 3 + [129, 128, 127, 0, 129], [4] * 41, [1] * 41),
    ([640, 640, 384, 640], [12, 12, 8, 8], [4, 4, 8, 8]),  # groups of 3, 3, 1, 1: equal costs across group sizes
    ([4000, 17, 4000, 256, 300], [256, 256, 6, 6, 6], [1, 1, 2, 2, 2]),
    ([0, 0, 0], [2, 2, 2], [1, 1, 1]),
])
def test_lists_match_the_oracle(env, lengths, hq, hkv):
    torch, B, W = env
    import oracle

    w = W.custom(lengths, hq, hkv)
    junk = torch.ones(1 << 28, device="cuda")
    for _ in range(4):
        junk.mul_(1.0)  # work queued on the caller's stream
    plan = B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv, w.head_dim)
    for p in (0, 1, 2):
        assert np.array_equal(B.nsp_plan_get(plan, p), oracle.plan_tiles(w.cu_seqlens, w.hq, w.hkv, 128, 128, p))


def test_new_plans_under_running_ones(env):
    torch, B, W = env
    from paper_2609_22755_b200.api import NspAttention

    rng = np.random.default_rng(5)
    loads = [W.custom(rng.integers(1, 1500, size=n).tolist(), 8, 2, seed=n) for n in (1, 2, 3, 5, 8, 13)]
    names = ("o", "lse", "dk", "dv")
    want = []
    for w in loads:
        e = NspAttention(w)
        e.load(W.make_tensors(w))
        e.step_device()
        torch.cuda.synchronize()
        assert e.status()[0] == 0
        want.append({n: getattr(e, n).clone() for n in names + ("dq",)})
    errors = []

    def loop(seed):
        try:
            order = np.random.default_rng(seed).permutation(np.tile(np.arange(len(loads)), 12))
            with torch.cuda.stream(torch.cuda.Stream()):
                engines = []
                for w in loads:
                    engines.append(NspAttention(w))
                    engines[-1].load(W.make_tensors(w))
                for i in order:  # a new plan for every step; the one before it is dropped while its kernels may run
                    w, e = loads[i], engines[i]
                    for n in names + ("dq",):
                        getattr(e, n).fill_(float("nan"))
                    e.plan = B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv, w.head_dim)
                    e.step_device()
                torch.cuda.current_stream().synchronize()
                for e, ref in zip(engines, want):
                    for n in names:
                        assert torch.equal(getattr(e, n), ref[n]), n
                    # dQ terms are added in any order in fp32, then rounded to bf16: see test_gpu_back_to_back_calls.py
                    a, b = e.dq.float(), ref["dq"].float()
                    assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-4 * b.abs().max()).all())
        except BaseException as ex:  # noqa: BLE001 - handed to the main thread
            errors.append(ex)

    threads = [threading.Thread(target=loop, args=(s,)) for s in (1, 2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    if errors:
        raise errors[0]


def test_memory_of_destroyed_plans_is_bounded_and_given_back(env):
    torch, B, W = env
    w = W.custom([1] * 20000, 32, 4)  # 13 MB of lists: a block of 16 MB, which is kept
    plan = lambda: B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv)
    plan().destroy()
    torch.cuda.synchronize()
    B.nsp_trim()
    used = lambda before: before - torch.cuda.mem_get_info()[0]
    free = torch.cuda.mem_get_info()[0]
    plans = [plan() for _ in range(8)]
    torch.cuda.synchronize()
    assert used(free) >= 8 * 13e6
    plans.clear()
    assert 13e6 <= used(free) <= 64 << 20  # some of them are kept
    kept = used(free)
    plans = [plan() for _ in range(2)]  # and used again
    assert used(free) == kept
    plans.clear()
    B.nsp_trim()
    assert used(free) <= 2 << 20
