"""Forward items run in pairs: two heads of an even group, or two neighbouring q tiles of one head of an odd group (one
head per KV head above all), the lower of which ends a key tile earlier and is staged behind the other's last product."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,hq,hkv,head_dim", [
    ([129, 256, 257, 384, 385, 512, 513], 3, 3, 128),  # 2 .. 5 tiles: paired tiles, single tiles, ragged upper tiles
    ([129, 256, 257, 384, 385, 512, 513], 3, 3, 64),
    ([1100, 128, 640], 5, 1, 128),                     # odd group
    ([3000], 1, 1, 128),                               # one head: long pairs, next round prefetched under an unequal one
    ([700, 300, 700], [3, 4, 1], [1, 2, 1], 64),       # odd and even groups in one list
    # first-tile items of two KV heads (more items than SMs): full tiles, ragged ones, packs, an odd head left over, and
    # groups of two and three before and behind them
    ([100, 128, 37, 90] * 15, 5, 5, 128),
    ([100, 128, 37, 90] * 15, 5, 5, 64),
    ([128, 64, 130] * 14, [4] * 3 + [6] * 36 + [3] * 3, [2] * 3 + [6] * 36 + [1] * 3, 128),
])
def test_pairs_every_element(lengths, hq, hkv, head_dim):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import parity_util as P
    from paper_2609_22755_b200 import workloads as W

    w = W.custom(lengths, hq, hkv, seed=51, head_dim=head_dim)
    run = P.GpuRun(w)
    run.forward()
    run.backward()
    assert run.status()[0] == 0
    P.compare_full(w, run.results(), P.oracle_full(w, run.host))


@pytest.mark.parametrize("head_dim", [128, 64])
def test_short_rounds_over_many_calls(head_dim):
    """Two-tile segments with one head per KV head: the shortest rounds of the general kernel, started while the first-tile
    kernel still runs. A lane of an MMA-issuing warp that fell behind the others used to miss a barrier phase about once in
    10^5 rounds; it waited until the wait limit ran out (two seconds) and the rest of its CTA's work was lost."""
    import time

    import numpy as np
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import workloads as W
    from paper_2609_22755_b200.api import NspAttention

    lengths = np.random.default_rng(3).integers(60, 300, size=300).tolist()
    w = W.custom(lengths, 16, 16, seed=52, head_dim=head_dim)
    e = NspAttention(w)
    e.load(W.make_tensors(w))
    e.forward()
    torch.cuda.synchronize()
    want = e.o.clone(), e.lse.clone()
    slowest = 0.0
    for _ in range(60):
        e.o.fill_(float("nan"))
        e.lse.fill_(float("nan"))
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(32):
            e.forward()
        torch.cuda.synchronize()
        slowest = max(slowest, time.perf_counter() - t)
        assert torch.equal(e.o, want[0]) and torch.equal(e.lse, want[1])
    assert e.status()[0] == 0
    assert slowest < 1.0, slowest  # 32 calls take about 0.02 s
