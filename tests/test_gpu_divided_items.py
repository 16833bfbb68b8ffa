"""Backward items divided into parts that add their dK / dV in turn, and ragged key tiles written whole rows at a time:
every element against the oracle at the sizes where a division or a row pass can go wrong, and the same bits twice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,hq,hkv,head_dim", [
    ([1000], 4, 1, 128),            # 28 steps: two parts, ragged last tile
    ([2304], 1, 1, 128),            # one head: the parts are ranges of q tiles
    ([2000, 129, 257], 5, 1, 64),   # odd group: a part starts inside a q tile's heads
    ([100, 28, 90, 20, 128, 60], 16, 1, 128),  # first-tile items divided; packs, a full tile and a ragged one
    ([130, 31], 32, 2, 64),         # one-row last tile
])
def test_divided_items_every_element(lengths, hq, hkv, head_dim):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import parity_util as P
    from paper_2609_22755_b200 import workloads as W

    w = W.custom(lengths, hq, hkv, seed=41, head_dim=head_dim)
    run = P.GpuRun(w)
    run.forward()
    run.backward()
    assert run.status()[0] == 0
    res = run.results()
    P.compare_full(w, res, P.oracle_full(w, run.host))
    for _ in range(3):  # the turn counters are back at zero, and the order of the additions is fixed
        for t in (run.dq, run.dk, run.dv):
            t.fill_(float("nan"))
        run.backward()
        assert run.status()[0] == 0
        again = run.results()
        for n in ("dk", "dv"):
            assert np.array_equal(again[n], res[n]), n
    for dt in ("bf16",):  # bf16 dK / dV: the same rows, rounded (their tolerance: one bf16 rounding of each of two parts)
        low = P.GpuRun(w, tensors=run.host, dkv_dtype=dt)
        low.forward()
        low.backward()
        got = low.results()
        for n in ("dk", "dv"):
            assert np.max(np.abs(got[n] - res[n])) <= 2.0 ** -7 * np.max(np.abs(res[n])), n
