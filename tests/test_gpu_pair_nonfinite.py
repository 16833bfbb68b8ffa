"""How far values that are not finite reach in the backward pass of long segments: as far on CTA pairs as on single CTAs. A pair walks
the q tile of its first key tile with both key tiles, and where a segment has an odd number of key tiles its second CTA holds
keys of the next segment; neither may reach a result through a product with zeros."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = 17 * 128  # an odd number of whole key tiles


@pytest.mark.parametrize("name,token,value", [
    ("v", 3 * 128 + 5, float("nan")),      # the second key tile of a pair: dQ of the tile before it
    ("k", 3 * 128 + 5, float("inf")),
    ("do", 2 * 128 + 5, float("inf")),     # the q tile of the first key tile: dK, dV of the one behind it
    ("q", 2 * 128 + 5, float("nan")),
    ("k", L, float("nan")),                # the segment behind an odd last tile: dQ of that tile
    ("v", L + 100, float("inf")),
    ("do", L - 1, float("nan")),
])
def test_reach_of_nonfinite_values(name, token, value):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import parity_util as P
    from paper_2609_22755_b200 import workloads as W

    hq, hkv = 16, 4
    w = W.custom([L] * 20, hq, hkv, seed=53)
    host = W.make_tensors(w)
    clean = {n: t.clone() for n, t in host.items()}
    row = host[name].view(-1, hq if name in ("q", "do") else hkv, 128)
    row[token, 1, 7] = value
    got = []
    for deterministic in (False, True):  # the ordered additions run every segment on single CTAs
        run = P.GpuRun(w, tensors=clean, dq_dtype="f32", deterministic=deterministic)
        assert (run.B.nsp_plan_pair_items(run.plan)[0] > 0) == (not deterministic)
        run.forward()  # O and LSE of finite inputs
        for n in ("q", "k", "v", "do"):
            getattr(run, n).copy_(host[n])
        run.backward()
        assert run.status() == (0, 0, 0, 0)
        got.append(run.results())
    bad = 0
    for n in ("dq", "dk", "dv"):
        pair, single = (np.isfinite(r[n]) for r in got)
        bad += int((~single).sum())
        assert np.array_equal(pair, single), (n, int((~pair).sum()), int((~single).sum()))
        a, b = (r[n][single] for r in got)
        assert np.max(np.abs(a - b)) <= 2e-5 * np.max(np.abs(b)), n  # as in the pair tests: order of the additions
    assert bad > 0  # the planted value reaches something
