"""Calls enqueued back to back, with no synchronisation in between: the kernels of a call and of neighbouring calls are
launched with programmatic dependencies and reset their own work-list cursors, so every call has to find its
predecessor's results complete and its own cursors at zero."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,hq,hkv,head_dim", [
    ([64, 128, 256, 512], 8, 2, 128),      # every kernel on a few SMs: all of them overlap
    ([7, 100, 1, 128, 90], 4, 1, 64),      # first-tile kernels only
    ([129], 1, 1, 128),                    # one item per kernel
    ([4096, 300, 5, 900], 40, 8, 128),     # more items than SMs, still the small-batch launches
    ([8192, 129], 16, 2, 128),             # above the line: preprocess and main kernel launched unchained
])
def test_back_to_back_steps_equal_separate_ones(lengths, hq, hkv, head_dim):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import workloads as W
    from paper_2609_22755_b200.api import NspAttention

    w = W.custom(lengths, hq, hkv, seed=31, head_dim=head_dim)
    names = ("o", "lse", "dq", "dk", "dv")
    engines, want = [], []
    for seed in (31, 32):  # two plans and two sets of tensors that take turns
        e = NspAttention(w)
        e.load(W.make_tensors(w, seed=seed))
        torch.cuda.synchronize()
        e.forward()
        torch.cuda.synchronize()
        e.backward()
        torch.cuda.synchronize()
        assert e.status()[0] == 0
        engines.append(e)
        want.append({n: getattr(e, n).clone() for n in names})
    for _ in range(6):
        for e in engines:
            for n in names:
                getattr(e, n).fill_(float("nan"))
            e.ws.fill_(0xFF)  # NaN in the accumulator and delta: the call clears what it adds to
            e.step_device()
            e.step_device()
    torch.cuda.synchronize()
    for e, ref in zip(engines, want):
        assert e.status()[0] == 0
        for n in ("o", "lse", "dk", "dv"):
            assert torch.equal(getattr(e, n), ref[n]), n
        # dQ terms are added in any order in fp32, then rounded to bf16: at most one bf16 step (2^-8) of the value,
        # and 1e-5 of the largest where terms cancel
        a, b = e.dq.float(), ref["dq"].float()
        assert bool(((a - b).abs() <= 2.0 ** -7 * b.abs() + 1e-4 * b.abs().max()).all())
