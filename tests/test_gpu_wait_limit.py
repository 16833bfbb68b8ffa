"""A wait limit that is long against every step of a kernel does not fail a healthy plan: the parts of a divided item wait for
one another, and that wait grows with the work before it."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,hq,hkv,head_dim", [
    ([128], 256, 1, 128),        # 64 parts of four heads, added one after the other
    ([128, 90], 256, 1, 64),     # a ragged tile: added row by row
    ([4500], 16, 1, 128),        # parts of ~70 steps
])
def test_parts_wait_longer_than_a_barrier(lengths, hq, hkv, head_dim):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import binding as B
    from paper_2609_22755_b200 import workloads as W
    from paper_2609_22755_b200.api import NspAttention

    e = NspAttention(W.custom(lengths, hq, hkv, seed=71, head_dim=head_dim))
    e.load(W.make_tensors(e.w))
    e.step_device()
    torch.cuda.synchronize()
    want = e.dk.clone(), e.dv.clone()
    B.nsp_plan_set_wait_limit(e.plan, 100_000)  # ten steps of the slowest kernel
    for _ in range(5):
        e.backward()
        assert e.status() == (0, 0, 0, 0)
        assert torch.equal(e.dk, want[0]) and torch.equal(e.dv, want[1])
