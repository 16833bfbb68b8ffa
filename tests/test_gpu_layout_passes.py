"""The head gathers and scatters at the edges of their four-token passes: fewer tokens than one pass, remainders, shared KV
heads (several gathered copies of a head, two and three partial gradients to add), launched back to back."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens", [1, 3, 37, 592, 20011])
@pytest.mark.parametrize("heads,per_block,first,head_dim,dtype", [
    (8, 2, [0, 2, 4, 6], 128, "bf16"),
    (2, 1, [0, 0, 1, 1], 128, "f32"),     # two partial sums per head
    (1, 1, [0, 0, 0], 64, "f32"),         # three
    (3, 1, [0, 2], 64, "bf16"),           # head 1 in no block
])
def test_gather_and_scatter(tokens, heads, per_block, first, head_dim, dtype):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import binding as B

    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(tokens)
    x = torch.randn(tokens, heads, head_dim, generator=g, device="cuda").to(dt)
    blocks = torch.empty(len(first), tokens, per_block, head_dim, dtype=dt, device="cuda")
    back = torch.full_like(x, 7.0)
    B.nsp_a2a_gather_heads(x, blocks, tokens, heads, per_block, head_dim, first)
    B.nsp_a2a_scatter_heads(blocks, back, tokens, heads, per_block, head_dim, first)  # reads what the gather wrote
    want = torch.stack([x[:, f:f + per_block] for f in first])
    assert torch.equal(blocks, want)
    for h in range(heads):
        parts = [want[p][:, h - f] for p, f in enumerate(first) if f <= h < f + per_block]
        if not parts:
            assert bool((back[:, h] == 7.0).all())
            continue
        total = parts[0] if len(parts) == 1 else sum((p.float() for p in parts[1:]), parts[0].float()).to(dt)
        assert torch.equal(back[:, h], total)
