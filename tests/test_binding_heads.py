"""The head maps of the layout calls: what reaches the library, and what is refused on the way. No GPU: the library call is a
stand-in."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2609_22755_b200 import binding as B


@pytest.fixture
def calls(monkeypatch):
    seen = []

    class Library:
        def take(self, src, dst, tokens, heads, per_block, n, head_dim, dtype, first_head, stream):
            array = first_head if isinstance(first_head, ctypes.Array) else (ctypes.c_int32 * n).from_address(first_head)
            seen.append(list(array))
            return B.NSP_OK

        nsp_a2a_gather_heads = nsp_a2a_scatter_heads = take

    monkeypatch.setattr(B, "lib", Library)
    return seen


@pytest.mark.parametrize("call", [B.nsp_a2a_gather_heads, B.nsp_a2a_scatter_heads])
def test_head_maps(calls, call):
    x = torch.zeros(64)
    for heads in ([0, 2, 4], (0, 2, 4), np.array([0, 2, 4]), np.array([0, 9, 2, 9, 4])[::2], [0.0, 2.0, 4.0]):
        call(x, x, 1, 8, 2, 8, heads, stream=0)
    assert calls == [[0, 2, 4]] * 5
    for heads in ([0, 2 ** 32], [0, 2 ** 31], [-(2 ** 31) - 1]):
        with pytest.raises(OverflowError):
            call(x, x, 1, 8, 2, 8, heads, stream=0)
    assert len(calls) == 5
