"""Many short items per CTA whose dK / dV tiles are staged in the operand buffers and written row by row (ragged tiles, bf16
gradients): the next item's loads overwrite the staged rows right behind the last read of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim", [128, 64])
@pytest.mark.parametrize("dkv_dtype", ["f32", "bf16"])
def test_staged_rows_are_not_overwritten_by_the_next_item(head_dim, dkv_dtype):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import parity_util as P
    from paper_2609_22755_b200 import workloads as W

    lengths = [129, 200, 255, 31, 128, 300, 1] * 8  # 8 KV heads: three items per SM in either kernel, most of them ragged
    w = W.custom(lengths, 8, 8, seed=61, head_dim=head_dim)
    run = P.GpuRun(w, dkv_dtype=dkv_dtype)
    run.forward()
    ref = P.oracle_full(w, run.host)
    first = None
    for _ in range(20):
        for t in (run.dk, run.dv):
            t.fill_(float("nan"))
        run.backward()
        assert run.status()[0] == 0
        res = run.results()
        for n in ("dk", "dv"):
            # bf16: two roundings of half a step (2^-8 of a value of at most the largest) each, on top of the usual bound
            step = 2.0 ** -7 * np.max(np.abs(ref[n])) if dkv_dtype == "bf16" else 0.0
            P.check(n, res[n], ref[n], max_abs_tol=P.MAX_ABS_TOL + step)
        if first is None:
            first = res
        for n in ("dk", "dv"):  # one fixed order of additions
            assert np.array_equal(res[n], first[n]), n


@pytest.mark.parametrize("head_dim", [128, 64])
@pytest.mark.parametrize("dkv_dtype", ["f32", "bf16"])
def test_last_tiles_of_few_rows(head_dim, dkv_dtype):
    """One row, a row short of a warp's 32, one past, and so on: warps and row passes without a valid row skip their part."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import parity_util as P
    from paper_2609_22755_b200 import workloads as W

    w = W.custom([129, 1, 159, 160, 161, 31, 192, 193, 225, 33, 255, 385], 4, 2, seed=62, head_dim=head_dim)
    run = P.GpuRun(w, dkv_dtype=dkv_dtype)
    run.forward()
    run.backward()
    assert run.status()[0] == 0
    res, ref = run.results(), P.oracle_full(w, run.host)
    for n in ("dk", "dv"):
        step = 2.0 ** -7 * np.max(np.abs(ref[n])) if dkv_dtype == "bf16" else 0.0  # two bf16 roundings, as above
        P.check(n, res[n], ref[n], max_abs_tol=P.MAX_ABS_TOL + step)
