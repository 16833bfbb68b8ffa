"""Backward pass of long segments on CTA pairs: against the oracle and against the plan option whose dQ additions are ordered,
which runs every segment on single CTAs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(lengths, hq, hkv):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_22755_b200 import workloads as W

    return W.custom(lengths, hq, hkv, seed=43)


def _pairs(lengths, hq, hkv):
    """Items of the pair kernel where the rule takes every segment that is long enough: two key tiles each, per KV head."""
    hq, hkv = (np.broadcast_to(h, len(lengths)) for h in (hq, hkv))
    tiles = np.array([-(-x // 128) for x in lengths])
    long = (tiles >= 16) & (hq // hkv * tiles >= 32)
    return int(((tiles + 1) // 2 * hkv * long).sum()), int((tiles * hkv * ~long).sum())


# The pair kernel takes segments of 16 key tiles (32 with one head per KV head) and more, of a batch that fills the chip.
@pytest.mark.parametrize("lengths,hq,hkv,dkv_dtype", [
    ([2048] * 20, 16, 4, "f32"),                             # whole tiles, an even number of them
    ([2049] * 30, 8, 2, "f32"),                              # an odd number: the second CTA of the last pair has no keys
    ([4100, 3969, 4097, 3968, 200, 40, 4200] * 3, 8, 8, "f32"),  # one head per KV head, ragged tiles, segments just below
    ([2200, 1999, 1921] * 14 + [1920, 129], 24, 8, "bf16"),  # bf16 gradients, odd groups, segments just below
    ([4300, 3500, 100, 4299] * 4, 64, 1, "f32"),             # the start alignment of long items
    ([4096] * 8 + [1900, 1500, 1300], 32, 4, "f32"),         # the items that are left are divided
    ([2050, 2048] * 8 + [4000] * 6 + [300], [16] * 16 + [8] * 7, [4] * 16 + [1] * 7, "f32"),  # two runs
])
def test_pairs_against_single_ctas(lengths, hq, hkv, dkv_dtype):
    import parity_util as P
    from paper_2609_22755_b200 import binding as B

    w = _batch(lengths, hq, hkv)
    run = P.GpuRun(w, dq_dtype="f32", dkv_dtype=dkv_dtype)
    single = P.GpuRun(w, tensors=run.host, dq_dtype="f32", dkv_dtype=dkv_dtype, deterministic=True)
    dtype = B.NSP_F32 if dkv_dtype == "f32" else B.NSP_BF16
    n_pairs, n_left = _pairs(lengths, hq, hkv)
    assert n_pairs > 0 and B.nsp_plan_pair_items(run.plan, dtype) == (n_pairs, n_left)
    assert B.nsp_plan_pair_items(single.plan, dtype)[0] == 0
    got = []
    for r in (run, single):
        r.forward()
        for _ in range(2):
            for t in (r.dq, r.dk, r.dv):
                t.fill_(float("nan"))
            r.backward()
        assert r.status()[0] == 0
        got.append(r.results())
    _compare(*got, dkv_dtype)


def _compare(pairs, single, dkv_dtype):
    # The same products of the same operands; what differs is the order in which the tensor core adds and in which up to 32
    # tiles are added to a row of dQ, one fp32 rounding each: 32 * 2^-24 of the largest partial sum. bf16 results: one step.
    for n in ("dq", "dk", "dv"):
        tol = 2.0 ** -8 if n != "dq" and dkv_dtype == "bf16" else 2e-5
        assert np.max(np.abs(pairs[n] - single[n])) <= tol * np.max(np.abs(single[n])), n


def test_pairs_with_recomputed_segments():
    import parity_util as P
    import torch
    from paper_2609_22755_b200 import binding as B

    w = _batch([2049, 2048, 2300, 1000] * 6, 16, 4)
    flags = np.arange(24, dtype=np.uint8) % 3 == 0  # paired segments and others
    host, got = None, []
    for deterministic in (False, True):
        run = P.GpuRun(w, tensors=host, dq_dtype="f32", deterministic=deterministic)
        host = run.host
        assert (B.nsp_plan_pair_items(run.plan)[0] > 0) == (not deterministic)
        run.forward()
        cu = w.cu_seqlens
        for s in np.flatnonzero(flags):  # neither O nor LSE of a marked segment is read
            run.o[int(cu[s]) * 16 * 128:int(cu[s + 1]) * 16 * 128] = float("nan")
            run.lse[int(cu[s]) * 16:int(cu[s + 1]) * 16] = float("nan")
        ws = torch.empty(B.nsp_plan_recompute_ws_bytes(run.plan), dtype=torch.uint8, device=run.dev)
        B.nsp_attn_bwd_recompute(run.plan, flags.astype(np.uint8), run.q, run.k, run.v, run.o, run.do, run.lse, run.dq, run.dk,
                                 run.dv, w.softmax_scale, ws)
        assert run.status()[0] == 0
        got.append(run.results())
    assert all(np.isfinite(got[0][n]).all() for n in ("dq", "dk", "dv"))
    _compare(*got, "f32")


def test_pairs_against_the_oracle():
    import parity_util as P
    from paper_2609_22755_b200 import binding as B
    from paper_2609_22755_b200 import workloads as W

    L, n, hq, hkv = 3073, 16, 8, 2
    w = _batch([L] * n, hq, hkv)
    run = P.GpuRun(w)
    assert B.nsp_plan_pair_items(run.plan) == _pairs([L] * n, hq, hkv)
    run.forward()
    run.backward()
    assert run.status()[0] == 0
    res = run.results()
    s = n - 1  # the last segment: behind its end lies the end of the tensors
    one = W.custom([L], hq, hkv, seed=43)
    q, kv, lse = (slice(s * L * h * x, (s + 1) * L * h * x) for h, x in ((hq, 128), (hkv, 128), (hq, 1)))
    host = {k: run.host[k][kv if k in "kv" else q] for k in ("q", "k", "v", "do")}
    cut = {k: res[k][{"lse": lse, "dk": kv, "dv": kv}.get(k, q)] for k in res}
    P.compare_full(one, cut, P.oracle_full(one, host))


# With bf16 gradients the items that are left are not divided: a long one beside few pairs keeps the whole batch on single CTAs.
@pytest.mark.parametrize("lengths,hq,hkv,paired_bf16", [
    ([2048] * 14 + [1900] * 4, 32, 4, False),
    ([4096] * 8 + [1900], 32, 4, False),
    ([2048] * 96 + [1900], 32, 4, True),
    ([2048] * 20, 16, 4, True),  # nothing is left
])
def test_long_items_behind_the_pairs(lengths, hq, hkv, paired_bf16):
    from paper_2609_22755_b200 import binding as B

    w = _batch(lengths, hq, hkv)
    plan = B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv, w.head_dim)
    pairs, left = _pairs(lengths, hq, hkv)
    assert B.nsp_plan_pair_items(plan, B.NSP_F32) == (pairs, left)
    everything = sum(-(-x // 128) for x in lengths) * hkv
    assert B.nsp_plan_pair_items(plan, B.NSP_BF16) == ((pairs, left) if paired_bf16 else (0, everything))


def test_first_tile_kernel_beside_pairs():
    """Its items are not divided into more parts than one wave takes (as such parts 32 segments of 4,096 tokens took 112 us, whole 90)."""
    import parity_util as P
    from paper_2609_22755_b200 import binding as B

    w = _batch([4096] * 32, 32, 4)
    host, best = None, []
    for deterministic in (False, True):  # the ordered plan divides nothing
        run = P.GpuRun(w, tensors=host, deterministic=deterministic)
        host = run.host
        run.forward()
        B.nsp_plan_set_profiling(run.plan, True)
        times = []
        for _ in range(8):
            run.backward()
            times.append(B.nsp_plan_kernel_ms(run.plan, B.KERNEL_BWD_FIRST))
        best.append(min(times))
        del run
    assert best[0] <= 1.12 * best[1], best
