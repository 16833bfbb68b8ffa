"""The work this library is used for, as cases that can be timed: packed variable-length causal GQA attention, forward
and backward, over one GPU's share of a nested sequence-parallel plan, and the layout steps around it.

A case describes a batch with plain values:
  work        "step"       forward and backward of one batch whose plan exists (micro-batches of the same shape)
              "forward"    the forward pass alone (evaluation, log-probabilities)
              "recompute"  forward, then the backward pass that recomputes the segments an activation budget left out
              "new_batch"  plan construction, forward and backward: every training iteration packs other lengths
              "layout"     the head gathers before and the head scatters behind the attention of a degree-d node
  segments    "lengths@hq/hkv; ..." segments written out, with the head counts this GPU has of them ("" = none)
  tail_*      a long-tailed degree-1 batch behind them: lognormal lengths around tail_median filling tail_tokens
  hq, hkv     heads of the model (of the tail's segments; of the whole tensors of a layout case)
"""
import math
import random

import numpy as np
import torch

from paper_2609_22755_b200 import binding as B
from paper_2609_22755_b200 import workloads as W
from paper_2609_22755_b200.api import NspAttention
from paper_2609_22755_b200.ulysses import NodeLayout

DEVICE = "cuda:0"


def _case(name, work, segments="", tail=(0, 1024, 1.3, 32768, 0), granularity=16, hq=32, hkv=4, head_dim=128, dq="bf16",
          dkv="f32", saved=0.0, degree=1):
    tokens, median, sigma, longest, seed = tail
    return {"name": name, "work": work, "segments": segments, "tail_tokens": tokens, "tail_median": median,
            "tail_sigma": sigma, "tail_longest": longest, "tail_seed": seed, "granularity": granularity, "hq": hq,
            "hkv": hkv, "head_dim": head_dim, "dq": dq, "dkv": dkv, "saved": saved, "degree": degree}


def listed():
    return [
        # the smallest call: four short sequences of a small model, launches and host time count
        _case("tiny_step", "step", "64,128,256,512@8/2", hq=8, hkv=2),
        # a small batch of odd lengths, an empty sequence, three head structures (GQA, MQA, MHA), fp32 dQ
        _case("ragged_step", "step", "1,17,0,127@8/2; 129,255,1000@4/1; 3,384@16/16", hq=8, hkv=2, dq="f32"),
        # one micro-batch as a training loop meets it: other lengths in every iteration, so the plan is part of it
        _case("new_batch_step", "new_batch", tail=(8192, 512, 1.2, 8192, 6), granularity=1),
        # the leaf of a tree: the many short samples of a long-tailed corpus, lengths as a tokenizer leaves them
        _case("leaf_batch_step", "step", tail=(131072, 432, 1.0, 8192, 1), granularity=1),
        # evaluation of a long-tailed batch: the forward pass alone
        _case("long_tail_forward", "forward", tail=(32768, 2048, 1.2, 16384, 7)),
        # the long-tailed 65,536-token batch at degree 1
        _case("long_tail_step", "step", tail=(65536, 1024, 1.3, 32768, 2)),
        # head dimension 64 and bf16 gradients, ragged long-tailed batch
        _case("head_dim_64_step", "step", tail=(65536, 1024, 1.3, 32768, 2), granularity=1, head_dim=64, dkv="bf16"),
        # a static packing: sixteen equal sequences
        _case("static_8k_step", "step", ",".join(["8192"] * 16) + "@32/4"),
        # one GPU's chain of a full tree over eight GPUs, with the activation budget of half of its attention outputs
        _case("full_tree_recompute", "recompute", "131072@4/1; 32768,16400@8/1; 8192,9744,4096,6160@16/2",
              tail=(16384, 1024, 1.2, 8192, 5), saved=0.5),
        # a model with 64 query heads: a long sequence at degree 4 beside a long-tailed batch
        _case("large_head_step", "step", "131072@16/1", tail=(131072, 4096, 1.0, 65536, 4), hq=64),
        # the largest: a 393,216-token sequence at degree 8 beside its degree-1 tail
        _case("nested_shard_step", "step", "393216@4/1", tail=(32768, 2048, 1.2, 16384, 3)),
        # what a degree-8 node does around the attention of that sequence: gathers of Q, K, V, dO, scatters of O, dQ,
        # and of the partial dK and dV of KV heads that two GPUs share
        _case("node_layout", "layout", "393216@4/1", degree=8),
    ]


_MOST_FLOPS = 5.5e14  # a little less than nested_shard_step


def draw(rng):
    """Another batch of the same ranges."""
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.1:
        degree = rng.choice([2, 4, 8])
        lengths = [degree * log(64, 393216 // degree // 4) for _ in range(rng.randint(1, 3))]
        hq, hkv = rng.choice([(32, 4), (64, 4), (8, 2)])
        return _drawn("layout", ",".join(map(str, lengths)) + "@%d/%d" % (hq // degree, max(1, hkv // degree)), hq=hq,
                      hkv=hkv, degree=degree, head_dim=rng.choice([128, 128, 64]))
    while True:
        hq, hkv = rng.choice([(8, 2), (32, 4), (32, 4), (64, 4), (16, 16)])
        work = rng.choice(["step", "step", "step", "forward", "new_batch", "recompute"])
        tokens = log(1024, 131072)
        groups = []
        if rng.random() < 0.4:  # a longer sequence at a higher degree
            degree = rng.choice([2, 4, 8])
            groups.append("%d@%d/%d" % (log(1024, 393216), max(hq // degree, 1), max(hkv // degree, 1)))
        c = _drawn(work, "; ".join(groups),
                   tail=(tokens, log(48, 8192), round(rng.uniform(0.3, 1.3), 2), max(64, min(tokens, 32768)), rng.randrange(1 << 20)),
                   granularity=rng.choice([1, 16]), hq=hq, hkv=hkv, head_dim=rng.choice([128, 128, 128, 64]),
                   dq=rng.choice(["bf16", "bf16", "f32"]), dkv=rng.choice(["f32", "f32", "bf16"]),
                   saved=round(rng.uniform(0.2, 0.8), 2) if work == "recompute" else 0.0)
        if work_flops(c) <= _MOST_FLOPS:
            return c


def _drawn(*a, **k):
    c = _case("", *a, **k)
    del c["name"]
    return c


# ---- from a case to its batch
def _batch(case):
    lengths, hq, hkv = [], [], []
    for group in filter(None, (g.strip() for g in case["segments"].split(";"))):
        ls, heads = group.split("@")
        for length in ls.split(","):
            lengths.append(int(length))
            hq.append(int(heads.split("/")[0]))
            hkv.append(int(heads.split("/")[1]))
    left, unit = case["tail_tokens"], case["granularity"]
    rng = random.Random(case["tail_seed"])
    while left > 0:
        x = case["tail_median"] * math.exp(case["tail_sigma"] * rng.gauss(0, 1))
        n = min(max(unit, unit * int(x / unit + 0.5)), case["tail_longest"], left)
        lengths.append(n)
        hq.append(case["hq"])
        hkv.append(case["hkv"])
        left -= n
    return W.custom(lengths, hq, hkv, head_dim=case["head_dim"], name="case")


def _marking(w, saved):
    """Save / recompute marks under an activation budget of that share of the attention outputs."""
    total = int((w.lengths * w.hq).sum()) * (2 * w.head_dim + 4)
    level = (w.hq.max() // w.hq).astype(np.int32)  # the SP degree of a segment's node
    return B.nsp_recompute_mark(w.cu_seqlens, w.hq, level, int(total * saved), w.head_dim)[0]


def _layout(case):
    lengths = [int(x) for x in case["segments"].split("@")[0].split(",")]
    return NodeLayout(lengths, case["degree"], 0, case["hq"], case["hkv"], case["head_dim"])


def prepare(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))

    def normal(n, dtype=torch.bfloat16):
        t = torch.empty(n, dtype=dtype, device=DEVICE)
        for a in range(0, n, 1 << 26):
            t[a:a + (1 << 26)] = torch.randn(min(1 << 26, n - a), generator=g, device=DEVICE)
        return t

    state = {"work": case["work"]}
    if case["work"] == "layout":
        lay = _layout(case)
        T, D, d = lay.t_loc, lay.head_dim, lay.degree
        state["layout"], state["out"] = lay, {}
        for name, kind in (("q", "q"), ("k", "kv"), ("v", "kv"), ("do", "q")):
            H, h_loc, _ = lay.heads(kind)
            state[name] = normal(T * H * D)
            state["out"][name] = torch.empty(d * T * h_loc * D, dtype=torch.bfloat16, device=DEVICE)
        for name, kind, dtype in (("o", "q", torch.bfloat16), ("dq", "q", torch.bfloat16), ("dk", "kv", torch.float32),
                                  ("dv", "kv", torch.float32)):
            H, h_loc, _ = lay.heads(kind)
            state[name] = normal(d * T * h_loc * D, dtype)
            state["out"][name] = torch.empty(T * H * D, dtype=dtype, device=DEVICE)
        return state
    w = _batch(case)
    eng = NspAttention(w, device=DEVICE, dq_dtype=case["dq"], dkv_dtype=case["dkv"])
    eng.q, eng.k, eng.v = normal(w.q_elems()), normal(w.kv_elems()), normal(w.kv_elems())
    if case["work"] != "forward":
        eng.do = normal(w.q_elems())
    state["batch"], state["engine"] = w, eng
    if case["work"] == "recompute":
        state["marks"] = _marking(w, case["saved"])
    return state


def run(state):
    if state["work"] == "layout":
        lay, out = state["layout"], state["out"]
        for name, kind in (("q", "q"), ("k", "kv"), ("v", "kv")):
            H, h_loc, first = lay.heads(kind)
            B.nsp_a2a_gather_heads(state[name], out[name], lay.t_loc, H, h_loc, lay.head_dim, first)
        H, h_loc, first = lay.heads("q")
        B.nsp_a2a_scatter_heads(state["o"], out["o"], lay.t_loc, H, h_loc, lay.head_dim, first)
        B.nsp_a2a_gather_heads(state["do"], out["do"], lay.t_loc, H, h_loc, lay.head_dim, first)
        for name, kind in (("dq", "q"), ("dk", "kv"), ("dv", "kv")):
            H, h_loc, first = lay.heads(kind)
            B.nsp_a2a_scatter_heads(state[name], out[name], lay.t_loc, H, h_loc, lay.head_dim, first)
        return out
    e = state["engine"]
    if state["work"] == "new_batch":
        w = state["batch"]
        e.plan = B.nsp_plan_tiles(w.cu_seqlens, w.hq, w.hkv, w.head_dim)  # the previous iteration's plan is dropped
    e.forward()
    if state["work"] == "forward":
        return {"o": e.o, "lse": e.lse}
    if state["work"] == "recompute":
        e.backward(recompute=state["marks"])
    else:
        e.backward()
    return {"o": e.o, "lse": e.lse, "dq": e.dq, "dk": e.dk, "dv": e.dv}


def work_flops(case):
    w = _batch(case)
    fwd, bwd = w.flops()
    if case["work"] == "forward":
        return float(fwd)
    if case["work"] == "recompute":
        again = _marking(w, case["saved"]).astype(bool)
        L = w.lengths
        return float(fwd + bwd + 4 * w.head_dim * int((w.hq * (L * (L + 1) // 2))[again].sum()))
    return float(fwd + bwd)


def work(case):
    if case["work"] == "layout":
        lay = _layout(case)
        row = lay.t_loc * lay.head_dim
        (hq, q_loc, _), (hkv, kv_loc, _) = lay.heads("q"), lay.heads("kv")
        q = hq + lay.degree * q_loc  # heads in and out
        kv = hkv + lay.degree * kv_loc
        return {"bytes": float(row * (2 * 4 * q + 2 * 2 * kv + 4 * 2 * kv)), "flops": 0.0}
    w = _batch(case)
    q, kv, lse = w.q_elems(), w.kv_elems(), w.lse_elems()
    forward = 2 * (q + 2 * kv) + 2 * q + 4 * lse
    backward = 2 * (3 * q + 2 * kv) + 4 * lse + (4 if case["dq"] == "f32" else 2) * q + 2 * (4 if case["dkv"] == "f32" else 2) * kv
    return {"bytes": float(forward if case["work"] == "forward" else forward + backward), "flops": work_flops(case)}


def tolerance(case):
    if case["work"] == "layout":
        # copies, and fp32 sums of two to four partial gradients in a fixed order
        return {"rel": 1e-6, "max": 1e-5}
    # bf16 inputs, P and dS, bf16 O and gradients. Against the same path in 64 bits on batches of up to 16,384 tokens the
    # outputs differ by 1.9e-3 .. 2.6e-3 (O, dQ, bf16 dK / dV) and by at most 0.046 of the larger of value and root
    # mean square; four times that.
    return {"rel": 9e-3, "max": 0.16}
