"""The work that a user of this library has it do, as a list of measurable cases.

An attention case is one pass of one attention layer: the forward alone (inference, evaluation) or a training
pass, i.e. forward, Delta preprocess and backward, through one of the routes of the binding:

  plain          nova_attn_fwd, nova_attn_bwd_preprocess, nova_attn_bwd on [B,H,T,D] tensors
  exact          the same with nova_attn_bwd_preprocess_exact (peaked softmax rows)
  static         the same with nova_attn_bwd_static_scratch (callers that cannot allocate)
  deterministic  the same with nova_attn_bwd_deterministic (bitwise reproducible gradients)
  fused          the strided entry points on views of a fused projection output [B,T,3,H,D]

A loss-head case is one nova_lmhead_fwd: hidden states against the vocabulary matrix, with the logits stored
(training, scoring) or left out (evaluation of a loss only), from one row per sequence up to whole batches.

Buffers, the workspace among them, are allocated once, as a training loop keeps them.
"""
import math

import torch

from paper_2608_00029_b200 import nova_attn as na
from paper_2608_00029_b200 import nova_lmhead as nl

VOCAB = 50304  # GPT-2's vocabulary padded to a multiple of 64
STATIC_ELEMENTS = 8 << 20  # the built-in accumulator of the static route holds this many


def attn(name, route, B, H, T, D, causal=True, qk=1.0, do=1.0):
    c = {"op": "attn", "route": route, "B": B, "H": H, "T": T, "D": D, "causal": causal, "qk": qk, "do": do}
    return dict(c, name=name) if name else c


def lmhead(name, M, N, K, logits, ignored=0):
    c = {"op": "lmhead", "M": M, "N": N, "K": K, "logits": logits, "ignored": ignored}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: two heads of 64 tokens, all launch latency
        attn("tiny_train", "plain", 1, 2, 64, 64),
        # one layer of GPT-2 small at its training batch: the headline workload of the benchmark
        attn("gpt2_small_train", "plain", 8, 12, 1024, 64, do=1e-2),
        # four times that batch with a peaked softmax, which is what the exact Delta is for
        attn("large_batch_peaked_exact", "exact", 32, 12, 1024, 64, qk=2.0),
        # one layer of GPT-2 medium reading the fused projection output in place
        attn("gpt2_medium_fused", "fused", 8, 16, 1024, 64),
        # long context, head dimension 128: the largest attention call
        attn("long_context_train", "plain", 2, 12, 8192, 128),
        # many heads of dimension 128 at a ragged, ordinary length (packed documents)
        attn("wide_train_ragged", "plain", 4, 32, 1000, 128),
        # reproducible training, ragged
        attn("deterministic_train", "deterministic", 4, 12, 1500, 64),
        # prefill of one prompt of odd length
        attn("prefill_one_prompt", "forward", 1, 12, 777, 64),
        # an encoder's forward: no mask, short ragged sequences
        attn("encoder_forward", "forward", 16, 16, 333, 128, causal=False),
        # the loss head of a GPT-2-small training step: 8 x 1024 tokens, logits kept for the backward
        lmhead("lm_head_train", 8192, VOCAB, 768, True),
        # loss of an evaluation batch with unlabelled positions, nothing but the loss wanted
        lmhead("lm_head_eval", 3001, VOCAB, 1024, False, ignored=7),
        # scoring one position of each of 24 sequences: a few rows against the whole vocabulary
        lmhead("lm_head_few_rows", 24, VOCAB, 768, True),
    ]


def _log_int(rng, low, high):
    return min(high, max(low, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def _attn_flops(c):
    pairs = c["T"] * (c["T"] + 1) / 2 if c["causal"] else c["T"] ** 2
    return c["B"] * c["H"] * pairs * c["D"] * (4.0 if c["route"] == "forward" else 14.0)


def draw(rng):
    """One more case of the same ranges, none dearer than the long-context one."""
    if rng.random() < 0.25:
        # a few rows, or a whole batch; vocabularies of ordinary sizes (multiples of 8), GPT-2's widths
        M = _log_int(rng, 1, 8192)
        N = 8 * _log_int(rng, 125, 8000)
        K = 64 * rng.choice([1, 8, 12, 16, 20, 25])
        return lmhead(None, M, N, K, rng.random() < 0.7, ignored=rng.choice([0, 0, 7]))
    route = rng.choice(["plain", "plain", "plain", "fused", "fused", "exact", "static", "deterministic", "forward",
                        "forward", "forward"])
    T = _log_int(rng, 16, 8192)
    if rng.random() < 0.4 and T >= 128:
        T = T // 128 * 128
    c = attn(None, route, _log_int(rng, 1, 64), rng.choice([1, 2, 5, 8, 12, 16, 20, 25, 32]), T,
             rng.choice([64, 64, 128]), causal=rng.random() < 0.75, qk=2.0 if route == "exact" else 1.0,
             do=rng.choice([1.0, 1e-2]))
    most = STATIC_ELEMENTS if route == "static" else 4 * STATIC_ELEMENTS
    for dim in ("B", "H", "T"):  # what would be dearer, or too large for the route, gets fewer sequences, then heads
        while c[dim] > 1 and (_attn_flops(c) > 9e11 or c["B"] * c["H"] * c["T"] * c["D"] > most):
            c[dim] //= 2
    return c


def _randn(g, shape, factor):
    x = torch.randn(shape, dtype=torch.float32, generator=g, device="cuda")
    return (x * factor if factor != 1.0 else x).to(torch.bfloat16)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case}
    if case["op"] == "lmhead":
        M, N, K = case["M"], case["N"], case["K"]
        # hidden states after the final normalisation; the embedding matrix at GPT-2's initialisation scale
        s["X"], s["W"] = _randn(g, (M, K), 1.0), _randn(g, (N, K), 0.02)
        t = torch.randint(0, N, (M,), generator=g, device="cuda").to(torch.int32)
        if case["ignored"]:
            t[:: case["ignored"]] = -1
        s["targets"] = t
        s["logits"] = torch.empty((M, N), dtype=torch.bfloat16, device="cuda") if case["logits"] else None
        s["lse"], s["loss"] = (torch.empty(M, dtype=torch.float32, device="cuda") for _ in range(2))
        s["ws"] = torch.empty(nl.nova_lmhead_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
        return s
    B, H, T, D, route = case["B"], case["H"], case["T"], case["D"], case["route"]
    s["scale"] = 1.0 / math.sqrt(D)
    names = ("q", "k", "v", "do") if route != "forward" else ("q", "k", "v")
    factors = {"q": case["qk"], "k": case["qk"], "v": 1.0, "do": case["do"]}
    s["lse"] = torch.empty((B, H, T), dtype=torch.float32, device="cuda")
    if route == "fused":
        qkv = torch.empty((B, T, 3, H, D), dtype=torch.bfloat16, device="cuda")
        for i, n in enumerate("qkv"):
            qkv[:, :, i] = _randn(g, (B, T, H, D), factors[n])
            s[n] = qkv[:, :, i].permute(0, 2, 1, 3)
        s["do"] = _randn(g, (B, T, H, D), factors["do"]).permute(0, 2, 1, 3)
        s["o"] = torch.empty((B, T, H, D), dtype=torch.bfloat16, device="cuda").permute(0, 2, 1, 3)
        s["dqkv"] = torch.empty_like(qkv)
        for i, n in enumerate(("dq", "dk", "dv")):
            s[n] = s["dqkv"][:, :, i].permute(0, 2, 1, 3)
    else:
        for n in names:
            s[n] = _randn(g, (B, H, T, D), factors[n])
        for n in ("o", "dq", "dk", "dv") if route != "forward" else ("o",):
            s[n] = torch.empty((B, H, T, D), dtype=torch.bfloat16, device="cuda")
    if route != "forward":
        s["delta"] = torch.empty_like(s["lse"])
        if route in ("plain", "exact", "fused"):
            s["ws"] = torch.empty(na.nova_attn_bwd_workspace_bytes(B, H, T, D), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    c = s["case"]
    if c["op"] == "lmhead":
        nl.nova_lmhead_fwd(s["X"], s["W"], s["targets"], s["logits"], s["lse"], s["loss"], s["ws"])
        return [t for t in (s["logits"], s["lse"], s["loss"]) if t is not None]
    route, scale, causal = c["route"], s["scale"], c["causal"]
    q, k, v, o, lse = s["q"], s["k"], s["v"], s["o"], s["lse"]
    if route == "fused":
        na.nova_attn_fwd_strided(q, k, v, o, lse, scale, causal)
        na.nova_attn_bwd_preprocess_strided(o, s["do"], s["delta"])
        na.nova_attn_bwd_strided(q, k, v, s["do"], lse, s["delta"], s["dq"], s["dk"], s["dv"], scale, causal, s["ws"])
        return [o, lse, s["delta"], s["dqkv"]]
    na.nova_attn_fwd(q, k, v, o, lse, scale, causal)
    if route == "forward":
        return [o, lse]
    do, delta, dq, dk, dv = s["do"], s["delta"], s["dq"], s["dk"], s["dv"]
    if route == "exact":
        na.nova_attn_bwd_preprocess_exact(q, k, v, do, lse, delta, scale, causal)
    else:
        na.nova_attn_bwd_preprocess(o, do, delta)
    if route == "deterministic":
        na.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, dq, dk, dv, scale, causal)
    elif route == "static":
        na.nova_attn_bwd_static_scratch(q, k, v, o, do, lse, delta, dq, dk, dv, scale, causal)
    else:
        na.nova_attn_bwd(q, k, v, o, do, lse, delta, dq, dk, dv, scale, causal, s["ws"])
    return [o, lse, delta, dq, dk, dv]


def work(case):
    """Inputs read once, outputs written once; only the kept (query, key) pairs count: two contractions in the
    forward, five in the backward (the exact Delta and the second kernel of the deterministic route recompute
    some, which the result does not need)."""
    if case["op"] == "lmhead":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (M * K + N * K) + 4 * M + (2 * M * N if case["logits"] else 0) + 8 * M,
                "flops": 2.0 * M * N * K}
    rows = case["B"] * case["H"] * case["T"]
    n = rows * case["D"]
    if case["route"] == "forward":
        return {"bytes": 2 * 4 * n + 4 * rows, "flops": _attn_flops(case)}
    return {"bytes": 2 * 8 * n + 2 * 4 * rows, "flops": _attn_flops(case)}


def tolerance(case):
    """About four times the distance of the outputs from the same arithmetic in 64 bits. Attention: 2.9e-3 (bf16
    operands and results; the largest over the root mean square 0.13, a gradient of the first tokens, at T = 6400).
    Loss head: 1.7e-3 and 3.9e-3 for the bf16 logits, 2e-7 for the 32-bit statistics."""
    if case["op"] == "attn":
        return {"rel": 1e-2, "max": 0.4}
    return {"rel": 7e-3, "max": 1.6e-2} if case["logits"] else {"rel": 1e-5, "max": 1e-4}
