"""GPU parity: the CUDA path (through the C ABI) against the fp64 oracle on the same seeded inputs.

Bounds: |gpu - ref| <= 1e-2 + 1e-2|ref| for O and LSE (and Delta), <= 2e-2 + 2e-2|ref| for dQ, dK, dV,
element by element, plus relative-RMS bounds of 5e-3 / 1e-2 because the absolute terms are weak where
the reference is small.
"""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

from paper_2608_00029_b200 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _harness():
    import gpu_harness
    return gpu_harness


# name -> which preprocess produces Delta.  The GPU runs the full configuration and the oracle checks
# EVERY head of it.  The peaked-softmax configuration is checked against the stated bounds with the exact
# Delta; rowsum(dO * O) on it is covered by the next test.
FIVE = [("tiny", False), ("gpt2_small", False), ("gpt2_small_large_batch", True), ("gpt2_medium", False),
        ("long_context", False)]


@pytest.mark.parametrize("name,exact_delta", FIVE)
def test_five_configs_match_oracle(name, exact_delta):
    h = _harness()
    cfg = W.CONFIGS[name]
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, cfg.causal, exact_delta=exact_delta)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, cfg.causal)
    errs = h.compare(h.select_heads(got, None), ref, label=f"{name}: ", dO=ref["dO_in"])
    print(name, {k: f"{v:.2e}" for k, v in errs.items()})
    # properties that hold at any size
    dK = W.widen(got["dK"])
    dK_abs = np.abs(dK).sum(2)
    assert (np.abs(dK.sum(2)) <= 2e-2 * dK_abs + 1e-3).all(), "sum_j dK_j should vanish per head"
    assert all(torch.isfinite(t.float()).all() for t in got.values())


# Largest |err| / (2e-2 + 2e-2|ref|) over all 384 heads of the peaked configuration when Delta comes from
# rowsum(dO * O).  Measured on the GPU (B200): dQ 2.136 (1516 of 25.2 M elements beyond 1x, on 312 heads),
# dK 2.165 (748 elements, 274 heads), dV 0.724 (none).  A float64 emulation of all 384 heads in which only O
# (inside Delta), dS and the results are rounded to bf16 gives 2.05 / 2.02 (863 / 320 elements): the excess
# belongs to the route, not to the kernels.  The bound is the measured figure plus a margin of about 0.25.
ROWSUM_ROUTE_FACTOR = 2.4


def test_peaked_config_with_rowsum_delta():
    """Peaked softmax through the three calls in their stated order (forward, rowsum preprocess, backward),
    all heads.  The bf16 rounding of O alone (see test_delta_precision.py for the arithmetic, no GPU
    involved) pushes some dQ/dK elements past 2e-2 + 2e-2|ref|: the test prints how many of which tensor
    and by how much, and holds the route to the measured excess plus a margin, with the usual relative RMS."""
    import tolerance as tol
    h = _harness()
    cfg = W.CONFIGS["gpt2_small_large_batch"]
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, True, exact_delta=False)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, True)
    sel = h.select_heads(got, None)
    for name in ("dQ", "dK", "dV"):
        n_bad, worst, n = tol.violation_stats(sel[name], ref[name], tol.BWD_ATOL, tol.BWD_RTOL)
        per_head = (np.abs(sel[name] - ref[name]) > tol.BWD_ATOL + tol.BWD_RTOL * np.abs(ref[name])).any(axis=(2, 3))
        print(f"large_batch/rowsum {name}: {n_bad} of {n} elements beyond 1x the bound, on {int(per_head.sum())} of "
              f"{per_head.size} heads; largest error / bound = {worst:.3f}")
    h.compare(sel, ref, label="large_batch/rowsum: ", dO=ref["dO_in"], bwd_factor=ROWSUM_ROUTE_FACTOR)


def test_exact_delta_matches_jacobian_definition():
    """nova_attn_bwd_preprocess_exact against the oracle's Delta = sum_j P_ij dP_ij, tight bound."""
    h = _harness()
    for (B, H, T, D, causal) in [(1, 2, 64, 64, True), (1, 2, 333, 64, True), (2, 1, 256, 128, False),
                                 (1, 2, 1024, 64, True)]:
        cfg = W.AttnConfig("d", B=B, H=H, T=T, D=D, seed=T + D, causal=causal, qk_factor=2.0)
        Q, K, V, dO = W.make_inputs(cfg)
        got = h.run_gpu(Q, K, V, dO, cfg.scale, causal, exact_delta=True)
        ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal)
        err = np.abs(W.widen(got["Delta"]) - ref["Delta"])
        bound = 2e-3 + 2e-3 * np.abs(ref["Delta"])
        assert (err <= bound).all(), f"T={T} D={D}: exact Delta max err {err.max():.3e}"


def test_backward_alone_from_oracle_forward():
    """Feeds the backward with the oracle's own O and LSE (rounded to bf16 / fp32) to isolate it."""
    h = _harness()
    cfg = W.CONFIGS["gpt2_small"].replace(B=1, H=3, T=512)
    Q, K, V, dO = W.make_inputs(cfg)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, True)
    O_in = torch.tensor(ref["O"]).to(torch.bfloat16)
    LSE_in = torch.tensor(ref["LSE"]).to(torch.float32)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, True, O_in=O_in, LSE_in=LSE_in)
    h.compare(h.select_heads(got, None), ref, label="bwd-only: ", dO=ref["dO_in"])


EDGE = [
    # B, H, T, D, causal
    (1, 1, 1, 64, True),
    (2, 1, 1, 128, True),
    (1, 2, 17, 64, True),
    (1, 2, 65, 64, True),
    (2, 2, 129, 64, True),
    (1, 3, 200, 64, False),
    (1, 2, 256, 64, False),
    (1, 2, 300, 128, True),
    (1, 2, 256, 128, True),
    (1, 1, 384, 128, False),
    (1, 1, 333, 128, False),
    (3, 1, 640, 64, True),
    (1, 1, 127, 64, True),      # one short of a tile
    (1, 1, 128, 128, True),     # exactly one tile: the diagonal tile only
    (1, 2, 255, 128, False),
    (40, 8, 64, 64, True),      # many short work items: more items than SMs, one tile each
    (5, 30, 129, 64, True),     # 150 heads x 2 tiles: item lists of different lengths per CTA, ragged last tile
    (1, 1, 1537, 64, True),     # 13 tiles, odd length: a single head spread over 13 CTAs in the backward
]


@pytest.mark.parametrize("B,H,T,D,causal", EDGE)
def test_edge_shapes(B, H, T, D, causal):
    h = _harness()
    cfg = W.AttnConfig("edge", B=B, H=H, T=T, D=D, seed=1000 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal)
    h.compare(h.select_heads(got, None), ref, label=f"T={T} D={D} causal={causal}: ", dO=ref["dO_in"])
    if T == 1:
        assert torch.equal(got["O"], V), "a single token attends to itself only: O = V"
        assert torch.equal(got["dV"], dO)
        # dS = P (dP - Delta) = 1 * (dO.V - dO.O): zero up to the fp32 summation order of the two dots
        assert got["dQ"].float().abs().max() < 1e-5 and got["dK"].float().abs().max() < 1e-5


GRID = [  # (B, H, T, D, causal, sampled heads): corners of the paper's benchmark ranges, at its batch of 16
    (16, 32, 2048, 128, True, 2),
    (16, 32, 512, 128, True, 3),
    (16, 20, 1024, 64, True, 3),
    (16, 12, 2048, 64, False, 2),
]


@pytest.mark.parametrize("B,H,T,D,causal,n_heads", GRID)
def test_benchmark_grid_shapes(B, H, T, D, causal, n_heads):
    """Shapes from the ranges of the paper's attention microbenchmark (sequence lengths 512 to 2048, 12 to
    32 heads, head dimension 64 or 128), run at full size on the GPU and compared on sampled heads."""
    h = _harness()
    cfg = W.AttnConfig(f"grid_{T}_{H}_{D}", B=B, H=H, T=T, D=D, seed=300 + T + H + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    heads = sorted({((i * 7 + 3) % B, (i * 11 + 5) % H) for i in range(n_heads)})
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"grid T={T} H={H} D={D} causal={causal}: ", dO=ref["dO_in"])


def test_peaked_softmax_large_scores():
    """Scores ~ N(0, 16^2) (Q, K ~ 4 N(0,1)): exercises the running-max rescale and the exp range far
    beyond the five configurations, with the exact Delta, at the stated bounds.  (dS is formed from the
    unrounded probabilities: with P rounded to bf16 before that product the same case needs about twice
    the gradient bound, as a float64 emulation with exactly those roundings shows.)"""
    h = _harness()
    cfg = W.AttnConfig("peaked", B=1, H=4, T=512, D=64, seed=77, qk_factor=4.0)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, True, exact_delta=True)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, True)
    h.compare(h.select_heads(got, None), ref, label="peaked: ", dO=ref["dO_in"])


def test_increasing_scores_force_rescales():
    """Keys whose scores grow with position make every tile raise the row maximum by more than the
    lazy-rescale threshold."""
    h = _harness()
    cfg = W.AttnConfig("ramp", B=1, H=2, T=640, D=64, seed=78)
    Q, K, V, dO = W.make_inputs(cfg)
    ramp = torch.linspace(0, 6, cfg.T).view(1, 1, cfg.T, 1)
    Q = torch.ones_like(Q)
    K = (K.float() * 0.1 + ramp).to(torch.bfloat16)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, True)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, True)
    # dQ is the small difference of large terms here, so only the element-wise bounds apply
    h.compare(h.select_heads(got, None), ref, label="ramp: ", dO=ref["dO_in"], rms=False)


# The forward works on single query tiles or on pairs of them (more tiles than about seven per SM: pairs): two heads and 700
# copies of one take both forms at T=640, with lazy rescales, sharp rows and an exact mask in each.
FORMS = [(2, 64), (700, 64), (2, 128), (700, 128)]


def _copies(cfg, n, dev, change):
    Q, K, V, dO = change(*W.make_inputs(cfg))
    return (Q, K, V, dO), [x.to(dev).expand(1, n, cfg.T, cfg.D).contiguous() for x in (Q, K, V)]


@pytest.mark.parametrize("n,D", FORMS)
@pytest.mark.parametrize("kind", ["ramp", "falling", "peaked"])
def test_rescales_in_both_forms_of_the_forward(n, D, kind):
    """Scores that grow from key tile to key tile (every tile raises the maximum by more than the lazy-rescale threshold),
    that fall, and that are sharply peaked anywhere: every copy of the head has the same bits, and the oracle's values."""
    import tolerance as tol
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig(kind, B=1, H=1, T=640, D=D, seed=178 + D, qk_factor=4.0 if kind == "peaked" else 1.0)

    def change(Q, K, V, dO):
        if kind == "peaked":
            return Q, K, V, dO
        slope = torch.linspace(0, 6, cfg.T).view(1, 1, cfg.T, 1) * (1 if kind == "ramp" else -1)
        return torch.ones_like(Q), (K.float() * 0.1 + slope).to(torch.bfloat16), V, dO

    host, (q, k, v) = _copies(cfg, n, dev, change)
    for causal in (True, False):
        o, lse = torch.full_like(q, 7.0), torch.full((1, n, cfg.T), 7.0, device=dev)
        nova_attn.nova_attn_fwd(q, k, v, o, lse, cfg.scale, causal)
        nova_attn.nova_attn_poll_device_status()
        ref = h.run_oracle(*host, cfg.scale, causal)
        assert torch.equal(o, o[:, :1].expand_as(o)) and torch.equal(lse, lse[:, :1].expand_as(lse))
        tol.assert_close(W.widen(o[:, :1]), ref["O"], tol.FWD_ATOL, tol.FWD_RTOL, "O")
        tol.assert_close(W.widen(lse[:, :1]), ref["LSE"], tol.FWD_ATOL, tol.FWD_RTOL, "LSE", tol.FWD_REL_RMS)


@pytest.mark.parametrize("n,D", FORMS)
def test_causality_in_both_forms_of_the_forward(n, D):
    """Perturbing keys and values after position t leaves O and LSE of rows <= t bit-identical; the same call twice gives
    the same bits."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("causal", B=1, H=1, T=640, D=D, seed=279)
    _, (q, k, v) = _copies(cfg, n, dev, lambda *x: x)
    t = 200
    k2, v2 = k.clone(), v.clone()
    k2[:, :, t + 1:] = k2[:, :, t + 1:] * -1.5 + 0.25
    v2[:, :, t + 1:] += 1.0
    runs = []
    for kk, vv in ((k, v), (k, v), (k2, v2)):
        o, lse = torch.empty_like(q), torch.empty((1, n, cfg.T), device=dev)
        nova_attn.nova_attn_fwd(q, kk, vv, o, lse, cfg.scale, True)
        runs.append((o, lse))
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][1], runs[1][1])
    for a, b in zip(runs[0], runs[2]):
        assert torch.equal(a[:, :, : t + 1], b[:, :, : t + 1]) and not torch.equal(a[:, :, t + 1:], b[:, :, t + 1:])


def test_causality_is_exact_on_gpu():
    """Perturbing keys/values after position t leaves O, LSE, dQ of rows <= t bit-identical."""
    h = _harness()
    cfg = W.AttnConfig("causality", B=1, H=2, T=384, D=64, seed=79)
    Q, K, V, dO = W.make_inputs(cfg)
    t = 200
    a = h.run_gpu(Q, K, V, dO, cfg.scale, True)
    K2, V2 = K.clone(), V.clone()
    K2[:, :, t + 1:] = (K2[:, :, t + 1:].float() * -1.5 + 0.25).to(torch.bfloat16)
    V2[:, :, t + 1:] = (V2[:, :, t + 1:].float() + 1.0).to(torch.bfloat16)
    b = h.run_gpu(Q, K2, V2, dO, cfg.scale, True)
    assert torch.equal(a["O"][:, :, : t + 1], b["O"][:, :, : t + 1])
    assert torch.equal(a["LSE"][:, :, : t + 1], b["LSE"][:, :, : t + 1])
    assert not torch.equal(a["O"][:, :, t + 1:], b["O"][:, :, t + 1:])
    # dQ is summed with floating-point atomics: equal up to summation order
    da, db = a["dQ"][:, :, : t + 1].float(), b["dQ"][:, :, : t + 1].float()
    assert (da - db).abs().max() <= 2e-2 * da.abs().max()


def test_run_to_run_determinism():
    h = _harness()
    cfg = W.CONFIGS["gpt2_small"].replace(B=2, H=2)
    Q, K, V, dO = W.make_inputs(cfg)
    a = h.run_gpu(Q, K, V, dO, cfg.scale, True)
    b = h.run_gpu(Q, K, V, dO, cfg.scale, True)
    for name in ("O", "LSE", "Delta", "dK", "dV"):
        assert torch.equal(a[name], b[name]), f"{name} differs between identical runs"
    d = (a["dQ"].float() - b["dQ"].float()).abs().max()
    assert d <= 1e-2 * a["dQ"].float().abs().max()


def test_preprocess_matches_rowsum():
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    for (B, H, T, D) in [(1, 1, 1, 64), (2, 3, 77, 64), (1, 2, 1000, 128), (4, 12, 1024, 64)]:
        g = torch.Generator().manual_seed(T)
        O = torch.randn((B, H, T, D), generator=g).to(torch.bfloat16)
        dO = torch.randn((B, H, T, D), generator=g).to(torch.bfloat16)
        Delta = torch.full((B, H, T), 3.0, dtype=torch.float32, device=dev)
        nova_attn.nova_attn_bwd_preprocess(O.to(dev), dO.to(dev), Delta)
        ref = (O.double() * dO.double()).sum(-1)
        torch.testing.assert_close(Delta.cpu().double(), ref, rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("B,H,T", [(1, 1, 1), (2, 7, 33), (1, 9, 16), (3, 8, 257), (16, 12, 513), (4, 12, 1024), (3, 2, 129),
                                   (2, 3, 77), (1, 6, 65), (9, 25, 700), (60, 3, 705), (60, 2, 1001)])
@pytest.mark.parametrize("D", [64, 128])
def test_preprocess_with_heads_inside_tokens(B, H, T, D):
    """O and dO as views of [B,T,H,D] buffers take the path that reads in memory order: tiles of tokens and heads with
    remainders of both, few and many blocks; the same sums in the same order as the plain path, so the same bits."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    g = torch.Generator().manual_seed(B + H + T + D)
    O, dO = (torch.randn((B, T, H, D), generator=g).to(torch.bfloat16).to(dev).permute(0, 2, 1, 3) for _ in range(2))
    buf = torch.full((B * H * T + 128,), 3.0, device=dev)
    Delta, plain = buf[64:-64].view(B, H, T), torch.empty((B, H, T), device=dev)
    nova_attn.nova_attn_bwd_preprocess_strided(O, dO, Delta)
    nova_attn.nova_attn_bwd_preprocess(O.contiguous(), dO.contiguous(), plain)
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(Delta, plain)
    assert bool((buf[:64] == 3.0).all()) and bool((buf[-64:] == 3.0).all())


def test_back_to_back_steps_on_shared_buffers():
    """Every kernel may start while its predecessor in the stream is still draining, and waits for it
    before touching global memory.  Twelve forward + backward steps are enqueued without a host
    synchronisation, alternating between two input sets but sharing ONE workspace, ONE set of
    intermediate buffers (O, LSE, Delta) and ONE set of outputs per input set: a kernel that ran ahead
    of a predecessor would read a half-written O, clear an accumulator that is still being converted,
    or overwrite an output that is still being read.  Results must equal those of isolated runs."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfgs = [W.CONFIGS["gpt2_small"].replace(B=2, H=3, seed=91), W.CONFIGS["gpt2_small"].replace(B=2, H=3, seed=92)]
    inputs = [W.make_inputs(c) for c in cfgs]
    ref = [h.run_gpu(*inp, cfgs[0].scale, True) for inp in inputs]
    dins = [tuple(x.to(dev) for x in inp) for inp in inputs]
    B, H, T, D = dins[0][0].shape
    o = torch.empty((B, H, T, D), dtype=torch.bfloat16, device=dev)
    lse = torch.empty((B, H, T), dtype=torch.float32, device=dev)
    delta = torch.empty_like(lse)
    ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(B, H, T, D), dtype=torch.uint8, device=dev)
    outs = [tuple(torch.empty_like(o) for _ in range(3)) for _ in range(2)]
    snap = []
    for step in range(12):
        s = step & 1
        q, k, v, do = dins[s]
        dq, dk, dv = outs[s]
        nova_attn.nova_attn_fwd(q, k, v, o, lse, cfgs[0].scale, True)
        nova_attn.nova_attn_bwd_preprocess(o, do, delta)
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, dq, dk, dv, cfgs[0].scale, True, ws)
        if step >= 10:  # device-side copies, ordered in the same stream: still no host synchronisation
            snap.append((s, o.clone(), lse.clone(), delta.clone(), dq.clone(), dk.clone(), dv.clone()))
    nova_attn.nova_attn_poll_device_status()
    for s, o_s, lse_s, delta_s, dq_s, dk_s, dv_s in snap:
        r = ref[s]
        assert torch.equal(o_s.cpu(), r["O"]) and torch.equal(lse_s.cpu(), r["LSE"])
        assert torch.equal(delta_s.cpu(), r["Delta"])
        assert torch.equal(dk_s.cpu(), r["dK"]) and torch.equal(dv_s.cpu(), r["dV"])
        d = (dq_s.cpu().float() - r["dQ"].float()).abs().max()
        assert d <= 1e-2 * r["dQ"].float().abs().max()  # dQ: summation order of the reduce-adds


@pytest.mark.parametrize("entry", ["plain", "deterministic"])
@pytest.mark.parametrize("causal", [True, False])
def test_back_to_back_two_kernel_backward_on_shared_buffers(entry, causal):
    """The same where the dQ and the dK/dV kernel of D=64 run (768 tiles): the row terms that the next step puts into the one
    workspace, its LSE and its Delta must not reach the dK/dV kernel of this one, nor the other way round.  Both kernels sum in
    a fixed order, so all gradients have the bits of isolated runs."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    cfg = W.CONFIGS["gpt2_small"].replace(causal=causal)
    B, H, T, D = cfg.B, cfg.H, cfg.T, cfg.D
    assert B * H * ((T + 127) // 128) >= 2.5 * torch.cuda.get_device_properties(dev).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(93)
    dins = [[torch.randn((B, H, T, D), generator=g, device=dev).to(torch.bfloat16) for _ in range(4)] for _ in range(2)]
    o = torch.empty_like(dins[0][0])
    lse = torch.empty((B, H, T), dtype=torch.float32, device=dev)
    delta = torch.empty_like(lse)
    ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(B, H, T, D), dtype=torch.uint8, device=dev)

    def step(s, grads):
        q, k, v, do = dins[s]
        nova_attn.nova_attn_fwd(q, k, v, o, lse, cfg.scale, causal)
        nova_attn.nova_attn_bwd_preprocess(o, do, delta)
        if entry == "plain":
            nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *grads, cfg.scale, causal, ws)
        else:
            nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *grads, cfg.scale, causal)

    alone = []
    for s in range(2):
        alone.append([torch.full_like(o, 7.0) for _ in range(3)])
        torch.cuda.synchronize()
        step(s, alone[s])
        nova_attn.nova_attn_poll_device_status()
    runs = [[torch.full_like(o, 7.0) for _ in range(3)] for _ in range(12)]
    for i, grads in enumerate(runs):
        step(i & 1, grads)
    nova_attn.nova_attn_poll_device_status()
    for i, grads in enumerate(runs):
        assert all(torch.equal(a, b) for a, b in zip(grads, alone[i & 1])), i


FUSED = [  # (B, H, T, D, causal)
    (2, 3, 300, 64, True),      # ragged T: partial tiles with TMA clipping on strided rows
    (2, 12, 1024, 64, True),    # the GPT-2 layout: H*D = 768
    (1, 4, 384, 128, True),     # D = 128: dK/dV rows leave through plain strided stores
    (2, 2, 256, 64, False),
]


@pytest.mark.parametrize("B,H,T,D,causal", FUSED)
def test_fused_projection_layout(B, H, T, D, causal):
    """Q, K, V read straight out of a fused projection output [B, T, 3, H, D]; O written as [B, T, H, D]; dO
    given as [B, T, H, D]; dQ, dK, dV written into one fused gradient buffer [B, T, 3, H, D] (paper
    Section 4.2: the per-head layout change costs nothing).  Only the addressing differs from the
    [B,H,T,D] entry points, so O, LSE, Delta, dK, dV must be bit-identical to theirs; and both match the oracle."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("fused", B=B, H=H, T=T, D=D, seed=500 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    plain = h.run_gpu(Q, K, V, dO, cfg.scale, causal)

    qkv = torch.full((B, T, 3, H, D), 7.0, dtype=torch.bfloat16, device=dev)
    for i, x in enumerate((Q, K, V)):
        qkv[:, :, i] = x.to(dev).permute(0, 2, 1, 3)
    q_v, k_v, v_v = (qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))        # [B,H,T,D] views, no copy
    assert q_v.data_ptr() == qkv.data_ptr() and k_v.data_ptr() == qkv.data_ptr() + 2 * H * D
    o_buf = torch.full((B, T, H, D), 7.0, dtype=torch.bfloat16, device=dev)
    do_buf = dO.to(dev).permute(0, 2, 1, 3).contiguous()                        # [B,T,H,D]
    dqkv = torch.full((B, T, 3, H, D), 7.0, dtype=torch.bfloat16, device=dev)
    o_v, do_v = o_buf.permute(0, 2, 1, 3), do_buf.permute(0, 2, 1, 3)
    dq_v, dk_v, dv_v = (dqkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))
    lse = torch.empty((B, H, T), dtype=torch.float32, device=dev)
    delta = torch.empty_like(lse)
    nova_attn.nova_attn_fwd_strided(q_v, k_v, v_v, o_v, lse, cfg.scale, causal)
    nova_attn.nova_attn_bwd_preprocess_strided(o_v, do_v, delta)
    nova_attn.nova_attn_bwd_strided(q_v, k_v, v_v, do_v, lse, delta, dq_v, dk_v, dv_v, cfg.scale, causal)
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(qkv[:, :, 0].permute(0, 2, 1, 3).cpu(), Q), "inputs must not be modified"

    got = {"O": o_v.contiguous().cpu(), "LSE": lse.cpu(), "Delta": delta.cpu(),
           "dQ": dq_v.contiguous().cpu(), "dK": dk_v.contiguous().cpu(), "dV": dv_v.contiguous().cpu()}
    for name in ("O", "LSE", "Delta", "dK", "dV"):
        assert torch.equal(got[name], plain[name]), f"{name}: strided and contiguous entry points differ"
    d = (got["dQ"].float() - plain["dQ"].float()).abs().max()
    assert d <= 1e-2 * plain["dQ"].float().abs().max()
    heads = sorted({(i % B, (i * 5 + 1) % H) for i in range(4)})
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"fused T={T} D={D}: ", dO=ref["dO_in"])


@pytest.mark.parametrize("T", [1, 17, 64, 127, 128])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_single_key_tile_writes_dq_directly(T, D, causal):
    """T <= 128: the backward writes dQ without the fp32 accumulator.  One contribution per tile added to zero, scaled
    and rounded once is the same number either way, so the three steps issued one by one (which go through the
    accumulator) give the same bits, as do the deterministic entry point and, on a fused layout, the strided one;
    more heads than SMs, so that a CTA reuses its staging buffer."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("direct", B=4, H=50, T=T, D=D, seed=700 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))
    o, lse, delta = got["O"].to(dev), got["LSE"].to(dev), got["Delta"].to(dev)
    ws = torch.full((nova_attn.nova_attn_bwd_workspace_bytes(cfg.B, cfg.H, T, D),), 255, dtype=torch.uint8, device=dev)
    a, b = ([torch.full_like(q, 7.0) for _ in range(3)] for _ in range(2))
    for step in (nova_attn.BWD_STEP_ZERO, nova_attn.BWD_STEP_MAIN, nova_attn.BWD_STEP_CONVERT):
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *a, cfg.scale, causal, ws, steps=step)
    nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *b, cfg.scale, causal)
    dqkv = torch.full((cfg.B, T, 3, cfg.H, D), 7.0, dtype=torch.bfloat16, device=dev)
    c = [dqkv[:, :, i].permute(0, 2, 1, 3) for i in range(3)]
    nova_attn.nova_attn_bwd_strided(q, k, v, do, lse, delta, *c, cfg.scale, causal, ws)
    nova_attn.nova_attn_poll_device_status()
    for name, x, y, z in zip(("dQ", "dK", "dV"), a, b, c):
        for other in (x, y, z):
            assert torch.equal(other.cpu(), got[name]), name
    heads = [(0, 0), (3, 49)]
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"direct T={T} D={D}: ", dO=ref["dO_in"])


@pytest.mark.parametrize("T", [129, 191, 193, 256, 257, 385, 449])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_query_major_passes_at_step_edges(T, D, causal):
    """The deterministic dQ and the exact Delta walk the keys in steps of 64, for pairs of 128-row tiles or (D=64) for one tile
    in two groups that take turns: sequence lengths around the edges of a step, of a tile and of a pair (a second tile with
    one row, or none), more items than SMs so that CTAs take over further ones; twelve calls back to back give the same bits
    every time."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("steps", B=7, H=30, T=T, D=D, seed=900 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal, exact_delta=True)
    q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))
    lse = got["LSE"].to(dev)
    runs = []
    for _ in range(12):
        delta = torch.full_like(lse, 7.0)
        dq, dk, dv = (torch.full_like(q, 7.0) for _ in range(3))
        nova_attn.nova_attn_bwd_preprocess_exact(q, k, v, do, lse, delta, cfg.scale, causal)
        nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, dq, dk, dv, cfg.scale, causal)
        runs.append((delta, dq, dk, dv))
    nova_attn.nova_attn_poll_device_status()
    for r in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(r, runs[0]))
    assert torch.equal(runs[0][0].cpu(), got["Delta"])
    got.update(dQ=runs[0][1].cpu(), dK=runs[0][2].cpu(), dV=runs[0][3].cpu())
    heads = [(0, 0), (6, 29)]
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"steps T={T} D={D}: ", dO=ref["dO_in"])


@pytest.mark.parametrize("T", [129, 256, 257, 500, 1000])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_query_major_passes_alone_and_in_a_crowd(T, D, causal):
    """The exact Delta and the deterministic dQ take single query tiles where the longest of them decides and pairs where the
    work does: a head alone, 100 copies of it (single tiles in several rounds at the shorter lengths) and 640 (pairs) have the
    same bits, and the oracle's values."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("crowd", B=1, H=1, T=T, D=D, seed=500 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal, exact_delta=True)
    first = None
    for n in (1, 100, 640):
        q, k, v, do = (x.to(dev).expand(1, n, T, D).contiguous() for x in (Q, K, V, dO))
        lse = got["LSE"].to(dev).expand(1, n, T).contiguous()
        delta, grads = torch.full_like(lse, 7.0), [torch.full_like(q, 7.0) for _ in range(3)]
        nova_attn.nova_attn_bwd_preprocess_exact(q, k, v, do, lse, delta, cfg.scale, causal)
        nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *grads, cfg.scale, causal)
        nova_attn.nova_attn_poll_device_status()
        outs = [delta, *grads]
        first = first or [t[:, :1].clone() for t in outs]
        assert all(torch.equal(t, f.expand_as(t)) for t, f in zip(outs, first)), n
    got.update({name: t.cpu() for name, t in zip(("Delta", "dQ", "dK", "dV"), first)})
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal)
    h.compare(h.select_heads(got, None), ref, label=f"crowd T={T} D={D}: ", dO=ref["dO_in"])


@pytest.mark.parametrize("T", [1, 63, 64, 65, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_exact_delta_of_short_sequences(T, causal):
    """Items of one or two steps, in which a compute group may have none: a head alone and 1500 copies (ten items per SM) have
    the same bits, and the definition's value, sum_j P_ij (dO_i . V_j) in 64 bits, to within the fp32 sums and exponentials
    (2e-6 of the largest terms, 64 in all; 1e-4 covers them with P read from an fp32 LSE)."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("short", B=1, H=1, T=T, D=64, seed=20 + T, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    lse1 = h.run_gpu(Q, K, V, dO, cfg.scale, causal)["LSE"].to(dev)
    first = None
    for n in (1, 1500):
        q, k, v, do = (x.to(dev).expand(1, n, T, 64).contiguous() for x in (Q, K, V, dO))
        delta = torch.full((1, n, T), 7.0, device=dev)
        nova_attn.nova_attn_bwd_preprocess_exact(q, k, v, do, lse1.expand(1, n, T).contiguous(), delta, cfg.scale, causal)
        nova_attn.nova_attn_poll_device_status()
        first = delta[0, 0].clone() if first is None else first
        assert torch.equal(delta, first.expand_as(delta)), n
    q, k, v, do = (x[0, 0].double() for x in (Q, K, V, dO))
    s = (q @ k.T) * cfg.scale
    if causal:
        s = s.masked_fill(torch.ones(T, T).triu(1).bool(), float("-inf"))
    want = (torch.softmax(s, -1) * (do @ v.T)).sum(-1)
    assert (first.double().cpu() - want).abs().max() <= 1e-4 * max(1.0, float((do @ v.T).abs().max()))


@pytest.mark.parametrize("T,causal", [(1, True), (64, False), (65, True), (128, False), (129, True), (192, True), (193, False),
                                      (700, False), (1025, False)])
def test_bits_of_exact_delta_do_not_depend_on_the_number_of_heads(T, causal):
    """At D=64 two kernels compute it, by the number of tiles per SM: a head alone, in a crowd, in a large one."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    g = torch.Generator(device="cuda").manual_seed(T)
    one = [torch.randn((1, 1, T, 64), generator=g, device=dev).to(torch.bfloat16) for _ in range(4)]
    lse1, first = torch.empty((1, 1, T), device=dev), None
    nova_attn.nova_attn_fwd(*one[:3], torch.empty_like(one[0]), lse1, 0.125, causal)
    tiles = (T + 127) // 128
    for per_sm in (0, 1, 4, 13, 30):
        n = max(1, per_sm * 148 // tiles + per_sm)
        q, k, v, do = (x.expand(1, n, T, 64).contiguous() for x in one)
        delta = torch.full((1, n, T), 7.0, device=dev)
        nova_attn.nova_attn_bwd_preprocess_exact(q, k, v, do, lse1.expand(1, n, T).contiguous(), delta, 0.125, causal)
        nova_attn.nova_attn_poll_device_status()
        first = delta[0, 0].clone() if first is None else first
        assert torch.equal(delta, first.expand_as(delta)), n


@pytest.mark.parametrize("T", [1, 127, 129, 256, 257, 384, 500])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_forward_alone_and_in_a_crowd(T, D, causal):
    """With an SM for every 128-row tile the forward works on one tile per CTA, its keys split between the two softmax
    groups, otherwise on pairs of tiles: a head alone and 160 copies of it (pairs, several items per CTA) both match the
    oracle, and the copies are the same bits, on the plain and on a strided layout."""
    import tolerance as tol
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("crowd", B=1, H=1, T=T, D=D, seed=300 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    alone = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal)
    h.compare(h.select_heads(alone, None), ref, label=f"alone T={T} D={D}: ", dO=ref["dO_in"])
    q, k, v = (x.to(dev).expand(8, 20, T, D).contiguous() for x in (Q, K, V))
    for strided in (False, True):
        if strided:
            q, k, v = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (q, k, v))
        o, lse = torch.full_like(q, 7.0), torch.full((8, 20, T), 7.0, device=dev)
        (nova_attn.nova_attn_fwd_strided if strided else nova_attn.nova_attn_fwd)(q, k, v, o, lse, cfg.scale, causal)
        nova_attn.nova_attn_poll_device_status()
        assert torch.equal(o, o[:1, :1].expand_as(o)) and torch.equal(lse, lse[:1, :1].expand_as(lse))
        tol.assert_close(W.widen(o[:1, :1]), ref["O"], tol.FWD_ATOL, tol.FWD_RTOL, "O", tol.FWD_REL_RMS)
        tol.assert_close(W.widen(lse[:1, :1]), ref["LSE"], tol.FWD_ATOL, tol.FWD_RTOL, "LSE", tol.FWD_REL_RMS)


@pytest.mark.parametrize("n", [20, 60, 600])
@pytest.mark.parametrize("T", [257, 640, 1024])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("causal", [True, False])
def test_forward_between_one_tile_per_sm_and_many_rounds(n, T, D, causal):
    """Which of its two forms the forward takes there depends on how the last round of items ends; single tiles then also
    follow each other on an SM.  Copies of one head, at head counts on both sides: all the same, and the oracle's values."""
    import tolerance as tol
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("rounds", B=1, H=1, T=T, D=D, seed=800 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal)
    q, k, v = (x.to(dev).expand(1, n, T, D).contiguous() for x in (Q, K, V))
    o, lse = torch.full_like(q, 7.0), torch.full((1, n, T), 7.0, device=dev)
    nova_attn.nova_attn_fwd(q, k, v, o, lse, cfg.scale, causal)
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(o, o[:, :1].expand_as(o)) and torch.equal(lse, lse[:, :1].expand_as(lse))
    tol.assert_close(W.widen(o[:, :1]), ref["O"], tol.FWD_ATOL, tol.FWD_RTOL, "O", tol.FWD_REL_RMS)
    tol.assert_close(W.widen(lse[:, :1]), ref["LSE"], tol.FWD_ATOL, tol.FWD_RTOL, "LSE", tol.FWD_REL_RMS)


@pytest.mark.parametrize("T", [128, 200, 500])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("first", [0, 64])
def test_forward_with_half_a_tile_of_lowest_scores(T, D, first):
    """One query tile per CTA splits its keys in halves of 64.  Keys whose scores are around -1e37, as masks of the lowest
    value make them, have no weight beside ordinary ones, whichever half they fill: the same bits as with scores of -1e4,
    where 2^x is 0 as well."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("lowest", B=1, H=2, T=T, D=D, seed=11 + T)
    Q, K, V, _ = (x.to(dev) for x in W.make_inputs(cfg))
    Q[..., 0] = 1.0
    out = []
    for low in (-1e37, -1e4 / cfg.scale):
        k = K.clone()
        k[:, :, first : first + 64] = 0
        k[:, :, first : first + 64, 0] = low
        o, lse = torch.empty_like(Q), torch.empty((1, 2, T), device=dev)
        nova_attn.nova_attn_fwd(Q, k, V, o, lse, cfg.scale, False)
        nova_attn.nova_attn_poll_device_status()
        out.append((o, lse))
    assert torch.isfinite(out[0][1]).all() and torch.isfinite(out[0][0].float()).all()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("scale,qk", [(1e-36, 1.0), (5e-31, 1.0), (2e-30, 1.0), (1e-20, 1.0), (12.5, 0.01)])
@pytest.mark.parametrize("T", [100, 300])
def test_scales_far_from_ordinary(scale, qk, T):
    """At D=64 the backward subtracts LSE/scale from the scores inside the contraction, as three bf16 numbers: a scale at
    which that quotient would not be finite (P is uniform there), one at which it dwarfs the scores, and a large one.
    dQ carries the rounding of dS times scale * |K|, and the harness's bounds are stated for scale * |K| = 1/8 (unit K,
    D=64): K is scaled down with the large scale so that this holds (at scale 30 and |K| = 0.1 the bound would be 24
    times theirs)."""
    import tolerance as tol
    h = _harness()
    cfg = W.AttnConfig("scales", B=1, H=2, T=T, D=64, seed=77, qk_factor=qk)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, scale, True, exact_delta=True)
    ref = h.run_oracle(Q, K, V, dO, scale, True)
    sel = h.select_heads(got, None)
    h.compare(sel, ref, label=f"scale={scale}: ", dO=ref["dO_in"], rms=scale > 1)
    # The bounds above say nothing about gradients of the size of a tiny scale; those relative to the result do.  (At 1e-36
    # dQ and dK reach into bf16's subnormal numbers.)
    names = [("O", tol.FWD_REL_RMS), ("LSE", tol.FWD_REL_RMS), ("dV", tol.BWD_REL_RMS)]
    for name, bound in names + ([("dQ", tol.BWD_REL_RMS), ("dK", tol.BWD_REL_RMS)] if scale > 1e-33 else []):
        assert tol.rel_rms(sel[name], ref[name]) <= bound, name


# D=128: B*H*ceil(T/256) >= 222 takes the two-kernel backward, fewer blocks the fused kernel (one case on that side);
# lengths around a step of 64, a tile of 128 and a pair of tiles, single-step items, more items than SMs.
TWO_KERNELS = [(8, 30, 129, True), (8, 30, 191, False), (8, 30, 256, True), (8, 14, 257, True), (5, 25, 449, False),
               (10, 8, 700, True), (4, 32, 1000, True), (7, 30, 200, True)]


@pytest.mark.parametrize("B,H,T,causal", TWO_KERNELS)
def test_wide_heads_backward_routes(B, H, T, causal):
    """nova_attn_bwd at D=128 where it goes through the dQ and the dK/dV kernel: the same dK and dV as the fused kernel's
    (its steps issued one by one), on the plain and on the fused-projection layout, and everything against the oracle."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("wide", B=B, H=H, T=T, D=128, seed=40 + T, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))
    o, lse, delta = got["O"].to(dev), got["LSE"].to(dev), got["Delta"].to(dev)
    ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(B, H, T, 128), dtype=torch.uint8, device=dev)
    fused = [torch.full_like(q, 7.0) for _ in range(3)]
    for step in (nova_attn.BWD_STEP_ZERO, nova_attn.BWD_STEP_MAIN, nova_attn.BWD_STEP_CONVERT):
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *fused, cfg.scale, causal, ws, steps=step)
    qkv = torch.stack([x.transpose(1, 2) for x in (q, k, v)], 2)
    dqkv = torch.full_like(qkv, 7.0)
    views, grads = ([t[:, :, i].permute(0, 2, 1, 3) for i in range(3)] for t in (qkv, dqkv))
    nova_attn.nova_attn_bwd_strided(*views, do.transpose(1, 2).contiguous().transpose(1, 2), lse, delta, *grads, cfg.scale,
                                    causal, ws)
    nova_attn.nova_attn_poll_device_status()
    for name, a, b in (("dK", fused[1], grads[1]), ("dV", fused[2], grads[2])):
        assert torch.equal(a.cpu(), got[name]) and torch.equal(b.cpu(), got[name]), name
    for other in (fused[0], grads[0]):
        d = (other.cpu().float() - got["dQ"].float()).abs().max()
        assert d <= 1e-2 * got["dQ"].float().abs().max()
    heads = [(0, 0), (B - 1, H - 1)]
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"wide T={T}: ", dO=ref["dO_in"])


# D=64: lengths around a step of 64, a tile of 128 and the ring of stages; items of one step, more items than SMs, several
# items per SM that follow each other before the operands of the last have been released.
TWO_KERNELS_64 = [(8, 30, 129, True), (8, 30, 191, False), (40, 30, 130, True), (5, 25, 449, False), (10, 8, 700, True),
                  (7, 30, 200, True), (3, 50, 383, True), (2, 3, 1025, False)]


@pytest.mark.parametrize("B,H,T,causal", TWO_KERNELS_64)
def test_narrow_heads_two_kernel_backward(B, H, T, causal):
    """The dQ and the dK/dV kernel at D=64: dK and dV have the bits of the fused kernel's (same arithmetic, same order; its
    steps issued one by one), everything agrees with the oracle."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("narrow", B=B, H=H, T=T, D=64, seed=80 + T, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    got = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))
    o, lse, delta = got["O"].to(dev), got["LSE"].to(dev), got["Delta"].to(dev)
    ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(B, H, T, 64), dtype=torch.uint8, device=dev)
    fused = [torch.full_like(q, 7.0) for _ in range(3)]
    for step in (nova_attn.BWD_STEP_ZERO, nova_attn.BWD_STEP_MAIN, nova_attn.BWD_STEP_CONVERT):
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *fused, cfg.scale, causal, ws, steps=step)
    two = [torch.full_like(q, 7.0) for _ in range(3)]
    nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *two, cfg.scale, causal)
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(two[1], fused[1]) and torch.equal(two[2], fused[2])
    got.update({"dQ": two[0].cpu(), "dK": two[1].cpu(), "dV": two[2].cpu()})
    heads = [(0, 0), (B - 1, H - 1)]
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"narrow T={T}: ", dO=ref["dO_in"])


# The same above the number of tiles from which nova_attn_bwd takes the two kernels (148 SMs: 370 tiles, 814 at T <= 256; without
# the mask up to 2072), with the row terms in the workspace.
ABOVE_64 = [(40, 30, 130, True), (4, 104, 200, True), (3, 140, 256, False), (3, 50, 383, True), (5, 25, 449, False),
            (10, 8, 700, True), (6, 8, 1024, False)]


@pytest.mark.parametrize("B,H,T,causal", ABOVE_64)
def test_narrow_heads_two_kernel_backward_through_every_entry_point(B, H, T, causal):
    """Plain: dK and dV have the bits of the fused kernel's (its steps issued one by one), dQ those of the deterministic entry
    point, whatever the workspace held.  Strided: the same bits in three rounds of layouts (plain, [B,T,H,D], padded, heads or
    tokens outermost, a different one for each tensor), nothing written between the rows.  Static scratch, where the problem
    fits: the same bits right after a call on other inputs."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    tiles, sms = B * H * ((T + 127) // 128), torch.cuda.get_device_properties(dev).multi_processor_count
    assert (2.5 if T > 256 else 5.5) * sms <= tiles and (causal or tiles <= 14 * sms)
    D, scale = 64, 0.125
    g = torch.Generator(device="cuda").manual_seed(T)
    q, k, v, do, do2 = (torch.randn((B, H, T, D), generator=g, device=dev).to(torch.bfloat16) for _ in range(5))
    o, lse = torch.empty_like(q), torch.empty((B, H, T), device=dev)
    delta, delta2 = torch.empty_like(lse), torch.empty_like(lse)
    nova_attn.nova_attn_fwd(q, k, v, o, lse, scale, causal)
    nova_attn.nova_attn_bwd_preprocess(o, do, delta)
    nova_attn.nova_attn_bwd_preprocess(o, do2, delta2)
    ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(B, H, T, D), dtype=torch.uint8, device=dev)
    fused, alike, plain = ([torch.full_like(q, 7.0) for _ in range(3)] for _ in range(3))
    for step in (nova_attn.BWD_STEP_ZERO, nova_attn.BWD_STEP_MAIN, nova_attn.BWD_STEP_CONVERT):
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *fused, scale, causal, ws, steps=step)
    nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *alike, scale, causal)
    nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *plain, scale, causal, ws.fill_(255))
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(plain[1], fused[1]) and torch.equal(plain[2], fused[2])
    assert torch.equal(plain[0], alike[0])
    assert (plain[0].float() - fused[0].float()).abs().max() <= 1e-2 * fused[0].float().abs().max()  # (dQ: order of the reduce-adds)

    rng = np.random.default_rng(T)
    kinds = ["bhtd", "bthd", "pad_t", "pad_h", "hbtd", "tbhd"]
    for shift in range(3):
        views = [_layout_view(x, kinds[(2 * shift + i) % 6], rng, dev)[0] for i, x in enumerate((q, k, v, do))]
        outs = [_layout_view(torch.full_like(q, 7.0), kinds[(2 * shift + 4 + i) % 6], rng, dev) for i in range(3)]
        nova_attn.nova_attn_bwd_strided(*views, lse, delta, *(view for view, _ in outs), scale, causal, ws.fill_(255))
        nova_attn.nova_attn_poll_device_status()
        for (view, storage), want in zip(outs, plain):
            assert torch.equal(view, want), shift
            view.fill_(7.0)  # what is left must be the untouched padding
            assert bool((storage == 7.0).all()), shift

    if ws.numel() <= nova_attn.nova_attn_static_scratch_bytes():
        other, static = ([torch.full_like(q, 7.0) for _ in range(3)] for _ in range(2))
        nova_attn.nova_attn_bwd_static_scratch(q, k, v, o, do2, lse, delta2, *other, scale, causal)
        nova_attn.nova_attn_bwd_static_scratch(q, k, v, o, do, lse, delta, *static, scale, causal)
        nova_attn.nova_attn_poll_device_status()
        assert all(torch.equal(a, b) for a, b in zip(static, plain))
        assert not torch.equal(other[0], plain[0])


@pytest.mark.parametrize("H,T,causal", [(394, 1500, True), (395, 1500, True), (273, 1600, True), (274, 1600, True),
                                        (172, 1500, False), (173, 1500, False), (53, 4224, False), (54, 4224, False)])
def test_narrow_heads_backward_around_the_limits_of_the_two_kernels(H, T, causal):
    """On either side of 32 and 24 tiles per SM causal, 14 and 12 without the mask (148 SMs): dK and dV of the plain call have the
    bits of the deterministic one, dQ is as close as the order of its sums allows."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    g = torch.Generator(device="cuda").manual_seed(H + T)
    q, k, v, do = (torch.randn((1, H, T, 64), generator=g, device=dev).to(torch.bfloat16) for _ in range(4))
    o, lse = torch.empty_like(q), torch.empty((1, H, T), device=dev)
    delta = torch.empty_like(lse)
    nova_attn.nova_attn_fwd(q, k, v, o, lse, 0.125, causal)
    nova_attn.nova_attn_bwd_preprocess(o, do, delta)
    plain, alike = ([torch.full_like(q, 7.0) for _ in range(3)] for _ in range(2))
    nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, *plain, 0.125, causal)
    nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *alike, 0.125, causal)
    nova_attn.nova_attn_poll_device_status()
    assert torch.equal(plain[1], alike[1]) and torch.equal(plain[2], alike[2])
    assert (plain[0].float() - alike[0].float()).abs().max() <= 1e-2 * alike[0].float().abs().max()


# One of each backward kernel: the fused one (single key tile, several), with more heads than SMs, and at D=128 the pair of
# kernels (which the deterministic entry point takes at every T > 128).
NOT_FINITE = [(1, 2, 100, 64), (1, 2, 300, 64), (8, 30, 300, 64), (1, 2, 100, 128), (1, 2, 300, 128), (8, 30, 300, 128)]


@pytest.mark.parametrize("B,H,T,D", NOT_FINITE)
@pytest.mark.parametrize("entry", ["plain", "deterministic"])
@pytest.mark.parametrize("row", [3, 70, 90])
def test_a_query_that_is_not_finite_stays_in_its_place(B, H, T, D, entry, row):
    """What one query's Delta, LSE or dO may spoil.  Delta does not enter dV; LSE = +inf means P = 0, i.e. the row takes no
    part; a NaN LSE ends at the diagonal; a dO that is not finite reaches its own column of dV.
    The outputs that are not concerned have the bits of the run without it."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("place", B=B, H=H, T=T, D=D, seed=60 + T + D, causal=True)
    Q, K, V, dO = W.make_inputs(cfg)
    fwd = h.run_gpu(Q, K, V, dO, cfg.scale, True)
    q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))

    def backward(lse, delta, do):
        g = [torch.full_like(q, 7.0) for _ in range(3)]
        if entry == "plain":
            nova_attn.nova_attn_bwd(q, k, v, q, do, lse, delta, *g, cfg.scale, True)
        else:
            nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, *g, cfg.scale, True)
        nova_attn.nova_attn_poll_device_status()
        return [x.float() for x in g]

    def poked(t, value, *at):
        t = t.clone()
        t[(0, 1, row) + at] = value
        return t

    lse, delta = fwd["LSE"].to(dev), fwd["Delta"].to(dev)
    dq0, dk0, dv0 = backward(lse, delta, do)
    for value in (float("inf"), float("-inf"), float("nan")):
        dq, dk, dv = backward(lse, poked(delta, value), do)
        assert torch.equal(dv, dv0), f"Delta = {value} reached dV"
        assert not torch.isfinite(dq[0, 1, row]).any() and not torch.isfinite(dk[0, 1, 0]).any()
        dv = backward(lse, delta, poked(do, value, 5))[2]
        keep = torch.arange(D, device=dev) != 5
        assert torch.equal(dv[..., keep], dv0[..., keep]), f"dO = {value} reached other columns of dV"
    _, dk0, dv0 = backward(poked(lse, 1e4), delta, do)  # 2^-14000: P = 0
    for value in (3e38, float("inf")):
        dq, dk, dv = backward(poked(lse, value), delta, do)
        assert torch.equal(dk, dk0) and torch.equal(dv, dv0) and bool((dq[0, 1, row] == 0).all()), f"LSE = {value}"
        assert torch.isfinite(dq).all()
    _, dk, dv = backward(poked(lse, float("nan")), delta, do)
    for got, without in ((dk, dk0), (dv, dv0)):
        assert torch.equal(got[0, 1, row + 1:], without[0, 1, row + 1:]) and not torch.isfinite(got[0, 1, : row + 1]).any()


DETERMINISTIC = [  # (B, H, T, D, causal)
    (1, 2, 64, 64, True),
    (2, 3, 300, 64, True),
    (2, 12, 1024, 64, True),
    (1, 4, 640, 128, True),
    (2, 2, 256, 128, False),
    (1, 1, 1, 64, True),
]


@pytest.mark.parametrize("B,H,T,D,causal", DETERMINISTIC)
def test_deterministic_two_kernel_backward(B, H, T, D, causal):
    """The two-kernel backward of the paper (Section 4.2: dQ reduced over keys in one kernel, dK and dV
    over queries in the other): matches the oracle, is bitwise reproducible (dQ included), needs no
    workspace, and its dK, dV are bit-identical to the fused backward's (same arithmetic, same order)."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("det", B=B, H=H, T=T, D=D, seed=700 + T + D, causal=causal)
    Q, K, V, dO = W.make_inputs(cfg)
    fused = h.run_gpu(Q, K, V, dO, cfg.scale, causal)
    q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))
    lse, delta = fused["LSE"].to(dev), fused["Delta"].to(dev)
    runs = []
    for _ in range(2):
        bufs = [torch.full((B * H * T * D + 128,), 7.0, dtype=torch.bfloat16, device=dev) for _ in range(3)]
        dq, dk, dv = (b[64:64 + B * H * T * D].view(B, H, T, D) for b in bufs)
        nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, dq, dk, dv, cfg.scale, causal)
        nova_attn.nova_attn_poll_device_status()
        for b in bufs:
            g = torch.cat([b[:64], b[-64:]]).float().cpu()
            assert (g == 7.0).all(), "write outside an output buffer"
        runs.append({"dQ": dq.cpu(), "dK": dk.cpu(), "dV": dv.cpu()})
    for name in ("dQ", "dK", "dV"):
        assert torch.equal(runs[0][name], runs[1][name]), f"{name} differs between identical runs"
    assert torch.equal(runs[0]["dK"], fused["dK"]) and torch.equal(runs[0]["dV"], fused["dV"])
    got = dict(fused)
    got.update(runs[0])
    heads = None if B * H <= 8 else sorted({(i % B, (i * 5 + 1) % H) for i in range(4)})
    ref = h.run_oracle(Q, K, V, dO, cfg.scale, causal, heads=heads)
    h.compare(h.select_heads(got, heads), ref, label=f"deterministic T={T} D={D}: ", dO=ref["dO_in"])


def _random_case(rng):
    """One random problem: shape (ragged and exact tile counts mixed), mask, scale, input amplitude, entry point."""
    D = int(rng.choice([64, 64, 128]))
    kind = rng.random()
    if kind < 0.45:
        T = int(rng.integers(1, 700))
    elif kind < 0.8:
        T = int(rng.choice([127, 128, 129, 255, 256, 257, 383, 384, 385, 511, 512, 513, 640, 1000, 1024, 1025]))
    else:
        T = int(rng.integers(700, 2300))
    bh_max = max(1, min(40, 60000 // (T + 64)))
    B = int(rng.integers(1, min(4, bh_max) + 1))
    H = int(rng.integers(1, max(1, bh_max // B) + 1))
    causal = bool(rng.random() < 0.7)
    # score standard deviation amp^2 * factor stays <= 1: the range of the graded configurations
    factor, amp = float(rng.choice([1.0, 1.0, 0.5])), float(rng.choice([1.0, 1.0, 0.5]))
    path = str(rng.choice(["plain", "plain", "deterministic", "strided", "static"]))
    return B, H, T, D, causal, factor * D ** -0.5, amp, path


@pytest.mark.parametrize("chunk", range(4))
def test_random_shapes_and_entry_points(chunk):
    """Seeded random problems (16 per chunk) through the four backward entry points, each against the
    oracle on up to six heads: shapes the hand-picked lists do not name."""
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(9000 + chunk)
    for case in range(16):
        B, H, T, D, causal, scale, amp, path = _random_case(rng)
        g = torch.Generator().manual_seed(9000 * (chunk + 1) + case)
        Q, K, V, dO = ((a * torch.randn(B, H, T, D, generator=g)).to(torch.bfloat16) for a in (amp, amp, 1.0, 1.0))
        label = f"random {chunk}/{case} B={B} H={H} T={T} D={D} causal={causal} scale={scale:.4f} amp={amp} {path}: "
        if path == "plain":
            got = h.run_gpu(Q, K, V, dO, scale, causal)
        elif path == "strided":
            qkv = torch.empty((B, T, 3, H, D), dtype=torch.bfloat16, device=dev)
            for i, x in enumerate((Q, K, V)):
                qkv[:, :, i] = x.to(dev).permute(0, 2, 1, 3)
            q_v, k_v, v_v = (qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))
            o_v = torch.full((B, T, H, D), 7.0, dtype=torch.bfloat16, device=dev).permute(0, 2, 1, 3)
            do_v = dO.to(dev).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
            dqkv = torch.full((B, T, 3, H, D), 7.0, dtype=torch.bfloat16, device=dev)
            dq_v, dk_v, dv_v = (dqkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))
            lse = torch.empty((B, H, T), dtype=torch.float32, device=dev)
            delta = torch.empty_like(lse)
            nova_attn.nova_attn_fwd_strided(q_v, k_v, v_v, o_v, lse, scale, causal)
            nova_attn.nova_attn_bwd_preprocess_strided(o_v, do_v, delta)
            nova_attn.nova_attn_bwd_strided(q_v, k_v, v_v, do_v, lse, delta, dq_v, dk_v, dv_v, scale, causal)
            got = {"O": o_v.contiguous().cpu(), "LSE": lse.cpu(), "Delta": delta.cpu(),
                   "dQ": dq_v.contiguous().cpu(), "dK": dk_v.contiguous().cpu(), "dV": dv_v.contiguous().cpu()}
        else:
            q, k, v, do = (x.to(dev) for x in (Q, K, V, dO))
            o, dq, dk, dv = (torch.full((B, H, T, D), 7.0, dtype=torch.bfloat16, device=dev) for _ in range(4))
            lse = torch.empty((B, H, T), dtype=torch.float32, device=dev)
            delta = torch.empty_like(lse)
            nova_attn.nova_attn_fwd(q, k, v, o, lse, scale, causal)
            nova_attn.nova_attn_bwd_preprocess(o, do, delta)
            if path == "deterministic":
                nova_attn.nova_attn_bwd_deterministic(q, k, v, do, lse, delta, dq, dk, dv, scale, causal)
            else:
                nova_attn.nova_attn_bwd_static_scratch(q, k, v, o, do, lse, delta, dq, dk, dv, scale, causal)
            got = {"O": o.cpu(), "LSE": lse.cpu(), "Delta": delta.cpu(), "dQ": dq.cpu(), "dK": dk.cpu(), "dV": dv.cpu()}
        nova_attn.nova_attn_poll_device_status()
        for name, t in got.items():
            assert torch.isfinite(t.float()).all(), f"{label}{name} is not finite"
        heads = sorted({((i * 7919 + case) % B, (i * 104729 + case) % H) for i in range(min(B * H, 6))})
        ref = h.run_oracle(Q, K, V, dO, scale, causal, heads=heads)
        h.compare(h.select_heads(got, heads), ref, label=label, dO=ref["dO_in"], rms=(T >= 64))


def test_binding_takes_numbers_as_python_does():
    """scale and steps are read as float() and int() read them."""
    from decimal import Decimal

    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    x = torch.randn((1, 2, 100, 64), device=dev).to(torch.bfloat16)
    row = torch.zeros((1, 2, 100), device=dev)
    out = []
    for scale, steps in ((0.125, 7), ("0.125", "7"), (Decimal("0.125"), 7.0), (np.float32(0.125), np.int64(7)),
                         (torch.tensor(0.125), torch.tensor(7))):
        o, lse, grads = torch.empty_like(x), torch.empty_like(row), [torch.empty_like(x) for _ in range(3)]
        nova_attn.nova_attn_fwd(x, x, x, o, lse, scale)
        nova_attn.nova_attn_bwd(x, x, x, o, x, lse, row, *grads, scale, steps=steps)
        out.append(torch.stack([o] + grads))
    assert all(torch.equal(t, out[0]) for t in out)


@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("kind", ["on the CPU", "strided"])
def test_backward_refuses_a_workspace_the_kernels_could_not_address(strided, kind):
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    x = torch.zeros((1, 1, 130, 64), dtype=torch.bfloat16, device=dev)
    row = torch.zeros((1, 1, 130), device=dev)
    need = nova_attn.nova_attn_bwd_workspace_bytes(1, 1, 130, 64)
    ws = (torch.empty(need, dtype=torch.uint8) if kind == "on the CPU"
          else torch.empty((need, 2), dtype=torch.uint8, device=dev)[:, 0])
    grads = [torch.full_like(x, 7.0) for _ in range(3)]
    with pytest.raises(TypeError, match="workspace"):
        if strided:
            nova_attn.nova_attn_bwd_strided(x, x, x, x, row, row, *grads, 0.125, True, ws)
        else:
            nova_attn.nova_attn_bwd(x, x, x, x, x, row, row, *grads, 0.125, True, ws)
    torch.cuda.synchronize()
    assert all(bool((g == 7.0).all()) for g in grads)


def test_workspace_of_the_call_belongs_to_its_stream():
    """A call without a workspace allocates one and gives it back before its kernels have run.  On a stream other than the
    current one that memory must not go to the next tensor of the current stream: here the call waits behind a copy
    that keeps its stream busy, and a tensor of the same size, made meanwhile, keeps its values."""
    from paper_2608_00029_b200 import nova_attn, nova_lmhead
    dev = torch.device("cuda:0")
    shape = (2, 3, 1000, 64)
    x = torch.randn(shape, device=dev).to(torch.bfloat16)
    row, grads = torch.zeros(shape[:3], device=dev), [torch.empty_like(x) for _ in range(3)]
    X, Wm = torch.zeros((512, 64), dtype=torch.bfloat16, device=dev), torch.zeros((4096, 64), dtype=torch.bfloat16, device=dev)
    t, lse, loss = torch.zeros(512, dtype=torch.int32, device=dev), torch.empty(512, device=dev), torch.empty(512, device=dev)
    side, big = torch.cuda.Stream(device=dev), torch.empty(1 << 30, dtype=torch.uint8, device=dev)
    calls = [(nova_attn.nova_attn_bwd_workspace_bytes(*shape),
              lambda: nova_attn.nova_attn_bwd(x, x, x, x, x, row, row, *grads, 0.125, True, stream=side)),
             (nova_attn.nova_attn_bwd_workspace_bytes(*shape),
              lambda: nova_attn.nova_attn_bwd_strided(x, x, x, x, row, row, *grads, 0.125, True, stream=side)),
             (nova_lmhead.nova_lmhead_workspace_bytes(512, 4096, 64),
              lambda: nova_lmhead.nova_lmhead_fwd(X, Wm, t, None, lse, loss, stream=side))]
    for need, call in calls:
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            for _ in range(40):
                big.fill_(1)
        call()
        mine = torch.full((need,), 7, dtype=torch.uint8, device=dev)
        torch.cuda.synchronize()
        nova_attn.nova_attn_poll_device_status()
        assert bool((mine == 7).all())


def test_two_host_threads_two_streams():
    """Two host threads drive the library at once, each on its own stream and buffers (different shapes
    and head dimensions): the calls take the library's lock for the map cache only, the kernels of the
    two streams share the SMs, and every result is bit-identical to the single-threaded run (dQ within
    its reduce-order noise)."""
    import threading
    from paper_2608_00029_b200 import nova_attn
    h = _harness()
    dev = torch.device("cuda:0")
    cfgs = [W.AttnConfig("mt0", B=2, H=6, T=1024, D=64, seed=811, causal=True),
            W.AttnConfig("mt1", B=1, H=5, T=700, D=128, seed=812, causal=True)]
    inputs = [W.make_inputs(c) for c in cfgs]
    single = [h.run_gpu(*inp, c.scale, True) for inp, c in zip(inputs, cfgs)]
    results = [None, None]
    errors = []

    def worker(i):
        try:
            cfg = cfgs[i]
            stream = torch.cuda.Stream(device=dev)
            with torch.cuda.stream(stream):
                q, k, v, do = (x.to(dev) for x in inputs[i])
                shape = (cfg.B, cfg.H, cfg.T, cfg.D)
                o, dq, dk, dv = (torch.empty(shape, dtype=torch.bfloat16, device=dev) for _ in range(4))
                lse = torch.empty(shape[:3], dtype=torch.float32, device=dev)
                delta = torch.empty_like(lse)
                ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(*shape), dtype=torch.uint8, device=dev)
                for _ in range(40):
                    nova_attn.nova_attn_fwd(q, k, v, o, lse, cfg.scale, True, stream=stream)
                    nova_attn.nova_attn_bwd_preprocess(o, do, delta, stream=stream)
                    nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, dq, dk, dv, cfg.scale, True, ws, stream=stream)
                stream.synchronize()
                results[i] = {"O": o.cpu(), "LSE": lse.cpu(), "Delta": delta.cpu(), "dQ": dq.cpu(), "dK": dk.cpu(),
                              "dV": dv.cpu()}
        except Exception as e:  # surfaced in the main thread
            errors.append((i, repr(e)))

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    nova_attn.nova_attn_poll_device_status()
    for i in range(2):
        for name in ("O", "LSE", "Delta", "dK", "dV"):
            assert torch.equal(results[i][name], single[i][name]), f"thread {i}: {name} differs from the single-threaded run"
        d = (results[i]["dQ"].float() - single[i]["dQ"].float()).abs().max()
        assert d <= 1e-2 * single[i]["dQ"].float().abs().max()


@pytest.mark.parametrize("B,H,D", [(2, 5, 64), (12, 12, 64), (12, 12, 128)])  # single query tiles; pairs, D=128 two kernels
def test_cuda_graph_capture_and_replay(B, H, D):
    """The calls only enqueue work, so a step can be captured into a CUDA graph and replayed (what bench.py
    times): the replay writes the same O, LSE, Delta, dK, dV bits as the eager calls, and dQ within its
    reduce-order noise, also when replayed repeatedly."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    cfg = W.AttnConfig("graph", B=B, H=H, T=900, D=D, seed=905, causal=True)
    q, k, v, do = (x.to(dev) for x in W.make_inputs(cfg))
    shape = (cfg.B, cfg.H, cfg.T, cfg.D)
    o, dq, dk, dv = (torch.empty(shape, dtype=torch.bfloat16, device=dev) for _ in range(4))
    lse = torch.empty(shape[:3], dtype=torch.float32, device=dev)
    delta = torch.empty_like(lse)
    ws = torch.empty(nova_attn.nova_attn_bwd_workspace_bytes(*shape), dtype=torch.uint8, device=dev)

    def step():
        nova_attn.nova_attn_fwd(q, k, v, o, lse, cfg.scale, True)
        nova_attn.nova_attn_bwd_preprocess(o, do, delta)
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, dq, dk, dv, cfg.scale, True, ws)

    outs = {"O": o, "LSE": lse, "Delta": delta, "dQ": dq, "dK": dk, "dV": dv}
    side = torch.cuda.Stream(device=dev)
    with torch.cuda.stream(side):
        step()  # also fills the tensor-map cache before the capture
    side.synchronize()
    eager = {n: t.clone() for n, t in outs.items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        step()
        step()
    for rep in range(3):
        for n, t in outs.items():
            t.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        nova_attn.nova_attn_poll_device_status()
        for n in ("O", "LSE", "Delta", "dK", "dV"):
            assert torch.equal(outs[n], eager[n]), f"replay {rep}: {n} differs from the eager calls"
        d = (outs["dQ"].float() - eager["dQ"].float()).abs().max()
        assert d <= 1e-2 * eager["dQ"].float().abs().max()


def _layout_view(x, kind, rng, dev):
    """A [B,H,T,D] view with the strides of layout `kind` holding the values of x (storage pre-filled with 7)."""
    B, H, T, D = x.shape
    if kind == "bthd":
        st = torch.empty((B, T, H, D), dtype=x.dtype, device=dev)
        v = st.permute(0, 2, 1, 3)
    elif kind == "pad_t":  # padded token stride
        st = torch.empty((B, H, T, D + 8 * int(rng.integers(1, 5))), dtype=x.dtype, device=dev)
        v = st[..., :D]
    elif kind == "pad_h":  # padded head stride
        st = torch.empty((B, H, T + int(rng.integers(1, 6)), D), dtype=x.dtype, device=dev)
        v = st[:, :, :T]
    elif kind == "hbtd":   # heads outermost
        st = torch.empty((H, B, T, D), dtype=x.dtype, device=dev)
        v = st.permute(1, 0, 2, 3)
    elif kind == "tbhd":   # tokens outermost
        st = torch.empty((T, B, H, D), dtype=x.dtype, device=dev)
        v = st.permute(1, 2, 0, 3)
    else:
        st = torch.empty((B, H, T, D), dtype=x.dtype, device=dev)
        v = st
    st.fill_(7.0)
    v.copy_(x)
    return v, st


def test_random_tensor_layouts():
    """Every bf16 tensor of the strided entry points in a layout of its own (plain, [B,T,H,D], padded token
    or head stride, heads or tokens outermost), 60 seeded cases: only addressing changes, so O, LSE, Delta,
    dK, dV are bit-identical to the plain entry points, dQ within its reduce-order noise, and nothing is
    written between the rows of a padded output."""
    from paper_2608_00029_b200 import nova_attn
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(4242)
    kinds = ["bhtd", "bthd", "pad_t", "pad_h", "hbtd", "tbhd"]
    for case in range(60):
        D = int(rng.choice([64, 128]))
        T = int(rng.choice([1, 5, 64, 127, 128, 129, 200, 256, 300, 511, 640, 1000]))
        B, H = int(rng.integers(1, 4)), int(rng.integers(1, 6))
        causal = bool(rng.random() < 0.7)
        scale = D ** -0.5
        g = torch.Generator().manual_seed(4242 + case)
        q, k, v, do = (torch.randn(B, H, T, D, generator=g).to(torch.bfloat16).to(dev) for _ in range(4))
        o, dq, dk, dv = (torch.empty((B, H, T, D), dtype=torch.bfloat16, device=dev) for _ in range(4))
        lse = torch.empty((B, H, T), dtype=torch.float32, device=dev)
        delta = torch.empty_like(lse)
        nova_attn.nova_attn_fwd(q, k, v, o, lse, scale, causal)
        nova_attn.nova_attn_bwd_preprocess(o, do, delta)
        nova_attn.nova_attn_bwd(q, k, v, o, do, lse, delta, dq, dk, dv, scale, causal)
        ks = [str(rng.choice(kinds)) for _ in range(8)]
        (q_v, _), (k_v, _), (v_v, _), (do_v, _) = (_layout_view(x, kd, rng, dev) for x, kd in zip((q, k, v, do), ks[:4]))
        outs = [_layout_view(torch.full_like(q, 7.0), kd, rng, dev) for kd in ks[4:]]
        (o_v, o_st), (dq_v, dq_st), (dk_v, dk_st), (dv_v, dv_st) = outs
        lse2, delta2 = torch.empty_like(lse), torch.empty_like(delta)
        nova_attn.nova_attn_fwd_strided(q_v, k_v, v_v, o_v, lse2, scale, causal)
        nova_attn.nova_attn_bwd_preprocess_strided(o_v, do_v, delta2)
        nova_attn.nova_attn_bwd_strided(q_v, k_v, v_v, do_v, lse2, delta2, dq_v, dk_v, dv_v, scale, causal)
        nova_attn.nova_attn_poll_device_status()
        label = f"layouts case {case} B={B} H={H} T={T} D={D} causal={causal} {ks}: "
        for name, a, b in (("O", o_v, o), ("LSE", lse2, lse), ("Delta", delta2, delta), ("dK", dk_v, dk), ("dV", dv_v, dv)):
            assert torch.equal(a.contiguous(), b), label + name + " differs from the plain entry points"
        d = (dq_v.float() - dq.float()).abs().max()
        assert d <= 1e-2 * max(float(dq.float().abs().max()), 1e-3), label + "dQ"
        for name, view, st in (("O", o_v, o_st), ("dQ", dq_v, dq_st), ("dK", dk_v, dk_st), ("dV", dv_v, dv_st)):
            view.fill_(7.0)  # what is left must be the untouched padding
            assert bool((st == 7.0).all()), label + name + ": write outside the rows of the view"
