"""GPU parity of the tensor-core decode path (up to 256 tokens) at the sizes where its tiling can go wrong."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_14156_b200 as cs

from gen import workloads as W
from parity_util import TIGHT_TOL, compare_layer_step, device_layer, make_plan, rel

pytestmark = pytest.mark.gpu


# Token tiles: packed value / remainder rows up to 64 tokens, two operands up to 128, two accumulators up to 256, and the
# first batch beyond.  Channel tiles: d_ff that the tiles of 8 x SM-share channels do not divide, and fewer channels than
# SMs x 8.  k small against G leaves groups out of every support.
@pytest.mark.parametrize("B", [2, 8, 15, 63, 64, 65, 127, 128, 129, 192, 193, 256, 257])
@pytest.mark.parametrize("d,G,m,k,norm", [(512, 13, 9, 3, True), (768, 101, 35, 11, False)])
def test_layer_step_token_and_channel_tile_edges(B, d, G, m, k, norm):
    base = W.CONFIGS["l3_8b_stack" if norm else "l2_7b_b64"]
    cfg = base.with_(n_layers=1, d=d, d_ff=128 * G, m=m, k=k, T=6, B=B, index=300 + B)
    L = W.make_layer(cfg, device="cuda:0")
    tk = W.make_tokens(cfg, L.A)
    plan = make_plan(cfg)
    plan.set_crossover(2)
    # output bound: 1e-4 (parity_util), f32 accumulation of bf16 value + remainder products
    rep, _, _ = compare_layer_step(cfg, L, plan, tk.h)
    assert rep.excused <= max(1, B // 16), rep
    plan.close()


# Gather path: a step's form of the kernel against the one for given supports, the same bits.  Rows that are whole slices of 512 chunks
# (one, two and four a thread); rows that are not have one form for both.
@pytest.mark.parametrize("dtype,d", [("bf16", 4096), ("bf16", 8192), ("bf16", 5120), ("bf16", 320), ("f32", 2048), ("f32", 8192), ("f32", 2112), ("f32", 64)])
def test_gather_step_and_given_supports_agree(dtype, d):
    cfg = W.CONFIGS["l2_7b_b64"].with_(n_layers=1, w_dtype=dtype, d=d, d_ff=64 * 20, group=64, m=12, k=5, T=6, B=2, index=350)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    lay, x = device_layer(plan, L), W.make_tokens(cfg, L.A).h.to("cuda:0")
    out, sup, _, _ = cs.cs_layer_step(plan, lay, x)
    assert torch.equal(cs.cs_ffn_exec(plan, lay, x, sup), out) and plan.device_status() == 0
    plan.close()


# Pairs of CTAs, more than 128 tokens: halves of the tokens that are no multiple of 8, a last pair whose second CTA has channels past d_ff or
# none, fewer pairs than SMs, the recovery's list lengths.
@pytest.mark.parametrize("B,norm", [(131, False), (145, True), (255, False)])
@pytest.mark.parametrize("d,G,m,k", [(256, 5, 4, 2), (256, 91, 40, 30), (512, 107, 33, 50)])
def test_layer_step_on_pairs_of_ctas(d, G, m, k, B, norm):
    cfg = W.CONFIGS["l3_8b_stack" if norm else "l2_7b_b64"].with_(n_layers=1, d=d, d_ff=128 * G, m=m, k=k, T=6, B=B, index=340 + B)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    rep, _, _ = compare_layer_step(cfg, L, plan, W.make_tokens(cfg, L.A).h)   # output bound 1e-4 (parity_util)
    assert rep.excused <= max(1, B // 16), rep
    plan.close()


# The same in layers so narrow that pairs without channels join in to recover: one and two tokens a CTA, the last CTA without any.
@pytest.mark.parametrize("B", [129, 148, 149, 200, 255, 256])
@pytest.mark.parametrize("d,G,m,k", [(256, 1, 2, 1), (256, 8, 6, 3), (1024, 24, 12, 6)])
def test_layer_step_on_pairs_of_ctas_narrow_layers(d, G, m, k, B):
    cfg = W.CONFIGS["l2_7b_b64"].with_(n_layers=1, d=d, d_ff=128 * G, m=m, k=k, T=6, B=B, index=360 + B)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    rep, _, _ = compare_layer_step(cfg, L, plan, W.make_tokens(cfg, L.A).h)   # output bound 1e-4 (parity_util)
    assert rep.excused <= max(1, B // 16), rep
    plan.close()


# Gather path: few rows for many CTAs, and three or four tokens of 55 to 60 groups.
@pytest.mark.parametrize("k,B", [(55, 4), (56, 4), (60, 3), (1, 3)])
def test_gather_rows_per_cta_edges(k, B):
    cfg = W.CONFIGS["l2_7b_b64"].with_(d=256, d_ff=64 * 64, group=64, m=20, k=k, T=5, B=B, w_dtype="f32", index=360 + k)
    L = W.make_layer(cfg, device="cuda:0")
    tk = W.make_tokens(cfg, L.A)
    plan = make_plan(cfg)
    compare_layer_step(cfg, L, plan, tk.h)   # output bound 1e-5 (parity_util): f32 weights
    plan.close()


# Gather path, rows per CTA at the bound of 160: four tokens of 92 groups are 160 rows for each of 37 CTAs, of 93 groups two
# waves of CTAs; eight of 45 groups one wave; sixteen of 128 groups, several waves.
@pytest.mark.parametrize("k,B", [(92, 4), (93, 4), (45, 8), (128, 16)])
def test_gather_rows_per_cta_bound(k, B):
    cfg = W.CONFIGS["l2_7b_b64"].with_(d=256, d_ff=64 * 128, group=64, m=20, k=k, T=5, B=B, w_dtype="f32", index=380 + k)
    L = W.make_layer(cfg, device="cuda:0")
    tk = W.make_tokens(cfg, L.A)
    plan = make_plan(cfg)
    compare_layer_step(cfg, L, plan, tk.h)   # output bound 1e-5 (parity_util): f32 weights
    plan.close()


def _replay_us(fn, calls=16, replays=20):
    """Median microseconds of a call, captured back to back."""
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        fn()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(calls):
            fn()
    times = []
    for _ in range(replays):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record(); graph.replay(); b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 1e3 / calls)
    return sorted(times)[replays // 2]


def test_gather_grid_has_no_nearly_empty_wave():
    """Four tokens of the 8B layer are a third more rows than three (measured 1.2 times the time); a few CTAs past a whole wave
    of them made it 1.7 times."""
    cfg = W.CONFIGS["l3_8b_stack"].with_(n_layers=1, B=4)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    lay = device_layer(plan, L)
    h = W.make_tokens(cfg, L.A).h.to("cuda:0")
    us = {}
    for B in (3, 4):
        x, out = h[:B].contiguous(), torch.empty((B, cfg.d), device="cuda:0")
        us[B] = _replay_us(lambda: cs.cs_layer_step(plan, lay, x, out, want_aux=False))
    assert plan.crossover > 4 and us[4] <= 1.45 * us[3], us
    plan.close()


# Steps on changing tokens, launched without a pause: masks, token matrices or supports of the step before would show in the
# bits.  Few groups per token (the down GEMM's list is the union), nearly all groups in use, and the recovery as a launch
# of its own (k > 56); one, two and four 64-row boxes of tokens.
@pytest.mark.parametrize("k", [3, 40, 60])
@pytest.mark.parametrize("B", [5, 64, 130, 256])
def test_back_to_back_steps_on_changing_tokens(k, B):
    cfg = W.CONFIGS["l3_8b_stack"].with_(n_layers=1, d=1024, d_ff=128 * 100, m=40, k=k, T=6, B=B, index=460)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    plan.set_crossover(2)
    lay = device_layer(plan, L)
    h = W.make_tokens(cfg, L.A).h.to("cuda:0")
    xs = [h.roll(i, 0) * (1.0 + i) + 0.1 * i for i in range(4)]
    alone = []
    for x in xs:
        torch.cuda.synchronize()
        alone.append([t.clone() for t in cs.cs_layer_step(plan, lay, x)])
    torch.cuda.synchronize()
    runs = [cs.cs_layer_step(plan, lay, xs[i % 4]) for i in range(24)]
    for i, run in enumerate(runs):
        for a, b in zip(run, alone[i % 4]):
            assert torch.equal(a, b), i
    assert plan.device_status() == 0
    plan.close()


# Given supports; beyond 128 tokens gate/up runs over the groups in use (units of 16 channels shared by the CTAs).  One group, a few,
# an odd number, every group; fewer units than CTAs (3 groups), several a CTA, and a share no smaller than without the list; the
# three token forms.  Weights of the other groups are NaN: nothing of them may reach the output.
@pytest.mark.parametrize("G,k,used", [(3, 1, 1), (3, 2, 3), (40, 2, 5), (101, 3, 7), (101, 3, 101), (128, 6, 33)])
@pytest.mark.parametrize("B", [4, 33, 64, 65, 129, 193, 256])
def test_ffn_exec_over_the_groups_in_use(G, k, used, B):
    cfg = W.CONFIGS["l2_7b_b64"].with_(d=512, d_ff=128 * G, m=9, k=k, T=4, B=B, index=500 + G)
    L = W.make_layer(cfg, device="cuda:0")
    rng = np.random.default_rng(B + used)
    groups = np.sort(rng.permutation(G)[:used])
    sup = np.sort(np.stack([rng.permutation(groups)[:k] for _ in range(B)]), axis=1).astype(np.int32)
    Lc = L.to("cpu")
    unused = torch.ones(G, dtype=torch.bool); unused[torch.from_numpy(np.unique(sup)).long()] = False
    rows = unused.repeat_interleave(128).to("cuda:0")
    for w in (L.W_gate, L.W_up, L.Wd_t):
        w[rows] = float("nan")
    h = W.make_tokens(cfg, L.A).h
    plan = make_plan(cfg)
    plan.set_crossover(2)
    out = cs.cs_ffn_exec(plan, device_layer(plan, L), h.to("cuda:0"), torch.from_numpy(sup).to("cuda:0")).cpu().numpy()
    assert plan.device_status() == 0
    for t in sorted({0, 1, 63 % B, 64 % B, 127 % B, 128 % B, B // 2, B - 1}):
        ref = oracle.ffn(Lc.W_gate, Lc.W_up, Lc.Wd_t, cfg.group, h[t].double().numpy(), sup[t])
        assert rel(out[t], ref) <= TIGHT_TOL["bf16"], t   # f32 activations (parity_util)
    plan.close()


def test_ffn_exec_time_follows_the_groups_in_use():
    """200 tokens on the same 6 of 86 groups stream a fourteenth of the weights of 200 tokens on all of them."""
    cfg = W.CONFIGS["l2_7b_b64"].with_(B=200, k=6)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    lay = device_layer(plan, L)
    h = W.make_tokens(cfg, L.A).h.to("cuda:0")
    out = torch.empty_like(h)
    us = {}
    for name, stride in (("six", 0), ("all", 6)):
        sup = torch.stack([(torch.arange(6) + stride * t) % 86 for t in range(200)]).sort(dim=1).values.int().to("cuda:0")
        us[name] = _replay_us(lambda: cs.cs_ffn_exec(plan, lay, h, sup, out=out))
    assert us["six"] <= 0.75 * us["all"], us
    plan.close()


def test_stage_times_of_a_fused_step_forget_an_earlier_recovery():
    """The recovery inside the sensing launch (3 tokens) or the gate/up launch (40) has no time of its own, not an earlier call's."""
    cfg = W.CONFIGS["l2_7b_b64"].with_(d=512, d_ff=128 * 20, m=9, k=5, T=6, B=40, index=520)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    lay = device_layer(plan, L)
    x = W.make_tokens(cfg, L.A).h.to("cuda:0")
    plan.enable_timing()
    for B, fused in ((3, 0), (40, 2)):
        y = cs.cs_sketch(plan, L.S, x[:B].contiguous())
        cs.cs_recover(plan, L.Phi, L.mu, y)
        assert plan.stage_times()[1] > 0.0
        cs.cs_layer_step(plan, lay, x[:B].contiguous())
        ms = plan.stage_times()
        assert ms[1] == 0.0 and ms[fused] > 0.0, (B, ms)
    plan.close()


# Many groups per token: the recovery inside gate/up with 32, 56 and 64 slots, from 65 groups on as a launch of its own in
# front of it (the dense form), at the edges of the token forms, with and without the RMSNorm.
@pytest.mark.parametrize("k", [28, 40, 56, 57, 64, 65, 100])
@pytest.mark.parametrize("B,norm", [(3, True), (64, False), (65, True), (129, False), (256, True)])
def test_layer_step_many_groups_per_token(k, B, norm):
    cfg = W.CONFIGS["l3_8b_stack" if norm else "l2_7b_b64"].with_(
        n_layers=1, d=512, d_ff=128 * 120, m=40 + k % 2, k=k, T=6, B=B, index=540 + k)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    plan.set_crossover(2)
    rep, _, _ = compare_layer_step(cfg, L, plan, W.make_tokens(cfg, L.A).h)   # output bound 1e-4 (parity_util)
    assert rep.excused <= max(1, B // 16), rep
    plan.close()
