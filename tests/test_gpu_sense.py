"""GPU parity of the launch that senses and recovers a token on a cluster of CTAs, at the sizes where its split can go wrong."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_14156_b200 as cs
from gen import workloads as W
from parity_util import compare_layer_step, device_layer, make_plan, recovery_matches, rel

pytestmark = pytest.mark.gpu


# d: slices of two float4 columns, a ragged and a full last chunk per lane, the widest; m: fewer rows than warps, odd, rows of S
# that do not fit in shared memory beside a large M (8192 x 64); G: padded to 4, all four warps; k: the list form's lengths
# and the dense form; 16 and 17 tokens: the last batch on clusters and the first beyond.
@pytest.mark.parametrize("d,G,m,k,B,norm", [(64, 2, 1, 1, 1, False), (192, 5, 5, 2, 16, True), (320, 33, 7, 9, 17, False),
                                            (4096, 50, 33, 24, 2, True), (5120, 108, 64, 57, 1, False), (8192, 128, 64, 32, 2, True)])
def test_layer_step_sense_cluster_edges(d, G, m, k, B, norm):
    cfg = W.CONFIGS["l3_8b_stack" if norm else "l2_7b_b64"].with_(
        n_layers=1, w_dtype="f32", d=d, d_ff=64 * G, group=64, m=m, k=k, T=7, B=B, index=400 + G)
    L = W.make_layer(cfg, device="cuda:0")
    tk = W.make_tokens(cfg, L.A)
    plan = make_plan(cfg)
    rep, _, _ = compare_layer_step(cfg, L, plan, tk.h)   # output bound 1e-5 (parity_util): f32 weights
    assert rep.excused <= max(1, B // 16), rep
    plan.close()


# A plain step's form of the sensing launch (with or without the RMSNorm; there is one only where every row of S fits in shared memory)
# against the form for options, which a request for the drift takes: the same bits.  List lengths around 8, 16 and 24.
@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("d,G,m,k", [(256, 16, 8, 4), (320, 40, 20, 8), (1088, 70, 33, 9), (256, 100, 40, 16), (512, 128, 64, 17), (2048, 128, 64, 24),
                                     (2048, 128, 64, 25), (256, 128, 30, 64)])
def test_sense_launch_plain_and_general_forms_agree(d, G, m, k, norm):
    cfg = W.CONFIGS["l3_8b_stack" if norm else "l2_7b_b64"].with_(n_layers=1, w_dtype="f32", d=d, d_ff=64 * G, group=64, m=m, k=k, T=7, B=3,
                                                                  index=470 + k)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    lay, x = device_layer(plan, L), W.make_tokens(cfg, L.A).h.to("cuda:0")
    plain = cs.cs_layer_step(plan, lay, x)
    opt = cs.StepOptions(plan, 3, support_prev=plain[1].clone(), want_drift=True)
    for a, b in zip(plain, cs.cs_layer_step_ex(plan, lay, x, opt)):
        assert torch.equal(a, b)
    assert not opt.delta.any() and plan.device_status() == 0
    plan.close()


# Steps with a warm start, the temporal term and the drift, and the plain steps before them, against the oracle: rows of S that do not fit in
# shared memory (64 of 4096 beside 128 groups), where both kinds of step are one form, and rows that do.
@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("d,G,m,k", [(4096, 128, 64, 24), (4096, 128, 64, 25), (4096, 128, 64, 8), (320, 40, 20, 9), (192, 31, 12, 24), (512, 60, 33, 33)])
def test_sense_launch_options_match_oracle(d, G, m, k, norm):
    cfg = W.CONFIGS["l3_8b_stack" if norm else "l2_7b_b64"].with_(n_layers=1, w_dtype="f32", d=d, d_ff=64 * G, group=64, m=m, k=k, T=7, B=3,
                                                                  index=490 + k)
    L = W.make_layer(cfg, device="cuda:0")
    Lc = L.to("cpu")
    h, h2 = W.make_tokens(cfg, L.A).h, W.make_tokens(cfg, L.A, batch=1).h
    plan = make_plan(cfg)
    lay = device_layer(plan, L)
    rep, _, _ = compare_layer_step(cfg, L, plan, h)
    _, sup0, z0, _ = cs.cs_layer_step(plan, lay, h.to("cuda:0"))
    x = 0.9 * h + 0.1 * h2
    opt = cs.StepOptions(plan, 3, T=4, support_prev=sup0, z_prev=z0, warm_start=True, gamma=0.25, want_drift=True)
    out, sup, z, resid = (t.cpu().numpy() for t in cs.cs_layer_step_ex(plan, lay, x.to("cuda:0"), opt))
    assert plan.device_status() == 0
    excused = rep.excused
    for t in range(3):
        n = oracle.rmsnorm(x[t], Lc.gamma, cfg.rms_eps) if norm else x[t].double().numpy()
        y = oracle.sketch(Lc.S, n)
        prev = np.zeros(G)
        prev[sup0[t].cpu().numpy()] = z0[t].cpu().numpy()
        ref = oracle.iht_temporal(Lc.Phi, y, k, 4, L.mu, 0.25, prev, prev)
        excused += not recovery_matches(sup[t], z[t], float(resid[t]), ref, Lc.Phi.numpy(), y, (t,))
        want = oracle.ffn(Lc.W_gate, Lc.W_up, Lc.Wd_t, cfg.group, n, sup[t])
        want = want + x[t].double().numpy() if norm else want
        assert rel(out[t], want) <= 1e-5, t   # f32 weights, on the support that was recovered
    assert excused <= 1
    assert opt.delta.cpu().numpy().tolist() == oracle.support_drift(sup0.cpu().numpy(), sup).tolist()
    plan.close()


# What decides between the sensing launch and the sketch and recovery launches: tokens (clusters resident at once, 15 on B200),
# the bytes of S (128 KB per CTA: 8192 x 32, 8192 x 33), the list form (64 groups).  The dense form and its prompt.
@pytest.mark.parametrize("d,G,m,k,B", [(256, 16, 8, 4, 12), (256, 16, 8, 4, 15), (256, 16, 8, 4, 16), (8192, 40, 32, 9, 2), (8192, 40, 33, 9, 2),
                                       (1024, 128, 48, 56, 3), (1024, 128, 48, 57, 3), (1024, 128, 48, 64, 3), (1024, 128, 48, 65, 3),
                                       (1024, 70, 48, 68, 2), (1024, 128, 48, 128, 2)])
def test_layer_step_sense_launch_limits(d, G, m, k, B):
    cfg = W.CONFIGS["l2_7b_b64"].with_(n_layers=1, w_dtype="f32", d=d, d_ff=64 * G, group=64, m=m, k=k, T=7, B=B, index=480 + k)
    L = W.make_layer(cfg, device="cuda:0")
    plan = make_plan(cfg)
    rep, _, _ = compare_layer_step(cfg, L, plan, W.make_tokens(cfg, L.A).h)   # output bound 1e-5 (parity_util): f32 weights
    assert rep.excused <= max(1, B // 16), rep
    plan.close()


def test_sense_launch_is_taken_up_to_the_resident_clusters():
    """Launches of a step: sense + gather + reduction, or sketch + recovery + gather + reduction."""
    def launches(**kw):
        cfg = W.CONFIGS["tiny_f32"].with_(**kw)
        L = W.make_layer(cfg, device="cuda:0")
        plan = make_plan(cfg)
        lay, x = device_layer(plan, L), W.make_tokens(cfg, L.A).h.to("cuda:0")
        before = plan.launches
        cs.cs_layer_step(plan, lay, x)
        n = plan.launches - before
        plan.close()
        return n
    assert launches(B=1) == 3 and launches(B=8) == 3 and launches(B=16) == 4
    assert launches(B=2, d=8192, m=33, d_ff=64 * 40) == 4 and launches(B=2, d_ff=64 * 128, m=48, k=65) == 4


# prompt lengths around the row blocks (16) and the rows a CTA has in flight (64): remainders, fewer rows than blocks
@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 65, 1025])
def test_prompt_support_row_block_edges(n):
    cfg = W.CONFIGS["l2_13b_prompt"].with_(B=n, d=320, d_ff=128 * 20, k=6, m=40, index=430)
    L = W.make_layer(cfg, device="cuda:0")
    tk = W.make_tokens(cfg, L.A)
    plan = cs.Plan(cfg.d, cfg.d_ff, cfg.group, cfg.m, cfg.k, cfg.T, torch.bfloat16, n, cfg.rms_eps)
    sup, z, resid = cs.cs_prompt_support(plan, L.S, L.Phi, L.mu, tk.h.to("cuda:0"))
    y, ref = oracle.prompt_support(L.S.cpu(), L.Phi.cpu(), tk.h, cfg.k, cfg.T, L.mu)
    recovery_matches(sup.cpu().numpy(), z.cpu().numpy(), float(resid.cpu()[0]), ref, L.Phi.cpu().numpy(), np.asarray(y))
    assert plan.device_status() == 0
    plan.close()


# d / 32 float4 columns per CTA that 32 lanes do not divide: lanes past the end read a column that another lane copied.  A layer
# whose S is all NaN leaves NaN in every byte of shared memory such a read could find too early.
@pytest.mark.parametrize("d", [192, 256, 1088, 2304, 5376])
def test_sense_cluster_ragged_columns_after_nan_sketch(d):
    cfg = W.CONFIGS["l2_7b_b64"].with_(n_layers=1, w_dtype="f32", d=d, d_ff=64 * 20, group=64, m=30, k=6, T=5, B=4, index=440)
    L = W.make_layer(cfg, device="cuda:0")
    x = W.make_tokens(cfg, L.A).h.to("cuda:0")
    plan = make_plan(cfg)
    good = device_layer(plan, L)
    bad = cs.Layer(plan, torch.full_like(L.S, float("nan")), L.Phi, L.W_gate, L.W_up, L.Wd_t, L.mu)
    ref = [t.clone() for t in cs.cs_layer_step(plan, good, x)]
    assert plan.device_status() == 0 and all(torch.isfinite(t).all() for t in ref)
    for _ in range(20):
        cs.cs_layer_step(plan, bad, x)
        for a, b in zip(cs.cs_layer_step(plan, good, x), ref):
            assert torch.equal(a, b)
    plan.device_status()   # the NaN layer's report
    plan.close()
