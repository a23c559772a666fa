"""Cases for timing the measure -> recover -> execute FFN step as programs use it.

What a case stands for is its "kind":
  step     one decode step of one layer for B tokens, called directly (cs_layer_step with all outputs)
  stack    the FFN layers of one decode step, RMSNorm and residual included, captured once in a CUDA graph and
           replayed per token.  The layers' inputs are separate hidden states: in a model the attention
           block stands between one FFN and the next
  host     one decode step on page-locked host buffers, ending when the result may be read
  control  the online loop: entropy of the previous logits and the measurement budget it sets, then a
           warm-started step from the previous token's support, with the drift between the two
  prompt   one prompt through one layer: support from the mean prompt sketch, then the FFN of every token

Shapes are those of gen/workloads.py (Llama-2-7B / Llama-3-8B / Llama-2-13B feed-forward layers, and the tiny f32
layer), batches and prompt lengths those around them.  Hidden states carry a planted support plus noise, weights
are N(0, 1/fan_in), as in gen/workloads.py; everything is drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

import paper_2604_14156_b200 as cs

_L2_7B = dict(d=4096, d_ff=11008, group=128, m=32, k=22, T=20, weights="bf16")
_L3_8B = dict(d=4096, d_ff=14336, group=128, m=48, k=28, T=20, weights="bf16")
_L2_13B = dict(d=5120, d_ff=13824, group=128, m=64, T=20, weights="bf16")
_TINY = dict(d=256, d_ff=1024, group=64, m=8, k=4, T=10, weights="f32")
_SIGMA = 0.05          # noise of the hidden states
_WARM_T = 5            # iterations of a warm-started recovery


def listed():
    return [
        # the smallest call: a toy f32 layer, four tokens; nothing but latency and launches
        dict(name="tiny_f32_b4", kind="step", B=4, **_TINY),
        # interactive decoding of one sequence, called layer by layer
        dict(name="step_7b_b1", kind="step", B=1, **_L2_7B),
        # a few sequences at once: below the batch from which the tensor cores take over
        dict(name="step_7b_b3", kind="step", B=3, **_L2_7B),
        # a serving batch
        dict(name="step_7b_b64", kind="step", B=64, **_L2_7B),
        # an odd batch beyond one tile of tokens
        dict(name="step_7b_b200", kind="step", B=200, **_L2_7B),
        # a model's worth of layers for one sequence, as a server replays it
        dict(name="stack_8b_b1", kind="stack", layers=16, B=1, **_L3_8B),
        # the 32-layer stack at its batch of 32
        dict(name="stack_8b_b32", kind="stack", layers=32, B=32, **_L3_8B),
        # activations in host memory, there and back
        dict(name="host_7b_b1", kind="host", B=1, **_L2_7B),
        # the online controller around a step of a small, odd batch
        dict(name="control_7b_b11", kind="control", V=32000, B=11, **_L2_7B),
        # prompts: a short ragged one at 10 % of the groups, the 2048-token one at 25 %, a long one at 50 %
        dict(name="prompt_13b_k11_n777", kind="prompt", B=777, k=11, **_L2_13B),
        dict(name="prompt_13b_k27_n2048", kind="prompt", B=2048, k=27, **_L2_13B),
        dict(name="prompt_13b_k54_n4096", kind="prompt", B=4096, k=54, **_L2_13B),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["step", "stack", "host", "control", "prompt"], [8, 3, 2, 3, 6])[0]
    case = dict(kind=kind)
    small = kind == "step" and rng.random() < 0.25
    if small:              # toy and test layers: either weight type, 64- or 128-channel groups, odd widths
        group = rng.choice([64, 128])
        G = rng.randint(8, 24)
        d, B, weights = 64 * rng.randint(4, 16), _log_int(rng, 1, 16), rng.choice(["f32", "bf16"])
    else:                  # model layers
        group, weights = 128, "bf16"
        G = rng.randint(40, 128)
        d = 256 * rng.randint(8, 24)
        if kind == "prompt":
            B = _log_int(rng, 100, 4096)
        elif kind == "control":
            B = _log_int(rng, 1, 64)
        else:
            B = _log_int(rng, 1, {"step": 256, "stack": 64, "host": 64}[kind])
    k = max(2, round(G * rng.uniform(0.1, 0.5)))
    if kind == "prompt":   # no dearer than the largest listed prompt
        B = min(B, int(4096 * 54 * 5120 / (k * d)))
    case.update(d=d, d_ff=G * group, group=group, m=rng.randint(max(4, G // 4), max(5, min(64, G // 2 + 8))), k=k,
                T=rng.randint(8, 20), weights=weights, B=B)
    if kind == "stack":
        case["layers"] = rng.randint(4, 16)
    if kind == "control":
        case["V"] = rng.choice([32000, 50257, 128256])
    return case


def _normal(gen, shape, std, dtype=torch.float32):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)


def _layer(case, plan, gen, norm=False):
    """Parameters of one layer; returns the library's handle and the probe the hidden states are planted with."""
    d, d_ff, m, G = case["d"], case["d_ff"], case["m"], plan.G
    A = _normal(gen, (G, d), 1.0, torch.float64)
    A /= A.norm(dim=1, keepdim=True)
    Phi = _normal(gen, (m, G), 1.0 / math.sqrt(m))
    S = (Phi.double() @ A).float()
    mu = 1.0 / float(torch.linalg.matrix_norm(Phi.cpu().double(), 2)) ** 2
    wt = plan.w_dtype
    Wg, Wu = (_normal(gen, (d_ff, d), 1.0 / math.sqrt(d), wt) for _ in range(2))
    Wdt = _normal(gen, (d_ff, d), 1.0 / math.sqrt(d_ff), wt)
    gamma = 1.0 + _normal(gen, (d,), 0.1) if norm else None
    return cs.Layer(plan, S, Phi, Wg, Wu, Wdt, mu, gamma, norm), A.float()


def _planted(gen, A, k, B):
    """Hidden states [B, d] on independent k-subsets of the probe; also the subsets (ascending) and coefficients."""
    G = A.shape[0]
    order = torch.rand((B, G), device="cuda", generator=gen).argsort(dim=1)
    sup = order[:, :k].sort(dim=1).values
    c = _normal(gen, (B, k), 1.0)
    z = torch.zeros((B, G), device="cuda").scatter_(1, sup, c)
    return z @ A + _normal(gen, (B, A.shape[1]), _SIGMA), sup.int(), c


def _prompt_states(gen, A, k, n):
    """Hidden states of a prompt: one support, coefficients around a mean that is at least 0.5 in magnitude."""
    rows = A[torch.rand((A.shape[0],), device="cuda", generator=gen).argsort()[:k]]
    cbar = _normal(gen, (k,), 1.0)
    cbar = torch.where(cbar < 0, cbar.clamp(max=-0.5), cbar.clamp(min=0.5))
    c = cbar + _normal(gen, (n, k), 0.25)
    return (c @ rows + _normal(gen, (n, A.shape[1]), _SIGMA)).bfloat16()


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    plan = cs.Plan(case["d"], case["d_ff"], case["group"], case["m"], case["k"], case["T"],
                   torch.float32 if case["weights"] == "f32" else torch.bfloat16, case["B"])
    kind, B, k = case["kind"], case["B"], case["k"]
    state = dict(kind=kind, plan=plan)
    if kind == "stack":
        pairs = [_layer(case, plan, gen, norm=True) for _ in range(case["layers"])]
        xs = [_planted(gen, A, k, B)[0] for _, A in pairs]
        outs = torch.empty((len(pairs), B, case["d"]), device="cuda")

        def layers():
            for (lay, _), x, out in zip(pairs, xs, outs):
                cs.cs_layer_step(plan, lay, x, x_out=out, want_aux=False)

        layers()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            layers()
        state.update(graph=graph, outs=outs, keep=(pairs, xs))
        return state
    layer, A = _layer(case, plan, gen)
    state["layer"] = layer
    if kind == "prompt":
        state["x"] = _prompt_states(gen, A, k, B)
        return state
    x, sup, c = _planted(gen, A, k, B)
    if kind == "host":
        state.update(x=x.cpu().pin_memory(), out=torch.empty(x.shape).pin_memory())
        return state
    state["x"] = x
    if kind == "control":   # the previous token: the state before a small drift, and its support
        state["x"] = x + _normal(gen, x.shape, 0.02)
        state["logits"] = _normal(gen, (B, case["V"]), 2.0)
        state["options"] = cs.StepOptions(plan, B, T=_WARM_T, support_prev=sup, z_prev=c, warm_start=True, want_drift=True)
    return state


def run(state):
    kind, plan = state["kind"], state["plan"]
    if kind == "step":
        return cs.cs_layer_step(plan, state["layer"], state["x"])
    if kind == "stack":
        state["graph"].replay()
        return state["outs"]
    if kind == "host":
        cs.cs_layer_step_host(plan, state["layer"], state["x"], state["out"])
        torch.cuda.current_stream().synchronize()   # the caller reads the buffer next
        return state["out"]
    if kind == "control":
        opt = state["options"]
        budget = cs.cs_uds_budget(plan, state["logits"], plan.m / 4, 0.15, max(1, plan.m // 8), plan.m)
        step = cs.cs_layer_step_ex(plan, state["layer"], state["x"], opt)
        return budget, step, opt.delta, opt.drift
    layer, H = state["layer"], state["x"]
    support, z, resid = cs.cs_prompt_support(plan, layer.S, layer.Phi, layer.mu, H)
    return cs.cs_ffn_exec_shared(plan, layer, H, support), support, z, resid


def work(case):
    """Weights of the groups that some token uses (a prompt's tokens share theirs), the sketch, activations in and out."""
    d, b, m, k, B = case["d"], case["group"], case["m"], case["k"], case["B"]
    G = case["d_ff"] // b
    wbytes = 4 if case["weights"] == "f32" else 2
    prompt = case["kind"] == "prompt"
    union = k if prompt else G * (1.0 - (1.0 - k / G) ** B)   # expected, for independent supports
    layers = case.get("layers", 1)
    nbytes = 3 * union * b * d * wbytes + 4 * m * (d + G) + 2 * B * d * (2 if prompt else 4)
    flops = 6.0 * B * k * b * d + 2.0 * m * d * (1 if prompt else B)
    if case["kind"] == "control":
        nbytes += 4.0 * B * case["V"]
    return {"bytes": layers * nbytes, "flops": layers * flops}


def tolerance(case):
    # Against the same path in 64 bits: f32 activations 1e-5 to 2e-5 on the tensor cores (activations enter as two
    # bf16 parts) and below 1e-6 otherwise, bf16 activations (prompts) 2.4e-3 in all and 1.1e-2 at most.  Supports
    # may differ where two magnitudes tie.
    if case["kind"] == "prompt":
        return {"rel": 1e-2, "max": 5e-2, "differ": 0.01}
    return {"rel": 8e-5, "max": 3e-4, "differ": 0.01}
