"""What this library is timed on: the MoE FFN layer as speculative-decoding verification runs it.

A case names a layer shape of ``workloads.CONFIGS``, the batch (B sequences, gamma draft tokens
each: T = B * (gamma + 1) token rows), the routing (balanced, or Zipf-skewed through a router
bias), a variant of the layer where one is used (``top_k`` other than the model's, or the dense
layer of the same active parameters), and the entry: ``layer`` is ``moe_verify_layer``, the
whole layer in one call; ``stages`` is what a program with a router of its own calls -- grouping,
expert FFNs, combine -- on its top-k indices and gate weights.
"""
import math

import numpy as np
import torch

from paper_2505_19645_b200 import api, workloads as wl


def _case(shape, B, gamma, zipf=0.0, top_k=0, dense=False, entry="layer"):
    return {"shape": shape, "B": B, "gamma": gamma, "zipf": zipf, "top_k": top_k, "dense": dense,
            "entry": entry}


def listed():
    return [
        # the smallest layer: what a call costs where there is next to nothing to stream
        dict(_case("tiny", 4, 3), name="tiny_t16"),
        # one sequence, plain decoding (no draft tokens): the latency-bound end
        dict(_case("qwen1.5-moe-a2.7b", 1, 0), name="qwen15_t1"),
        # one sequence verifying four draft tokens
        dict(_case("qwen1.5-moe-a2.7b", 1, 4), name="qwen15_t5"),
        # an engine with its own router hands over its routing; an odd token count
        dict(_case("qwen1.5-moe-a2.7b", 11, 6, entry="stages"), name="qwen15_stages_t77"),
        # a large batch of a small model
        dict(_case("qwen1.5-moe-a2.7b", 128, 4), name="qwen15_t640"),
        # a skewed expert popularity, groups of one to a few hundred rows
        dict(_case("qwen2-57b-a14b", 64, 4, zipf=1.2), name="qwen2_zipf_t320"),
        # the compute-bound end of a wide shared expert and 64 routed ones
        dict(_case("qwen2-57b-a14b", 256, 4), name="qwen2_t1280"),
        # few experts with long reductions, a moderate batch
        dict(_case("mixtral-8x7b", 16, 4), name="mixtral_t80"),
        # few experts, compute-bound
        dict(_case("mixtral-8x7b", 256, 4), name="mixtral_t1280"),
        # one sequence on the largest layer
        dict(_case("deepseek-v3", 1, 3), name="deepseek_t4"),
        # the benchmark's headline: nearly every expert activated by a few tokens each
        dict(_case("deepseek-v3", 32, 3), name="deepseek_t128"),
        # the largest verify batch of the largest layer
        dict(_case("deepseek-v3", 512, 5), name="deepseek_t3072"),
    ]


# Largest token count per shape in draw(): the end of its benchmark grid, or of the tables beyond it.
_MAX_TOKENS = {"tiny": 640, "qwen1.5-moe-a2.7b": 640, "qwen2-57b-a14b": 2048, "mixtral-8x7b": 1280,
               "deepseek-v3": 3072}


def draw(rng):
    shape = rng.choice(["tiny"] + 2 * [n for n in wl.CONFIG_ORDER if n != "tiny"])
    gamma = rng.randint(0, 6)
    most = max(1, _MAX_TOKENS[shape] // (gamma + 1))
    B = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    zipf, top_k, dense = 0.0, 0, False
    if shape in ("qwen2-57b-a14b", "deepseek-v3") and rng.random() < 0.35:
        zipf = rng.choice([1.0, 1.2])
    elif shape == "qwen2-57b-a14b" and rng.random() < 0.3:
        # the sparsity sweep's variants (at most the model's own active parameters)
        if rng.random() < 0.3:
            dense = True
        else:
            top_k = rng.choice([k for k in wl.SPARSITY_TOP_KS if k < 8])
    entry = "stages" if rng.random() < 0.2 else "layer"
    return _case(shape, B, gamma, zipf, top_k, dense, entry)


def _shape(case):
    shape = wl.CONFIGS[case["shape"]]
    if case["dense"]:
        shape = wl.dense_contrast(shape)
    elif case["top_k"]:
        shape = wl.with_top_k(shape, case["top_k"])
    return shape


def prepare(case, seed):
    """Weights, token rows, output and workspace of one layer, as a serving program keeps them."""
    shape = _shape(case)
    B, gamma = case["B"], case["gamma"]
    T = B * (gamma + 1)
    w = wl.make_weights(shape, seed, "cuda", zipf_s=case["zipf"] or None)
    x = wl.make_tokens(shape, T, seed, "cuda")
    cfg = api.make_config(shape)
    state = {"entry": case["entry"], "B": B, "gamma": gamma, "w": w, "x": x, "cfg": cfg,
             "cw": api.make_weights(w), "ws": api.alloc_workspace(cfg, T),
             "out": torch.empty_like(x)}
    if case["entry"] == "stages":
        # the caller's routing: top-k of Gaussian logits (with the skew's bias where there is one)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 15485863)
        logits = torch.empty((T, shape.n_experts), device="cuda")
        logits.normal_(0.0, 0.02 * math.sqrt(shape.hidden), generator=gen)
        if w["router_bias"] is not None:
            logits += w["router_bias"]
        score = logits.sigmoid() if shape.score_fn == wl.SCORE_SIGMOID else logits.softmax(dim=1)
        gate, idx = score.topk(shape.top_k, dim=1)
        if shape.renormalize:
            gate = gate / gate.sum(dim=1, keepdim=True)
        has_shared = shape.shared_inter > 0
        state["idx"] = idx.to(torch.int32).contiguous()
        state["gate"] = gate.contiguous()
        state["shared_scale"] = None
        if has_shared and shape.shared_gate:
            state["shared_scale"] = torch.sigmoid(x.float() @ w["w_shared_gate"].float())
        state["grouping"] = api.alloc_grouping(cfg, T)
        state["y"] = torch.empty((T * shape.top_k, shape.hidden), dtype=torch.bfloat16, device="cuda")
        state["shared_y"] = torch.empty_like(x) if has_shared else None
    return state


def run(state):
    s = state
    if s["entry"] == "layer":
        api.moe_verify_layer(s["cfg"], s["cw"], s["x"], s["B"], s["gamma"], s["out"], s["ws"])
        return s["out"]
    g = s["grouping"]
    api.moe_permute(s["cfg"], s["idx"], g)
    api.moe_grouped_swiglu(s["cfg"], s["cw"], s["x"], g, s["y"], s["shared_y"], s["ws"])
    api.moe_combine(s["cfg"], s["y"], g.inv_perm, s["gate"], s["shared_y"], s["shared_scale"], s["out"])
    return {"out": s["out"], "y": s["y"], "shared_y": s["shared_y"], "counts": g.counts,
            "offsets": g.offsets, "perm": g.perm, "inv_perm": g.inv_perm, "active": g.active,
            "n_active": g.n_active}


def _activated(case, shape):
    """Activated experts of a batch: Gaussian logits, the case's bias, top-k, counted."""
    T = case["B"] * (case["gamma"] + 1)
    E, k = shape.n_experts, shape.top_k
    z = np.random.RandomState(20250519).standard_normal((T, E)) * (0.02 * math.sqrt(shape.hidden))
    if case["zipf"]:
        z += wl.zipf_router_bias(E, shape.hidden, case["zipf"], 0).numpy()
    return len(np.unique(np.argpartition(-z, k - 1, axis=1)[:, :k]))


def work(case):
    shape = _shape(case)
    T = case["B"] * (case["gamma"] + 1)
    H, E, k, I, Is = shape.hidden, shape.n_experts, shape.top_k, shape.inter, shape.shared_inter
    weights = 6 * H * (_activated(case, shape) * I + Is)
    flops = 6 * T * H * (k * I + Is)
    if case["entry"] == "layer":
        # + the router matrix; the token rows in, the layer's output rows out
        return {"bytes": weights + 4 * E * H + 4 * T * H, "flops": flops + 2 * T * H * E}
    # + the indices and gate weights in; expert outputs, tables and the layer's output out
    y = 2 * T * H * (k + (1 if Is else 0))
    return {"bytes": weights + 4 * T * H + y + 4 * T * k * 4, "flops": flops}


def tolerance(case):
    # out against the same layer in fp64 on the same routing: 2-norm of the difference over 2-norm
    # of the result 2.3e-3 to 2.9e-3, no single value off by more than 2.1e-2 (three bf16
    # roundings: the SwiGLU intermediate, the expert outputs, the sum); four times that.  Inside
    # the whole layer a token whose k-th and (k+1)-th logit agree to fp32 rounding may take either
    # expert, which moves single rows by a good part of their size: "max" leaves room for those.
    return {"rel": 1.2e-2, "max": 0.9 if case["entry"] == "layer" else 0.1}
