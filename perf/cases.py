"""The work a serving program has the library do, as cases to time.

A program drives the library in three ways, and each is a task here:

  decode    one generated token per sequence on caches that have reached their budgets: one
            sq_decode_step per layer (a model computes a layer's query from the layer below), or,
            with per_layer False, one call for the whole stack;
  generate  a batch from its prompt on: importance of every layer, budget allocation, the prompt's
            K/V into every layer's cache, then `steps` generated tokens;
  evict     caches filled under set budgets, then tightened to half by one sq_evict over all layers
            (memory pressure from new requests), then one generated token.

Shapes are those of the repository's workloads (synth.py) and of its tests.
"""
from __future__ import annotations

import math

import torch

from paper_2404_04793_b200 import binding, engine, synth

DEV = "cuda:0"
POLICIES = {"sliding_window": synth.SLIDING_WINDOW, "streaming_llm": synth.STREAMING_LLM, "h2o": synth.H2O}
DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}
N_INPUT_SETS = 4    # decode: tokens' q / k / v kept ready, taken in turn
N_SINK = 4

# layers, query heads, KV heads, head_dim, hidden
SHAPES = {
    "tiny": (4, 2, 2, 64, 128),
    "llama2_7b": (32, 32, 32, 128, 4096),
    "mistral_7b": (32, 32, 8, 128, 4096),
    "llama2_70b": (80, 64, 8, 128, 8192),
    "falcon_7b": (32, 71, 1, 64, 4544),
    "grouped_small": (12, 16, 4, 128, 2048),     # a small grouped-query model
    "multi_query": (16, 20, 1, 64, 1280),        # a small multi-query model
}


def _case(name, task, shape, batch, prompt, policy, budget_pct, p, dtype="bf16", steps=1, per_layer=True,
          per_sequence=False, fused_importance=False):
    return dict(name=name, task=task, shape=shape, batch=batch, prompt=prompt, policy=policy, budget_pct=budget_pct, p=p,
                dtype=dtype, steps=steps, per_layer=per_layer, per_sequence=per_sequence, fused_importance=fused_importance)


def listed():
    return [
        # the smallest whole generation: a toy fp32 model as used to try the method out
        _case("tiny_generate_fp32", "generate", "tiny", 1, 256, "h2o", 40.0, 0.3, dtype="fp32", steps=16, per_layer=False),
        # one interactive user: latency of a token
        _case("mistral_b1_decode_h2o", "decode", "mistral_7b", 1, 3001, "h2o", 20.0, 0.35),
        # small-batch serving of a model with one query head per KV head
        _case("llama7b_b8_decode_sw", "decode", "llama2_7b", 8, 2048, "sliding_window", 20.0, 0.3),
        # grouped-query serving with heavy-hitter scores
        _case("mistral_b16_decode_h2o", "decode", "mistral_7b", 16, 4096, "h2o", 20.0, 0.35),
        # a deep grouped-query model at a throughput batch
        _case("llama70b_b32_decode_streaming", "decode", "llama2_70b", 32, 4096, "streaming_llm", 30.0, 0.3),
        # the whole stack in one call, every sequence with its own budgets, ragged sizes
        _case("mistral_b37_decode_stack", "decode", "mistral_7b", 37, 1111, "sliding_window", 25.0, 0.35, per_layer=False,
              per_sequence=True),
        # the largest decode step: long prompts, large batch, 71 query heads on one KV head
        _case("falcon_b224_decode_sw", "decode", "falcon_7b", 224, 16384, "sliding_window", 50.0, 0.3),
        # the same model at an ordinary batch, with heavy-hitter scores, ragged sizes
        _case("falcon_b33_decode_h2o", "decode", "falcon_7b", 33, 8191, "h2o", 50.0, 0.3),
        # time to the first token, policies that need no scores
        _case("llama7b_b8_first_token_sw", "generate", "llama2_7b", 8, 2048, "sliding_window", 20.0, 0.3),
        # time to the first token with heavy-hitter scores of the prompt; the importance is taken
        # where the residual stream is summed
        _case("mistral_b4_first_token_h2o", "generate", "mistral_7b", 4, 4096, "h2o", 20.0, 0.35, fused_importance=True),
        # the same for 71 query heads on one KV head, a ragged prompt
        _case("falcon_b2_first_token_h2o", "generate", "falcon_7b", 2, 5003, "h2o", 30.0, 0.3),
        # memory pressure: caches tightened in place
        _case("mistral_b16_evict_h2o", "evict", "mistral_7b", 16, 4096, "h2o", 20.0, 0.35),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        task = rng.choice(["decode", "decode", "decode", "generate", "generate", "evict"])
        shape = rng.choice(list(SHAPES))
        policy = rng.choice(list(POLICIES))
        c = _case("", task, shape, _log_int(rng, 1, 224), _log_int(rng, 128, 16384), policy, float(rng.choice([10, 20, 30, 40, 50])),
                  rng.choice([0.2, 0.3, 0.35, 0.5]), dtype="fp32" if rng.random() < 0.15 else "bf16",
                  steps=_log_int(rng, 1, 16) if task == "generate" else 1, per_layer=rng.random() < 0.8,
                  per_sequence=rng.random() < 0.15, fused_importance=rng.random() < 0.5)
        del c["name"]
        w = _workload(c, 0)
        if int(w.b_init * w.p) // (2 if task == "evict" else 1) <= N_SINK + 1:
            continue                              # StreamingLLM needs room beyond its sinks
        if c["per_sequence"] and task == "generate" and c["batch"] * w.n_layer > 2048:
            continue
        cost = work(c)
        fp32 = c["dtype"] == "fp32"
        scored = task == "generate" and policy == "h2o"
        if cost["bytes"] > 14e9 or cost["flops"] > (3e10 if scored and fp32 else 7e12) or _state_bytes(c) > 20e9:
            continue
        return c


# ---------------------------------------------------------------------------------------------

def _workload(case, seed):
    L, hq, hkv, d, hidden = SHAPES[case["shape"]]
    policy = POLICIES[case["policy"]]
    heavy = "none" if policy != synth.H2O else ("uniform4" if case["shape"] == "tiny" else "zipf")
    # the workload's id enters every draw of synth.py: the seed of the case's inputs
    return synth.Workload(case["task"], seed, L, hq, hkv, d, hidden, case["batch"], case["prompt"], case["steps"],
                          DTYPES[case["dtype"]], policy, case["budget_pct"], case["p"], n_sink=N_SINK, heavy_mode=heavy)


def _state_bytes(case):
    w = _workload(case, 0)
    e = 4 if w.dtype == torch.float32 else 2
    n = w.n_layer * w.b_init * w.batch * w.n_kv_head * 2 * w.head_dim
    if case["task"] == "generate":
        n += w.n_layer * w.batch * w.prompt * (3 * w.hidden + (2 * w.n_kv_head + w.n_q_head) * w.head_dim)
    elif case["task"] == "evict":
        n += 4 * w.batch * w.prompt * 2 * w.n_kv_head * w.head_dim
    return n * e


def _budgets(w):
    """Per-layer budgets of the workload, by the library's own allocator on a slice of its hidden states."""
    small = w.replace(batch=1, prompt=256, steps=1, budget_pct=0.0, budget_tokens=w.b_init)
    ctx = engine.context_for(small, DEV)
    ctx.begin_sequence_batch(1, 256)
    for l in range(w.n_layer):
        ctx.layer_importance(l, *synth.hidden_pair(small, l, DEV))
    ctx.allocate_budgets(w.b_init, w.p)
    return ctx.get_budgets()[0]


def _context(w, case):
    # a serving program sets no small limit on the tokens of a conversation
    ctx = engine.context_for(w.replace(steps=1 << 24), DEV, per_sequence_budgets=int(case["per_sequence"]))
    ctx.pool.zero_()
    return ctx


def _spread(w, case, budgets):
    """One vector for the batch, or, with per-sequence budgets, one per sequence (rotations of it)."""
    if not case["per_sequence"]:
        return budgets
    L = w.n_layer
    return [[budgets[(i + s) % L] for i in range(L)] for s in range(w.batch)]


def _decode_inputs(w, n_sets):
    sets = []
    for t in range(n_sets):
        q, k, v = synth.decode_qkv(w, t, DEV)
        sets.append((q, k, v, list(q), list(k), list(v)))    # the whole stack, and layer by layer
    return sets


def prepare(case, seed):
    w = _workload(case, seed)
    s = dict(case=case, w=w, turn=0)
    ctx = s["ctx"] = _context(w, case)
    n_out = case["steps"]
    s["decode"] = _decode_inputs(w, N_INPUT_SETS if case["task"] == "decode" else n_out)
    out = torch.zeros(n_out, w.n_layer, w.batch, w.n_q_head, w.head_dim, dtype=w.dtype, device=DEV)
    s["out"], s["out_layers"] = out, [list(o) for o in out]
    h2o = w.policy == synth.H2O
    if case["task"] == "generate":
        s["hidden"], s["prompt"] = [], []
        for l in range(w.n_layer):
            a, b = synth.hidden_pair(w, l, DEV)
            if case["fused_importance"]:
                s["hidden"].append((a, b.sub_(a), torch.empty_like(a)))     # residual, attention output, their sum
            else:
                s["hidden"].append((a, b))
            s["prompt"].append(synth.prompt_qkv(w, l, DEV, need_q=h2o))
    else:
        budgets = _spread(w, case, _budgets(w))
        fill = []
        ctx.begin_sequence_batch(w.batch, w.prompt)
        ctx.set_budgets(budgets)
        for l in range(w.n_layer):
            # eviction refills its caches in every pass: from four layers' prompts in turn
            if case["task"] == "decode" or l < 4:
                _, k, v = synth.prompt_qkv(w, l, DEV, need_q=False)
                acc = synth.prompt_scores_standin(w, l, DEV) if h2o else None
            if case["task"] == "decode":
                ctx.prefill_compress(l, k, v, None, acc)
            elif l < 4:
                fill.append((k, v, acc))
        if case["task"] == "evict":
            s["fill"], s["budgets"] = fill, budgets
            s["tighter"] = [[b // 2 for b in r] for r in budgets] if case["per_sequence"] else [b // 2 for b in budgets]
    s["cache"] = _cache_views(s)
    return s


def _cache_views(s):
    """What a pass leaves in the caches.  Sliding Window and StreamingLLM keep the same tokens
    whatever the rounding, so the pool is compared as it is.  H2O on caches filled from given scores:
    every layer's scores, of its live slots (which tokens a unit holds shows in them).  H2O from the
    prompt on: two correct programs may order near-equal scores differently, which moves a unit's
    later slots by one, so there the generated tokens' attention outputs stand alone."""
    w, case, ctx = s["w"], s["case"], s["ctx"]
    if w.policy != synth.H2O:
        return [ctx.pool_view.view(torch.int32)]
    if case["task"] == "generate" or w.n_layer * (w.batch if case["per_sequence"] else 1) > 60:
        return []
    rows = []
    for e in ctx.export_layout():
        n = e.n_unit * e.cap
        acc = ctx.pool_view[e.acc_off:e.acc_off + 4 * n].view(torch.float32).view(e.n_unit, e.cap)
        rows.append(acc[:, :e.budget // (2 if case["task"] == "evict" else 1)])
    return rows


def _token(s, inputs, slot):
    ctx, w = s["ctx"], s["w"]
    q, k, v, ql, kl, vl = inputs
    if s["case"]["per_layer"]:
        out = s["out_layers"][slot]
        for l in range(w.n_layer):
            ctx.decode_step(l, l + 1, ql[l], kl[l], vl[l], out[l])
    else:
        ctx.decode_step(0, w.n_layer, q, k, v, s["out"][slot])


def run(s):
    case, w, ctx = s["case"], s["w"], s["ctx"]
    task = case["task"]
    if task == "decode":
        _token(s, s["decode"][s["turn"] % N_INPUT_SETS], 0)
        s["turn"] += 1
    elif task == "generate":
        ctx.begin_sequence_batch(w.batch, w.prompt)
        if case["fused_importance"]:
            for l, (a, b, c) in enumerate(s["hidden"]):
                ctx.layer_importance_fused(l, a, b, c)
        else:
            for l, (a, b) in enumerate(s["hidden"]):
                ctx.layer_importance(l, a, b)
        ctx.allocate_budgets(w.b_init, w.p)
        for l, (q, k, v) in enumerate(s["prompt"]):
            ctx.prefill_compress(l, k, v, q)
        for t in range(w.steps):
            _token(s, s["decode"][t], t)
    else:
        ctx.begin_sequence_batch(w.batch, w.prompt)
        ctx.set_budgets(s["budgets"])
        for l in range(w.n_layer):
            k, v, acc = s["fill"][l % len(s["fill"])]
            ctx.prefill_compress(l, k, v, None, acc)
        ctx.evict(0, w.n_layer, s["tighter"])
        _token(s, s["decode"][0], 0)
    return {"out": s["out"], "cache": s["cache"]}


def work(case):
    """Bytes and operations a pass cannot do without.  The budgets of a stack sum to
    n_layer * b_init; a row is the K and V of one token and KV head."""
    w = _workload(case, 0)
    e = 4 if w.dtype == torch.float32 else 2
    h2o = w.policy == synth.H2O
    L, B, P, G = w.n_layer, w.batch, w.prompt, w.batch * w.n_kv_head
    row = 2 * w.head_dim * e
    side = 4 + (4 if h2o else 0)                  # a kept token's position, and its score
    kept = L * w.b_init                           # tokens per unit, all layers
    io = L * w.head_dim * e * B * 2 * (w.n_q_head + 2 * w.n_kv_head)    # q, k_new, v_new in; out, the appended row out
    share = 0.5 if case["task"] == "evict" else 1.0
    step = G * kept * share * (row + (12 if h2o else 0)) + io           # scores: read, written; positions read
    bytes_, flops = w.steps * step, w.steps * 4.0 * B * w.n_q_head * w.head_dim * kept * share
    if case["task"] == "generate":
        bytes_ += L * B * P * w.hidden * e * (3 if case["fused_importance"] else 2)
        flops += L * B * P * w.hidden * 6.0
        bytes_ += G * kept * (row * 2 + side)     # kept rows read and stored
        if h2o:                                   # causal scores, once; the rest of K, and Q
            bytes_ += L * B * P * w.head_dim * e * (w.n_q_head + w.n_kv_head) - G * kept * row / 2
            flops += 1.0 * L * B * w.n_q_head * P * P * w.head_dim
    elif case["task"] == "evict":
        bytes_ += G * kept * (row * 2 + side)     # the fill
        if h2o:
            bytes_ += L * G * P * 4.0
        bytes_ += G * kept * 0.5 * (row * 2 + 2 * side)   # the rows that stay, read and stored
    return {"bytes": float(bytes_), "flops": float(flops)}


def tolerance(case):
    """Four times what was measured.  One call for the stack against one call per layer (other
    pieces, so sums in another order): bf16 1.5e-3 in the 2-norm and 1.4e-2 at the largest, against
    the outputs' spread; fp32 1.7e-7 and 1.7e-6.  H2O also keeps another one of two nearly equal
    tokens in a unit or two when its scores move by 1e-6, and that unit's outputs then differ by the
    token's share: 4.6e-4 over all outputs and 3.2e-2 at the largest (prompts of 4096 tokens), more for
    a smaller cache."""
    h2o, fp32 = case["policy"] == "h2o", case["dtype"] == "fp32"
    return {"rel": (2e-3 if h2o else 1e-5) if fp32 else 6e-3, "max": 0.2 if h2o else 1e-4 if fp32 else 0.06, "differ": 0.0}
