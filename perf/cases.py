"""What the MoE layer is used for, as cases that can be timed.

A case is one pass of a serving program through the layer's public calls: a decode step of a few tokens, a batch that
mixes decode and prompt chunks, a whole prompt, a step of a layer stack with a switch of its significant channels, a
call on host buffers.  The layer shapes are this repository's configurations (``workloads.CONFIGS``): ``decode`` and
``prefill`` are Mixtral-8x7B-shaped layers, ``finegrained`` is shaped like DeepSeek-MoE-16B, ``tiny`` is small.

Keys of a case: ``config``; ``tokens``; ``entry`` (how the layer is called: ``logits``, ``router`` with the gate's GEMM
in front, ``host`` buffers, ``stack`` of layers behind a switch event, ``adapt`` = forward with statistics and the
selection that follows); ``out`` (``f32`` or ``bf16`` results); ``operand`` (rounding of the hidden activations);
``down_sig`` (significant hidden units per expert on the d_ff side, 0 = none); ``layers`` (of a stack).
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2503_21135_b200 import binding
from paper_2503_21135_b200 import workloads as wl


def _case(name, config, tokens, entry="logits", out="f32", operand="fp16", down_sig=0, layers=1):
    c = {"config": config, "tokens": tokens, "entry": entry, "out": out, "operand": operand, "down_sig": down_sig,
         "layers": layers}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one user's next token: two of eight experts are read, latency counts
        _case("decode_1", "decode", 1, out="bf16"),
        # a small decode batch: nearly every expert is read for one to three rows each
        _case("decode_8", "decode", 8),
        # the full decode batch from host buffers to host buffers: what a caller without device buffers pays
        _case("decode_64_host", "decode", 64, entry="host"),
        # decode batch of many users, odd size: every expert has a few dozen rows
        _case("batch_139", "decode", 139, out="bf16"),
        # decode tokens and a prompt chunk in one batch
        _case("batch_500", "decode", 500, out="bf16"),
        # a prompt of ordinary length with a skewed router; hidden activations rounded to bf16
        _case("prefill_1000", "prefill", 1000, out="bf16", operand="bf16"),
        # the long prompt
        _case("prefill_4096", "prefill", 4096),
        # many small experts, decode batch, with significant hidden units on the d_ff side
        _case("fine_16_down", "finegrained", 16, out="bf16", down_sig=32),
        # many small experts, short prompt, the gate computed by the layer; statistics on, selection behind the forward
        _case("fine_300_adapt", "finegrained", 300, entry="adapt"),
        # many small experts, the long prompt: popular experts have a thousand rows, unpopular ones a handful
        _case("fine_2048", "finegrained", 2048, out="bf16"),
        # a small layer: nothing but latency and launches
        _case("tiny_64", "tiny", 64),
        # a stack of layers at a decode batch of 16, its significant channels swapped before the step
        _case("stack_16_switch", "switch", 16, entry="stack", out="bf16", layers=4),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    """Sizes over the range of each configuration (over their logarithm), every entry and option."""
    config = rng.choice(["decode", "decode", "prefill", "finegrained", "finegrained", "tiny", "switch"])
    if config == "switch":
        return _case(None, "switch", _log_int(rng, 1, 48), entry="stack", out=rng.choice(["f32", "bf16"]),
                     layers=rng.choice([2, 3, 4]))
    lo, hi = {"decode": (1, 700), "prefill": (300, 4000), "finegrained": (1, 2048), "tiny": (1, 1024)}[config]
    tokens = _log_int(rng, lo, hi)
    entries = ["logits", "logits", "router"] + (["host"] if tokens <= 128 else []) + (["adapt"] if tokens >= 8 else [])
    return _case(None, config, tokens, entry=rng.choice(entries), out=rng.choice(["f32", "bf16"]),
                 operand=rng.choice(["fp16", "fp16", "bf16"]), down_sig=rng.choice([0, 0, 0, 32]))


def _layer_weights(cfg, layer, gen, device):
    """N(0, 0.02^2), the outlier input channels of every routed expert x20 in W_gate and W_up, rounded to bf16."""
    n, d, f = cfg.n_total, cfg.d_model, cfg.d_ff
    mats = []
    for shape, outliers in (((f, d), True), ((f, d), True), ((d, f), False)):
        w = torch.empty((n,) + shape, dtype=torch.bfloat16, device=device)
        for e in range(n):
            t = torch.empty(shape, dtype=torch.float32, device=device).normal_(0.0, 0.02, generator=gen)
            if outliers and e < cfg.n_experts:
                cols = torch.from_numpy(wl.outlier_channels(cfg, layer, e).astype(np.int64)).to(device)
                t[:, cols] *= 20.0
            w[e] = t.to(torch.bfloat16)
        mats.append(w)
    return mats


def prepare(case, seed):
    """Packed layers, the step's inputs and (stack) the sets of the next switch events."""
    device = torch.device("cuda", torch.cuda.current_device())
    cfg = wl.CONFIGS[case["config"]]
    T, n_layers = case["tokens"], case["layers"]
    gen = torch.Generator(device=device)
    gen.manual_seed(seed * 7919 + cfg.config_id)
    layers, pools, sets, workspace = [], [], [], None
    for l in range(n_layers):
        wg, wu, wd = _layer_weights(cfg, l, gen, device)
        bits, pool = wl.bits_assignment(cfg, l), wl.cache_pool(cfg, l)
        layer = binding.DynamoLayer.from_config(cfg, max_tokens=max(T, max(cfg.tokens)), workspace=workspace,
                                                device=device)
        layer.pack_experts(wg, wu, wd, bits, pool)
        cur = wl.initial_sig_sets(cfg, pool, l)
        layer.set_channel_switch(cur)
        if case["down_sig"]:
            pool_d = wl.cache_pool_down(cfg, 2 * case["down_sig"], l)
            layer.pack_down_cache(wd, bits, pool_d, case["down_sig"])
            layer.set_channel_switch_down(wl.sig_sets_down(cfg, pool_d, case["down_sig"], l))
        layer.set_operand_dtype(binding.OPERAND_BF16 if case["operand"] == "bf16" else binding.OPERAND_FP16)
        layer.set_stats_collection(case["entry"] == "adapt")
        workspace = layer.workspace
        layers.append(layer)
        pools.append(pool)
        sets.append(cur)
        del wg, wu, wd
    bias = torch.from_numpy(wl.popularity_bias(cfg).astype(np.float32)).to(device)
    xs, logits = [], []
    for l in range(n_layers):
        xs.append(torch.randn((T, cfg.d_model), generator=gen, device=device).to(torch.bfloat16))
        logits.append(torch.randn((T, cfg.n_experts), generator=gen, device=device) + bias)
    state = {"case": case, "cfg": cfg, "layers": layers, "x": xs, "logits": logits,
             "y_dtype": binding.F32 if case["out"] == "f32" else binding.BF16}
    if case["entry"] in ("router", "adapt"):
        w = torch.randn((cfg.n_experts, cfg.d_model), generator=gen, device=device) / cfg.d_model ** 0.5
        state["router"] = (w.to(torch.bfloat16), bias)
    if case["entry"] == "host":
        state["x_host"] = xs[0].cpu().pin_memory()
        state["logits_host"] = logits[0].cpu().pin_memory()
        state["y_host"] = torch.empty((T, cfg.d_model), dtype=torch.float32 if case["out"] == "f32" else torch.bfloat16,
                                      pin_memory=True)
    if case["entry"] == "stack":
        # the event swaps a quarter of every set
        state["event"] = [wl.switch_event(cfg, pools[l], sets[l], l, seed % 4096) for l in range(n_layers)]
    return state


def run(state):
    entry, layers, y_dtype = state["case"]["entry"], state["layers"], state["y_dtype"]
    if entry == "logits":
        return layers[0].forward(state["x"][0], state["logits"][0], y_dtype)
    if entry == "router":
        return layers[0].forward_router(state["x"][0], *state["router"], y_dtype=y_dtype, want_logits=True)
    if entry == "host":
        return layers[0].forward_host(state["x_host"], state["logits_host"], state["y_host"], y_dtype)
    if entry == "adapt":
        y, logits = layers[0].forward_router(state["x"][0], *state["router"], y_dtype=y_dtype, want_logits=True)
        stats = layers[0].channel_stats()
        layers[0].select_significant(state["cfg"].max_sig, reset=True, wait=False)
        return {"y": y, "logits": logits, "stats": stats}
    binding.set_channel_switch_many(layers, state["event"])
    return [layer.forward(x, lg, y_dtype) for layer, x, lg in zip(layers, state["x"], state["logits"])]


def work(case):
    """Packed codes and parameters of the experts that a draw of the router reaches, their significant columns, inputs
    and outputs; multiply-adds of every (token, expert) pair."""
    cfg, T = wl.CONFIGS[case["config"]], case["tokens"]
    d, f, E = cfg.d_model, cfg.d_ff, cfg.n_experts
    nbytes = flops = 0.0
    for l in range(case["layers"]):
        bits = wl.bits_assignment(cfg, l)
        lg = np.random.default_rng(l).standard_normal((T, E)) + wl.popularity_bias(cfg)[None, :]
        rows = np.bincount(np.argsort(-lg, axis=1)[:, : cfg.top_k].ravel(), minlength=E)
        rows = np.concatenate([rows, np.full(cfg.n_shared, T)])
        for e in range(cfg.n_total):
            if rows[e] == 0:
                continue
            switchable = e < E and bits[e] < 8
            nbytes += 3.0 * d * f * bits[e] / 8 + 3.0 * d * f / cfg.group_size * 4
            flops += 6.0 * d * f * rows[e]
            if switchable:
                nbytes += 2.0 * f * cfg.max_sig * 2 + 2.0 * d * case["down_sig"]
                flops += rows[e] * (4.0 * f * cfg.max_sig + 2.0 * d * case["down_sig"])
        nbytes += T * (2.0 * d + 4.0 * E + d * (4.0 if case["out"] == "f32" else 2.0))
        if case["entry"] in ("router", "adapt"):
            nbytes += 2.0 * E * d
            flops += 2.0 * T * E * d
        if case["entry"] == "adapt":
            nbytes += 8.0 * E * cfg.cache_size
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Relative error (2-norm).  Against a float64 evaluation of the same quantized layers the fp16-operand path shows
    2.4e-4 (few tokens: hidden activations rounded to 11 bits) to 3.7e-4 (many: the dequantized weight as well), a bf16
    result or bf16 hidden activations 1.7e-3, both together 2.4e-3; four times that is allowed.  Statistics and scores
    are fp32 sums and far inside."""
    eight_bit = (case["out"] == "bf16") + (case["operand"] == "bf16")
    return {"rel": (1.5e-3, 6.5e-3, 9e-3)[eight_bit]}
