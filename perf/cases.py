"""The work that users have this library do, as cases that can be timed and compared.

A case is one decode step of one tensor-parallel shard: a single layer
(preserve_decode_step), a linked chain of layers (preserve_decode_chain: the
layers of a model, one token) or a layer with host activation buffers
(preserve_decode_step_host).  Values follow inputs.py: weights ~ N(0, 0.02^2),
gains 1 + N(0, 0.1^2), partial sums, residual and cached K/V ~ N(0, 1).

The layers, their caches, the buffers and the marshalled step descriptions are
kept by a serving program from token to token and are made in prepare();
run() is one call, on the program's own stream.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2501_08192_b200 import binding as P

HEAD = 128
EPS, THETA = 1e-5, 500000.0
_streams = []


def _stream():
    """The program's stream: one for all of its calls."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def _case(name, entry, layers, hidden, q_heads, kv_heads, ffn, tp, max_batch, batch, ctx_min, ctx,
          int8_weights=False, int8_kv=False):
    """ctx_min..ctx: cached tokens per sequence (ragged where they differ); ctx is also the capacity."""
    c = dict(entry=entry, layers=layers, hidden=hidden, q_heads=q_heads, kv_heads=kv_heads, ffn=ffn, tp=tp,
             max_batch=max_batch, batch=batch, ctx_min=ctx_min, ctx=ctx, int8_weights=int8_weights, int8_kv=int8_kv)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one layer, one sequence; kernel launches and hand-overs are most of it
        _case("tiny_tp2_b1", "step", 1, 1024, 4, 4, 1408, 2, 1, 1, 512, 512),
        # a small model's shard on a sparse server: odd sizes throughout, short ragged contexts
        _case("odd_tp3_b3_ragged", "chain", 4, 2688, 6, 2, 1824, 3, 4, 3, 1, 777),
        # Llama-3-8B-shaped shard, the latency-bound serving batch (batch below the tensor-core path)
        _case("8b_tp8_b8", "chain", 8, 4096, 4, 1, 1792, 8, 8, 8, 4096, 4096),
        # the same at the paper's precisions, a partly filled batch of unequal sequences
        _case("8b_tp8_b5_int8", "chain", 8, 4096, 4, 1, 1792, 8, 8, 5, 500, 4000, True, True),
        # the same layer for a program that keeps its activations in (pinned) host memory
        _case("8b_tp8_b8_host", "host", 1, 4096, 4, 1, 1792, 8, 8, 8, 4096, 4096),
        # Llama-3-70B-shaped shard, weight-dominated layers larger than L2
        _case("70b_tp8_b16", "chain", 4, 8192, 8, 1, 3584, 8, 16, 16, 8192, 8192),
        # a server sized for 128 sequences that holds 20 at the moment (continuous batching)
        _case("70b_tp8_b20_of_128", "chain", 4, 8192, 8, 1, 3584, 8, 128, 20, 200, 2000),
        # the same server full, with short conversations: the largest batch
        _case("70b_tp8_b128", "chain", 4, 8192, 8, 1, 3584, 8, 128, 128, 64, 1000),
        # Llama-3-70B-shaped shard at batch 64, ragged contexts
        _case("70b_tp4_b64_ragged", "chain", 2, 8192, 16, 2, 7168, 4, 64, 64, 512, 4096),
        # the same at the paper's precisions
        _case("70b_tp4_b64_int8", "chain", 2, 8192, 16, 2, 7168, 4, 64, 64, 512, 4096, True, True),
        # long contexts: the KV-cache is nearly all of the bytes
        _case("8b_tp8_b32_long", "step", 1, 4096, 4, 1, 1792, 8, 32, 32, 32768, 32768),
        _case("8b_tp8_b32_long_int8", "step", 1, 4096, 4, 1, 1792, 8, 32, 32, 32768, 32768, True, True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MOST_BYTES = 1.1e9


def draw(rng):
    while True:
        entry = rng.choice(["step", "chain", "chain", "host"])
        layers = rng.randint(2, 4) if entry == "chain" else 1
        int8_weights, int8_kv = rng.random() < 0.25, rng.random() < 0.25
        max_batch = _log(rng, 1, 128)
        batch = max_batch if rng.random() < 0.5 else rng.randint(1, max_batch)
        hidden = 128 * max(8, min(64, round(_log(rng, 1024, 8192) / 128)))
        kv_heads = rng.choice([1, 1, 2, 4])
        q_heads = kv_heads * rng.choice([1, 4, 5, 6, 7, 8] + ([] if int8_kv else [12, 16]))
        unit = 128 if max_batch >= 16 else 64 if int8_weights else 32
        ffn = unit * max(1024 // unit, min(7168 // unit, round(_log(rng, 1024, 7168) / unit)))
        ctx = _log(rng, 64, 32768)
        ctx_min = ctx if rng.random() < 0.4 else max(1, ctx // 8)
        c = _case(None, entry, layers, hidden, q_heads, kv_heads, ffn, rng.randint(1, 8), max_batch, batch, ctx_min,
                  ctx, int8_weights, int8_kv)
        if work(c)["bytes"] <= MOST_BYTES and layers * 2 * kv_heads * max_batch * ctx * HEAD * 2 <= 4e9:
            return c


# ------------------------------------------------------------------ inputs

def _contexts(case, seed):
    r = np.random.Generator(np.random.PCG64([seed, 77]))
    if case["ctx_min"] == case["ctx"]:
        return np.full(case["batch"], case["ctx"], np.int32)
    return r.integers(case["ctx_min"], case["ctx"] + 1, size=case["batch"]).astype(np.int32)


def _config(case):
    flags = (P.FLAG_INT8_WEIGHTS if case["int8_weights"] else 0) | (P.FLAG_INT8_KV if case["int8_kv"] else 0)
    return P.LayerConfig(case["hidden"], case["q_heads"], case["kv_heads"], HEAD, case["ffn"], case["tp"],
                         case["max_batch"], case["ctx"], EPS, THETA, flags)


def _layer_inputs(case, seed, layer):
    """Everything layer `layer` reads, on the GPU, in a fixed order of draws."""
    g = torch.Generator("cuda").manual_seed(seed * 1009 + layer)

    def normal(*shape, std=1.0, mean=0.0):
        return (torch.randn(*shape, generator=g, device="cuda") * std + mean).to(torch.bfloat16)

    H, F, B, nq, nkv = case["hidden"], case["ffn"], case["batch"], case["q_heads"] * HEAD, case["kv_heads"] * HEAD
    t = {"g_attn": normal(H, std=0.1, mean=1.0), "g_mlp": normal(H, std=0.1, mean=1.0)}
    for name, shape in (("w_q", (H, nq)), ("w_k", (H, nkv)), ("w_v", (H, nkv)), ("w_o", (nq, H)), ("w_gate", (H, F)),
                        ("w_up", (H, F)), ("w_down", (F, H))):
        t[name] = normal(*shape, std=0.02)
    t["residual"] = normal(B, H)
    t["partials"] = [normal(B, H) for _ in range(case["tp"])]
    t["peers"] = [normal(B, H) for _ in range(case["tp"] - 1)]
    cache = (case["max_batch"], case["kv_heads"], case["ctx"] + 1, HEAD)
    if not case["int8_kv"]:
        for name in ("k", "v"):
            t[name] = torch.empty(cache, dtype=torch.bfloat16, device="cuda")
            for b in range(case["max_batch"]):
                t[name][b] = normal(*cache[1:])
        return t
    off, scap, total = P.preserve_kv8_layout(_config(case))
    for name in ("k", "v"):
        buf = torch.zeros(total, dtype=torch.uint8, device="cuda")
        n = cache[0] * cache[1] * cache[2] * HEAD
        codes = buf[:n].view(torch.int8).view(cache)
        for b in range(case["max_batch"]):
            codes[b] = (torch.randn(*cache[1:], generator=g, device="cuda") * 42).round().clamp(-127, 127).to(torch.int8)
        scales = buf[off:off + cache[0] * cache[1] * scap * 4].view(torch.float32).view(cache[0], cache[1], scap)
        scales.copy_(0.02 + 0.01 * torch.randn(scales.shape, generator=g, device="cuda").abs())
        t[name], t[name + "_codes"], t[name + "_scales"] = buf, codes, scales
    return t


WEIGHTS = ("w_q", "w_k", "w_v", "w_o", "w_gate", "w_up", "w_down", "g_attn", "g_mlp")


def prepare(case, seed):
    cfg, ctx = _config(case), _contexts(case, seed)
    B, H = case["batch"], case["hidden"]
    state = {"entry": case["entry"], "stream": _stream(), "layers": [], "ios": [], "outputs": []}
    ctx_dev = torch.from_numpy(ctx).cuda()
    before = None
    for i in range(case["layers"]):
        t = _layer_inputs(case, seed, i)
        layer = P.Layer(cfg, {n: t.pop(n) for n in WEIGHTS})
        if case["entry"] == "host":
            parts, peers = [x.cpu().pin_memory() for x in t["partials"]], [x.cpu().pin_memory() for x in t["peers"]]
            out = [torch.empty((B, H), dtype=torch.bfloat16).pin_memory() for _ in range(2)]
            io = P.make_host_io(cfg, B, ctx, parts, peers, t["residual"].cpu().pin_memory(), t["k"], t["v"], *out)
        else:
            out = [torch.empty((B, H), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
            residual, partials = t["residual"], t["partials"]
            if before is not None:          # linked: the previous layer's outputs are this layer's inputs
                residual, partials = before[0], [before[1]] + partials[1:]
            io = layer.make_io(B, ctx_dev, ctx, partials, t["peers"], residual, t["k"], t["v"], *out)
        before = out
        state["layers"].append(layer)
        state["ios"].append(io)
        state["outputs"].append({"residual": out[0], "mlp_partial": out[1], "k_cache": t["k"], "v_cache": t["v"]})
    torch.cuda.current_stream().synchronize()
    return state


def run(state):
    if state["entry"] == "step":
        state["layers"][0].decode_step(state["ios"][0], state["stream"])
    elif state["entry"] == "host":
        state["layers"][0].decode_step_host(state["ios"][0], state["stream"])
    else:
        P.preserve_decode_chain(state["layers"], state["ios"], True, state["stream"])
    return state["outputs"]


# ------------------------------------------------------------------ what it costs, and the answer

def work(case):
    """Weights, cached K/V and activations each once (gains, the step's inputs, outputs and the appended entry)."""
    H, F, B, tp = case["hidden"], case["ffn"], case["batch"], case["tp"]
    nq, nkv = case["q_heads"] * HEAD, case["kv_heads"] * HEAD
    weights = H * (nq + 2 * nkv) + nq * H + 3 * H * F
    tokens = B * (case["ctx_min"] + case["ctx"]) / 2          # expected; exact for equal lengths
    per_token = 2 * case["kv_heads"] * (HEAD + 4 if case["int8_kv"] else 2 * HEAD)
    activations = 2 * B * H * (tp + 1 + tp - 1 + 2)           # partial sums, peers, residual; the two outputs
    layer = weights * (1 if case["int8_weights"] else 2) + tokens * per_token + B * per_token + activations + 4 * H
    return {"bytes": case["layers"] * layer,
            "flops": case["layers"] * (2 * B * weights + 4 * (tokens + B) * case["q_heads"] * HEAD)}


def tolerance(case):
    if case["int8_kv"]:
        # one code of an appended vector may fall to the other side of a rounding boundary
        return {"rel": 1e-2, "max": 0.2, "differ": 1e-3}
    return {"rel": 1e-2, "max": 0.1, "differ": 0.0}


def _quantised(w):
    """Symmetric int8 per output feature, decided in fp32; as float64."""
    w = w.float()
    scale = w.abs().amax(0) / 127.0
    code = torch.where(scale > 0, torch.round(w / scale), torch.zeros_like(w))
    return code.double() * scale.double()


def _norm(h, gain):
    return h * torch.rsqrt((h * h).mean(-1, keepdim=True) + EPS) * gain.double()


def _rotated(u, ctx):
    freq = THETA ** (-2.0 * torch.arange(HEAD // 2, dtype=torch.float64, device="cuda") / HEAD)
    angle = ctx.double()[:, None, None] * freq
    a, b = u[..., :HEAD // 2], u[..., HEAD // 2:]
    return torch.cat([a * angle.cos() - b * angle.sin(), b * angle.cos() + a * angle.sin()], -1)


def exact(case, seed):
    B, nq, nkv = case["batch"], case["q_heads"], case["kv_heads"]
    ctx = torch.from_numpy(_contexts(case, seed)).cuda()
    outputs, before = [], None
    for i in range(case["layers"]):
        t = _layer_inputs(case, seed, i)
        w = {n: _quantised(t[n]) if case["int8_weights"] else t[n].double() for n in WEIGHTS[:7]}
        parts, residual = [p.double() for p in t["partials"]], t["residual"].double()
        if before is not None:
            residual, parts[0] = before
        h = residual + sum(parts)
        x = _norm(h, t["g_attn"])
        q = _rotated((x @ w["w_q"]).view(B, nq, HEAD), ctx)
        new = {"k": _rotated((x @ w["w_k"]).view(B, nkv, HEAD), ctx), "v": (x @ w["w_v"]).view(B, nkv, HEAD)}
        o = torch.empty(B, nq, HEAD, dtype=torch.float64, device="cuda")
        for b in range(B):
            n, kv = int(ctx[b]), {}
            for name in ("k", "v"):
                u = new[name][b].float()
                if case["int8_kv"]:          # the new entry takes part as the cache stores it
                    scale = u.abs().amax(-1, keepdim=True) / 127.0
                    entry = (torch.round(u / scale).double() * scale.double())[:, None]
                    past = t[name + "_codes"][b, :, :n].double() * t[name + "_scales"][b, :, :n, None].double()
                else:
                    entry, past = u.to(torch.bfloat16).double()[:, None], t[name][b, :, :n].double()
                kv[name] = torch.cat([past, entry], 1)
            s = torch.softmax(q[b].view(nkv, nq // nkv, HEAD) @ kv["k"].transpose(1, 2) / math.sqrt(HEAD), -1)
            o[b] = (s @ kv["v"]).reshape(nq, HEAD)
        h2 = h + o.view(B, -1) @ w["w_o"] + sum(p.double() for p in t["peers"])
        x2 = _norm(h2, t["g_mlp"])
        mlp = (torch.nn.functional.silu(x2 @ w["w_gate"]) * (x2 @ w["w_up"])) @ w["w_down"]
        caches = {"k": None, "v": None}      # int8: whole numbers
        if not case["int8_kv"]:
            for name in caches:
                caches[name] = t[name].double()
                caches[name][torch.arange(B, device="cuda"), :, ctx.long()] = new[name]
        outputs.append({"residual": h2, "mlp_partial": mlp, "k_cache": caches["k"], "v_cache": caches["v"]})
        before = (h2, mlp)
    return outputs
