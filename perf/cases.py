"""Performance cases of the depth-sparse forward: the work a user's program has
this library do, through the entry points of paper_2607_21291_gb300.adadsf.

Kinds of case
  layer      one sparse layer in place on hidden states (adadsf_sparse_layer_forward)
  model      the whole sparse forward, or with stats the dense calibration pass
             that also accumulates the Eq. 4 sums (adadsf_sparse_model_forward)
  decode     generated tokens after a prompt that was prefilled once: the cache
             is taken back to the end of the prompt, then `steps` decode steps
             run (several continuations of one prompt; adadsf_decode_step)
  generate   prompt and continuation in one pass (adadsf_prefill, then steps)
  attention  causal attention among packed tokens (adadsf_causal_attention)
  align      one training step of a layer's router: gated and plain layer
             forwards, the Eq. 9 loss with its gradient, the router's gradient
             (what align.router_alignment_step sequences; returns the gradients)
  kl         the Eq. 10 loss over an LM head (adadsf_align_output)

Inputs: hidden states N(0, 1) whose rows spread in norm as a residual stream's
do, weights N(0, 0.02) with the projections that write to the residual stream
scaled by 1 / sqrt(2 layers) (the usual initialisation of these backbones, which
keeps a layer's update small against its input as in a trained model), norm
gains around 1, router output weights wide enough that scores spread over a few
units.
"""
from __future__ import annotations

import math

import torch

from paper_2607_21291_gb300 import adadsf as A
from paper_2607_21291_gb300 import synth as S

SHAPES = {s.name: s for s in (S.PYTHIA_70M, S.PYTHIA_160M, S.PYTHIA_1_4B, S.QWEN25_1_5B, S.QWEN25_7B)}
EXACT_FLOPS = 9e12   # fp64 references above this take over about 20 s


def listed():
    return [
        # the smallest call: one fp32 layer on a short sequence (latency and launches)
        {"name": "layer_f32_small", "kind": "layer", "shape": "pythia-70m", "B": 1, "T": 128, "K": 64, "gate": False},
        # fp32 on a ragged batch: evaluation of a small fp32 checkpoint
        {"name": "layer_f32_batch", "kind": "layer", "shape": "pythia-70m", "B": 4, "T": 511, "K": 383, "gate": False},
        # an ordinary layer of a mid-size model, odd kept count
        {"name": "layer_1_4b", "kind": "layer", "shape": "pythia-1.4b", "B": 8, "T": 2048, "K": 1023, "gate": False},
        # one ragged sequence through a gated layer (prompt processing at batch 1)
        {"name": "layer_1_5b_single", "kind": "layer", "shape": "qwen2.5-1.5b", "B": 1, "T": 777, "K": 389, "gate": True},
        # the largest: a 7B layer on 16 sequences of 4096 tokens
        {"name": "layer_7b", "kind": "layer", "shape": "qwen2.5-7b", "B": 16, "T": 4096, "K": 2048, "gate": False},
        # a whole small model on an ordinary batch
        {"name": "model_160m", "kind": "model", "shape": "pythia-160m", "layers": 12, "B": 4, "T": 512, "keep": 0.5,
         "stats": False},
        # calibration: dense layers with the Eq. 4 statistics
        {"name": "calibrate_1_4b", "kind": "model", "shape": "pythia-1.4b", "layers": 2, "B": 8, "T": 2048, "keep": 1.0,
         "stats": True},
        # token generation of a 7B model at batch 16 (two of its layers), steps in a graph
        {"name": "decode_7b", "kind": "decode", "shape": "qwen2.5-7b", "layers": 2, "B": 16, "T": 1500, "keep": 0.5,
         "steps": 16, "graph": True},
        # one user's prompt and answer on a small model, steps in a graph
        {"name": "generate_160m", "kind": "generate", "shape": "pythia-160m", "layers": 12, "B": 1, "T": 100,
         "keep": 0.75, "steps": 16, "graph": True},
        # attention alone, ragged
        {"name": "attention_7b", "kind": "attention", "shape": "qwen2.5-7b", "B": 4, "K": 1900},
        # a router training step (forward twice, loss, backward)
        {"name": "align_1_4b", "kind": "align", "shape": "pythia-1.4b", "B": 4, "T": 1024, "K": 512},
        # the output loss on a chunk of rows over a full vocabulary
        {"name": "kl_160m", "kind": "kl", "shape": "pythia-160m", "rows": 1000, "classes": 50304},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("layer", "layer", "layer", "layer_f32", "model", "model", "decode", "generate", "attention",
                       "align", "kl"))
    if kind == "layer_f32":
        B, T = rng.randint(1, 4), _log_int(rng, 64, 700)
        return {"kind": "layer", "shape": "pythia-70m", "B": B, "T": T, "K": max(1, int(T * rng.uniform(0.2, 1.0))),
                "gate": rng.random() < 0.3}
    if kind == "layer":
        shape = rng.choice(("pythia-160m", "pythia-1.4b", "qwen2.5-1.5b", "qwen2.5-7b"))
        tokens = _log_int(rng, 128, 32768)
        B = rng.choice([b for b in (1, 2, 3, 4, 7, 8, 16) if tokens // b >= 32])
        T = min(4096, tokens // B)
        K = T if rng.random() < 0.1 else max(1, int(T * rng.uniform(0.2, 0.9)))
        return {"kind": "layer", "shape": shape, "B": B, "T": T, "K": K, "gate": rng.random() < 0.3}
    if kind == "model":
        stats = rng.random() < 0.3
        shape, layers = rng.choice((("pythia-160m", 12), ("pythia-1.4b", 2), ("qwen2.5-1.5b", 2)))
        return {"kind": "model", "shape": shape, "layers": layers, "B": rng.randint(1, 8), "T": _log_int(rng, 48, 1500),
                "keep": 1.0 if stats else rng.uniform(0.25, 0.75), "stats": stats}
    if kind in ("decode", "generate"):
        shape, layers = rng.choice((("pythia-160m", 12), ("pythia-1.4b", 3), ("qwen2.5-1.5b", 3), ("qwen2.5-7b", 2)))
        B = _log_int(rng, 1, 24) if kind == "decode" else _log_int(rng, 1, 6)
        return {"kind": kind, "shape": shape, "layers": layers, "B": B,
                "T": _log_int(rng, 32, 1500 if kind == "decode" else 400), "keep": rng.uniform(0.25, 0.9),
                "steps": rng.randint(4, 12), "graph": rng.random() < 0.7}
    if kind == "attention":
        return {"kind": "attention", "shape": rng.choice(("pythia-160m", "pythia-1.4b", "qwen2.5-1.5b", "qwen2.5-7b")),
                "B": rng.randint(1, 6), "K": _log_int(rng, 32, 3000)}
    if kind == "align":
        T = _log_int(rng, 64, 1024)
        return {"kind": "align", "shape": rng.choice(("pythia-160m", "pythia-1.4b", "qwen2.5-1.5b")),
                "B": rng.randint(1, 4), "T": T, "K": max(1, int(T * rng.uniform(0.25, 0.75)))}
    return {"kind": "kl", "shape": rng.choice(("pythia-160m", "pythia-1.4b")), "rows": _log_int(rng, 32, 1000),
            "classes": 50304}


# ------------------------------------------------------------------ inputs
def _gen(seed, tag):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFFFFFF)


def _normal(g, shape, std, mean=0.0):
    t = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    return t.mul_(std).add_(mean) if mean else t.mul_(std)


def _shape(case):
    return SHAPES[case["shape"]].replace(n_layers=case.get("layers", 1))


def _dtype(s):
    return torch.bfloat16 if s.dtype == "bf16" else torch.float32


def _layer(s, seed, layer):
    """Weights of one layer in the storage type."""
    depth = SHAPES[s.name].n_layers
    out = {}
    for i, (name, shp) in enumerate(sorted(S.layer_weight_shapes(s).items())):
        g = _gen(seed, 100 + 50 * layer + i)
        if name in ("ln1_w", "ln2_w"):
            t = _normal(g, shp, 0.1, 1.0)
        elif name in ("ln1_b", "ln2_b"):
            t = _normal(g, shp, 0.1)
        elif name == "router_w2":
            t = _normal(g, shp, 0.25)
        elif name in ("w_o", "w_down"):
            t = _normal(g, shp, 0.02 / math.sqrt(2.0 * depth))
        else:
            t = _normal(g, shp, 0.02)
        out[name] = t.to(_dtype(s))
    return out


def _extra(s, seed):
    """Embedding and final norm."""
    out = {"embed": _normal(_gen(seed, 1), (s.vocab, s.d), 1.0).to(_dtype(s)),
           "final_w": _normal(_gen(seed, 2), (s.d,), 0.1, 1.0).to(_dtype(s))}
    if s.arch == S.NEOX:
        out["final_b"] = _normal(_gen(seed, 3), (s.d,), 0.1).to(_dtype(s))
    return out


def _hidden(s, seed, B, T):
    rows = torch.exp(_normal(_gen(seed, 5), (B, T, 1), 0.3))
    return (_normal(_gen(seed, 4), (B, T, s.d), 1.0) * rows).to(_dtype(s))


def _ids(s, seed, tag, shape):
    return torch.randint(0, s.vocab, shape, generator=_gen(seed, tag), device="cuda", dtype=torch.int32)


def _plan(case):
    """Kept counts per layer, falling with depth as the allocation's do."""
    L, T, r = case["layers"], case["T"], case["keep"]
    if r >= 1.0:
        return [T] * L
    return [max(1, min(T, int(T * r * (1.12 - 0.24 * l / max(1, L - 1))))) for l in range(L)]


def _head(case, s, seed):
    hd = _normal(_gen(seed, 11), (case["rows"], s.d), 1.0)
    hs = hd + _normal(_gen(seed, 12), (case["rows"], s.d), 0.3)
    return hs.to(_dtype(s)), hd.to(_dtype(s)), _normal(_gen(seed, 13), (case["classes"], s.d), 0.02).to(_dtype(s))


def _dense_target(s, x, seed):
    """The dense layer's output that the alignment compares with."""
    return (x.float() + _normal(_gen(seed, 14), tuple(x.shape), 0.25)).to(x.dtype)


def prepare(case, seed):
    s = _shape(case)
    st = {"case": case}
    kind = case["kind"]
    if kind == "layer":
        B, T, K = case["B"], case["T"], case["K"]
        st["cfg"] = A.make_cfg(s, A.FLAG_GATE_SIGMOID if case["gate"] else 0)
        st["w"] = _layer(s, seed, 0)
        st["x"] = _hidden(s, seed, B, T)
        st["ws"] = A.workspace(A.adadsf_layer_workspace_size(st["cfg"], B, T, K))
        return st
    if kind == "attention":
        B, K = case["B"], case["K"]
        st["cfg"] = A.make_cfg(s)
        st["qkv"] = _normal(_gen(seed, 6), (B * K, s.qkv_dim), 1.0).to(_dtype(s))
        st["out"] = torch.empty(B * K, s.q_dim, device="cuda", dtype=_dtype(s))
        st["ws"] = A.workspace(A.adadsf_attention_workspace_size(st["cfg"], B, K))
        return st
    if kind == "align":
        B, T, K = case["B"], case["T"], case["K"]
        st["cfg"], st["cfg_gate"] = A.make_cfg(s), A.make_cfg(s, A.FLAG_GATE_SIGMOID)
        st["w"] = _layer(s, seed, 0)
        st["x"] = _hidden(s, seed, B, T)
        st["hd"] = _dense_target(s, st["x"], seed)
        st["base"] = torch.arange(B, device="cuda", dtype=torch.int32)[:, None] * T
        st["ws"] = A.workspace(A.adadsf_layer_workspace_size(st["cfg_gate"], B, T, K))
        st["ws_align"] = A.workspace(A.lib().adadsf_align_workspace_size(B * T, 0))
        st["ws_back"] = A.workspace(A.lib().adadsf_router_backward_workspace_size(st["cfg"], B * K))
        return st
    if kind == "kl":
        st["hs"], st["hd"], st["head"] = _head(case, s, seed)
        st["acc"] = torch.zeros(2, device="cuda", dtype=torch.float64)
        st["ws"] = A.workspace(A.lib().adadsf_align_workspace_size(case["rows"], case["classes"]))
        return st
    # whole models
    B, T, K = case["B"], case["T"], _plan(case)
    model = A.DeviceModel(A.make_cfg(s), [_layer(s, seed, l) for l in range(s.n_layers)], _extra(s, seed))
    st.update(model=model, K=K, ids=_ids(s, seed, 7, (B, T)))
    st["hidden"] = torch.empty(B, T, s.d, device="cuda", dtype=_dtype(s))
    st["ws"] = A.workspace(A.adadsf_model_workspace_size(model.cfg, B, T, K, case.get("stats", False)))
    if kind == "model":
        st["acc"] = torch.zeros(2 * s.n_layers, device="cuda", dtype=torch.float64)
        return st
    steps = case["steps"]
    C_max = T + steps + 1
    st["C_max"] = C_max
    st["cache"] = A.kv_cache(model.cfg, B, C_max)
    st["ws_step"] = A.workspace(A.adadsf_decode_workspace_size(model.cfg, B, C_max))
    st["next"] = _ids(s, seed, 8, (steps, B))
    st["out"] = torch.empty(steps, B, s.d, device="cuda", dtype=_dtype(s))
    st["kept"] = torch.zeros(steps, s.n_layers, B, device="cuda", dtype=torch.int32)
    A.adadsf_prefill(model, st["ids"], K, st["hidden"], st["cache"], C_max, ws=st["ws"])
    st["prompt"] = st["cache"].clone()
    if case["graph"]:
        # one decode step captured once and replayed for every token
        st["tok"] = st["next"][0].clone()
        st["h"], st["k"] = torch.empty_like(st["out"][0]), torch.zeros_like(st["kept"][0])
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            A.adadsf_decode_step(model, st["tok"], st["h"], st["cache"], C_max, kept_out=st["k"], ws=st["ws_step"])
        torch.cuda.synchronize()
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"], stream=stream):
            A.adadsf_decode_step(model, st["tok"], st["h"], st["cache"], C_max, kept_out=st["k"], ws=st["ws_step"])
    return st


# ------------------------------------------------------------------ one pass
def _steps(st):
    if not st["case"]["graph"]:
        for i in range(st["case"]["steps"]):
            A.adadsf_decode_step(st["model"], st["next"][i], st["out"][i], st["cache"], st["C_max"],
                                 kept_out=st["kept"][i], ws=st["ws_step"])
        return
    for i in range(st["case"]["steps"]):
        st["tok"].copy_(st["next"][i])
        st["graph"].replay()
        st["out"][i].copy_(st["h"])
        st["kept"][i].copy_(st["k"])


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "layer":
        A.adadsf_sparse_layer_forward(st["cfg"], st["w"], st["x"], case["K"], ws=st["ws"])
        return st["x"]
    if kind == "attention":
        A.adadsf_causal_attention(st["cfg"], st["qkv"], case["B"], case["K"], st["out"], ws=st["ws"])
        return st["out"]
    if kind == "model":
        if case["stats"]:
            st["acc"].zero_()
        A.adadsf_sparse_model_forward(st["model"], st["ids"], st["K"], st["hidden"],
                                      stats_acc=st["acc"] if case["stats"] else None, ws=st["ws"])
        return (st["hidden"], st["acc"]) if case["stats"] else st["hidden"]
    if kind == "decode":
        st["cache"].copy_(st["prompt"])
        _steps(st)
        return st["out"], st["kept"]
    if kind == "generate":
        A.adadsf_prefill(st["model"], st["ids"], st["K"], st["hidden"], st["cache"], st["C_max"], ws=st["ws"])
        _steps(st)
        return st["hidden"], st["out"], st["kept"]
    if kind == "align":
        x, w = st["x"], st["w"]
        B, T, K = case["B"], case["T"], case["K"]
        idx = torch.empty(B, K, dtype=torch.int32, device=x.device)
        y_gate, y_plain = x.clone(), x.clone()
        A.adadsf_sparse_layer_forward(st["cfg_gate"], w, y_gate, K, idx, None, st["ws"])
        A.adadsf_sparse_layer_forward(st["cfg"], w, y_plain, K, idx, None, st["ws"])
        acc = torch.zeros(2, dtype=torch.float64, device=x.device)
        grad_y = torch.empty(B * T, x.shape[-1], dtype=torch.float32, device=x.device)
        A.adadsf_align_hidden(y_gate, st["hd"], acc, grad_y, ws=st["ws_align"])
        rows = (st["base"] + idx).reshape(-1)
        grad = A.adadsf_router_backward(st["cfg_gate"], w, x, y_plain, rows, grad_y, ws=st["ws_back"])
        return {"loss": acc, "grad_y": grad_y, "grad_router": grad, "y": y_gate}
    st["acc"].zero_()
    A.adadsf_align_output(st["hs"], st["hd"], st["head"], st["acc"], ws=st["ws"])
    return st["acc"]


# ------------------------------------------------------------------ work
def _weights_elems(s):
    return sum(math.prod(shp) for shp in S.layer_weight_shapes(s).values())


def _layer_flops(s, B, T, K):
    per_tok = 2.0 * (s.qkv_dim * s.d + s.d * s.q_dim + (3 if s.arch == S.QWEN else 2) * s.d * s.ffn)
    router = 2.0 * B * T * s.router_hidden * s.d if K < T else 0.0
    return B * K * per_tok + 2.0 * B * s.n_heads * s.head_dim * K * (K + 1) + router


def work(case):
    s = _shape(case)
    es = 2 if s.dtype == "bf16" else 4
    kind = case["kind"]
    if kind == "kl":
        r, c = case["rows"], case["classes"]
        return {"bytes": (2.0 * r + c) * s.d * es, "flops": 4.0 * r * c * s.d}
    B, W = case["B"], _weights_elems(s)
    if kind == "attention":
        K = case["K"]
        return {"bytes": float(B * K * (s.qkv_dim + s.q_dim) * es),
                "flops": 2.0 * B * s.n_heads * s.head_dim * K * (K + 1)}
    T = case["T"]
    if kind == "layer":
        K = case["K"]
        return {"bytes": float((W + B * (T + K) * s.d) * es), "flops": _layer_flops(s, B, T, K)}
    if kind == "align":
        K = case["K"]
        return {"bytes": float((W + 4 * B * T * s.d) * es + 4 * B * T * s.d + 4 * s.router_hidden * s.d),
                "flops": 2.0 * _layer_flops(s, B, T, K) + 4.0 * B * K * s.router_hidden * s.d}
    plan = _plan(case)
    nbytes, flops = 0.0, 0.0
    if kind in ("model", "generate"):
        nbytes += s.n_layers * W * es + 2.0 * B * T * s.d * es
        flops += sum(_layer_flops(s, B, T, K) for K in plan)
    if kind in ("decode", "generate"):
        kv = sum(2.0 * B * K * s.kv_dim * es for K in plan)
        nbytes += case["steps"] * (s.n_layers * W * es + kv + 2.0 * B * s.d * es)
        flops += case["steps"] * B * sum(_layer_flops(s, 1, 1, 1) + 4.0 * s.q_dim * K for K in plan)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    f32 = SHAPES[case["shape"]].dtype == "f32"
    return {
        "layer": {"rel": 3e-7} if f32 else {"rel": 5e-3, "max": 0.2},
        "model": {"rel": 2e-2, "max": 0.9},
        "decode": {"rel": 2e-2, "max": 0.9, "differ": 0.01},
        "generate": {"rel": 2e-2, "max": 0.9, "differ": 0.01},
        "attention": {"rel": 8e-3, "max": 0.2},
        "align": {"rel": 2e-2, "max": 0.9},
        "kl": {"rel": 1e-6},
    }[case["kind"]]


# ------------------------------------------------------------------ 64-bit references (plain torch)
def _ln(x, g, b, eps):
    mu = x.mean(-1, keepdim=True)
    var = ((x - mu) ** 2).mean(-1, keepdim=True)
    return (x - mu) / torch.sqrt(var + eps) * g + b


def _rms(x, g, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * g


def _norm(s, x, w, which):
    return _ln(x, w[which + "_w"], w[which + "_b"], s.norm_eps) if s.arch == S.NEOX else _rms(x, w[which + "_w"], s.norm_eps)


def _rope(s, v, pos):
    """v [n, heads, hd] at positions pos [n]."""
    half = s.rotary_dim // 2
    inv = s.rope_theta ** (-(torch.arange(half, device=v.device, dtype=torch.float64) * 2.0) / s.rotary_dim)
    ang = pos.double()[:, None] * inv[None, :]
    c, sn = torch.cos(ang)[:, None, :], torch.sin(ang)[:, None, :]
    out = v.clone()
    a, b = v[..., :half], v[..., half:s.rotary_dim]
    out[..., :half] = a * c - b * sn
    out[..., half:s.rotary_dim] = b * c + a * sn
    return out


def _split(s, qkv):
    n = qkv.shape[0]
    q, k, v = qkv.split([s.q_dim, s.kv_dim, s.kv_dim], dim=1)
    return (q.reshape(n, s.n_heads, s.head_dim), k.reshape(n, s.n_kv_heads, s.head_dim),
            v.reshape(n, s.n_kv_heads, s.head_dim))


def _attend(s, q, k, v, causal):
    """q [n, H, hd], k and v [m, Hkv, hd] -> [n, H hd]; causal: n == m."""
    out = torch.empty_like(q)
    group = s.n_heads // s.n_kv_heads
    mask = torch.ones(q.shape[0], k.shape[0], device=q.device, dtype=torch.bool).triu(1) if causal else None
    for h in range(s.n_heads):
        p = q[:, h] @ k[:, h // group].T / math.sqrt(s.head_dim)
        if causal:
            p = p.masked_fill(mask, -math.inf)
        out[:, h] = torch.softmax(p, -1) @ v[:, h // group]
    return out.reshape(q.shape[0], -1)


def _mlp(s, m, w):
    if s.arch == S.NEOX:
        return torch.nn.functional.gelu(m @ w["w_up"].T + w["b_up"]) @ w["w_down"].T + w["b_down"]
    return (torch.nn.functional.silu(m @ w["w_gate"].T) * (m @ w["w_up"].T)) @ w["w_down"].T


def _delta(s, x, o, w):
    """The layer's update of rows x given their attention outputs o."""
    attn = o @ w["w_o"].T
    if s.arch == S.NEOX:
        return attn + w["b_o"] + _mlp(s, _norm(s, x, w, "ln2"), w)
    h = x + attn
    return attn + _mlp(s, _norm(s, h, w, "ln2"), w)


def _scores(x, w):
    return torch.nn.functional.silu(x @ w["router_w1"].T + w["router_b1"]) @ w["router_w2"] + w["router_b2"]


def _double(w):
    return {k: v.double() for k, v in w.items()}


def _exact_layer(s, w, x, K, gate, sink=None):
    """x [B, T, d] float64, in place; returns (delta rows, idx, scores) for the gradient's reference."""
    B, T, _ = x.shape
    sc = _scores(x, w)
    order = torch.sort(-sc, dim=1, stable=True).indices[:, :K]
    idx = torch.sort(order, dim=1).values
    deltas = []
    for b in range(B):
        xp = x[b, idx[b]]
        q, k, v = _split(s, _norm(s, xp, w, "ln1") @ w["w_qkv"].T + w["b_qkv"])
        q, k = _rope(s, q, idx[b]), _rope(s, k, idx[b])
        d = _delta(s, xp, _attend(s, q, k, v, True), w)
        deltas.append(d)
        if sink is not None:
            sink.append((k, v, sc[b, idx[b]].min()))
        x[b, idx[b]] = xp + (torch.sigmoid(sc[b, idx[b]])[:, None] * d if gate else d)
    return torch.stack(deltas), idx, sc


def _final(s, x, e):
    return _ln(x, e["final_w"], e["final_b"], s.norm_eps) if s.arch == S.NEOX else _rms(x, e["final_w"], s.norm_eps)


def _exact_model(case, s, seed):
    """(final hidden states, Eq. 4 sums, layers' caches, extra weights, layers' weights)."""
    e = _double(_extra(s, seed))
    layers = [_double(_layer(s, seed, l)) for l in range(s.n_layers)]
    x = e["embed"][_ids(s, seed, 7, (case["B"], case["T"])).long()]
    acc, caches = [], []
    for w, K in zip(layers, _plan(case)):
        x0, sink = x.clone(), []
        _exact_layer(s, w, x, K, False, sink)
        cos = (x0 * x).sum(-1) / (x0.norm(dim=-1).clamp_min(1e-8) * x.norm(dim=-1).clamp_min(1e-8))
        acc += [cos.sum(), torch.tensor(float(cos.numel()), device=x.device, dtype=torch.float64)]
        caches.append(sink)
    return _final(s, x, e), torch.stack(acc), caches, e, layers


def _exact_steps(case, s, seed, caches, e, layers):
    nxt = _ids(s, seed, 8, (case["steps"], case["B"]))
    outs = []
    for i in range(case["steps"]):
        x = e["embed"][nxt[i].long()]
        pos = torch.full((1,), case["T"] + i, device=x.device)
        for w, cache in zip(layers, caches):
            sc = _scores(x, w)
            q, k, v = _split(s, _norm(s, x, w, "ln1") @ w["w_qkv"].T + w["b_qkv"])
            y = x.clone()
            for b in range(case["B"]):
                kc, vc, thr = cache[b]
                if not bool(sc[b] > thr):
                    continue
                kc = torch.cat([kc, _rope(s, k[b:b + 1], pos)])
                vc = torch.cat([vc, v[b:b + 1]])
                cache[b] = (kc, vc, thr)
                o = _attend(s, _rope(s, q[b:b + 1], pos), kc, vc, False)
                y[b] = x[b] + _delta(s, x[b:b + 1], o, w)[0]
            x = y
        outs.append(_final(s, x, e))
    return torch.stack(outs)


def exact(case, seed):
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    s = _shape(case)
    kind = case["kind"]
    if kind == "layer":
        x = _hidden(s, seed, case["B"], case["T"]).double()
        _exact_layer(s, _double(_layer(s, seed, 0)), x, case["K"], case["gate"])
        return x
    if kind == "attention":
        B, K = case["B"], case["K"]
        qkv = _normal(_gen(seed, 6), (B * K, s.qkv_dim), 1.0).to(_dtype(s)).double().reshape(B, K, -1)
        return torch.cat([_attend(s, *_split(s, qkv[b]), True) for b in range(B)])
    if kind == "model":
        hidden, acc = _exact_model(case, s, seed)[:2]
        return (hidden, acc) if case["stats"] else hidden
    if kind in ("decode", "generate"):
        hidden, _, caches, e, layers = _exact_model(case, s, seed)
        out = _exact_steps(case, s, seed, caches, e, layers)
        return (out, None) if kind == "decode" else (hidden, out, None)
    if kind == "align":
        w = _double(_layer(s, seed, 0))
        x0 = _hidden(s, seed, case["B"], case["T"])
        hd = _dense_target(s, x0, seed).double().reshape(-1, s.d)
        x0 = x0.double()
        y = x0.clone()
        delta, idx, sc = _exact_layer(s, w, y, case["K"], True)
        p = torch.softmax(y.reshape(-1, s.d), -1)
        r = p - torch.softmax(hd, -1)
        n = r.norm(dim=-1, keepdim=True)
        grad_y = p * (r - (p * r).sum(-1, keepdim=True)) / n
        rows = (torch.arange(case["B"], device=x0.device)[:, None] * case["T"] + idx).reshape(-1)
        xk = x0.reshape(-1, s.d)[rows]
        u = xk @ w["router_w1"].T + w["router_b1"]
        sig, sg = torch.sigmoid(sc.reshape(-1)[rows]), torch.sigmoid(u)
        ds = sig * (1 - sig) * (grad_y[rows] * delta.reshape(-1, s.d)).sum(-1)
        du = ds[:, None] * w["router_w2"] * sg * (1 + u * (1 - sg))
        grad = torch.cat([(du.T @ xk).reshape(-1), du.sum(0), (ds[:, None] * u * sg).sum(0), ds.sum()[None]])
        loss = torch.stack([n.sum(), torch.tensor(float(n.numel()), device=n.device, dtype=torch.float64)])
        return {"loss": loss, "grad_y": grad_y, "grad_router": grad, "y": y}
    hs, hd, head = (t.double() for t in _head(case, s, seed))
    ls, ld = torch.log_softmax(hs @ head.T, -1), torch.log_softmax(hd @ head.T, -1)
    kl = (ld.exp() * (ld - ls)).sum()
    return torch.stack([kl, torch.tensor(float(case["rows"]), device=kl.device, dtype=torch.float64)])
