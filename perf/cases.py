"""Workloads of the quantised linear layer and the operators around it, as a user's program runs them.

Five kinds, each through the public entry points of the package:

  linear  one layer on M tokens, called directly
  block   the linear path of whole decoder blocks: norm, q/k/v, rotary embedding, output projection, norm, gated
          feed-forward (the attention core is the caller's; the rotated queries stand in for its result)
  a8      the seven projections of a block with activations quantised to int8
  kv      attention over a KV cache held as weights: append the new tokens, scores, output
  ends    the two ends of a model: embedding lookup of a prompt, last norm and LM head

Decode-sized steps (few tokens) are replayed as a CUDA graph that the program captured once, the way a serving loop
does; everything else is called directly.  Weights are scaled like a trained layer's (a projection keeps the variance of its
input), activations are N(0, 1) in fp16.
"""
from __future__ import annotations

import math

import torch

import paper_2505_00232_b200 as P

DEVICE = "cuda:0"
GRAPH_MAX_M = 64            # token counts up to this are what a serving loop captures as a graph

GEMMA2_2B = {"hidden": 2304, "q_heads": 8, "kv_heads": 4, "d_h": 256, "ffn": 9216, "act": "gelu_tanh"}
LLAMA31_8B = {"hidden": 4096, "q_heads": 32, "kv_heads": 8, "d_h": 128, "ffn": 14336, "act": "silu"}
# (bits, group) of the attention projections and of the feed-forward layers
SCHEMES = {"q8": ((8, 0), (8, 0)), "844": ((8, 0), (4, 0)), "844g32": ((8, 0), (4, 32))}


def listed():
    return [
        # a single small projection called from a program's own loop: launch and call overhead
        {"name": "linear_small", "kind": "linear", "N": 2304, "K": 2304, "bits": 8, "group": 0, "M": 1},
        # a generated token on the two models, one user
        {"name": "decode_gemma2_2b", "kind": "block", **GEMMA2_2B, "scheme": "844g32", "M": 1, "layers": 4},
        {"name": "decode_llama31_8b", "kind": "block", **LLAMA31_8B, "scheme": "844g32", "M": 1, "layers": 2},
        # the same for a handful of users with int8 weights everywhere
        {"name": "decode_llama31_8b_q8_m4", "kind": "block", **LLAMA31_8B, "scheme": "q8", "M": 4, "layers": 2},
        # a batch of users, more than the few that the one-token kernels take
        {"name": "batch_llama31_8b_m32", "kind": "block", **LLAMA31_8B, "scheme": "844g32", "M": 32, "layers": 2},
        # prompts: a ragged one on the small model, a long one on the large model
        {"name": "prefill_gemma2_2b_m777", "kind": "block", **GEMMA2_2B, "scheme": "844g32", "M": 777, "layers": 1},
        {"name": "prefill_llama31_8b_m2048", "kind": "block", **LLAMA31_8B, "scheme": "844g32", "M": 2048, "layers": 1},
        # the per-channel scheme with int8 activations: a token, and a prompt
        {"name": "a8_decode_llama31_8b", "kind": "a8", **LLAMA31_8B, "scheme": "844", "M": 1},
        {"name": "a8_prefill_llama31_8b_m1024", "kind": "a8", **LLAMA31_8B, "scheme": "844", "M": 1024},
        # attention over a long cache: a generated token, and a chunk of a prompt
        {"name": "kv_decode_8192", "kind": "kv", "heads": 8, "group": 4, "d_h": 128, "cache": 8192, "filled": 8000, "new": 1, "layers": 4},
        {"name": "kv_chunk_256_of_4096", "kind": "kv", "heads": 8, "group": 4, "d_h": 128, "cache": 4096, "filled": 3000, "new": 256, "layers": 1},
        # a prompt's embedding rows and the logits of its last token
        {"name": "ends_llama31_8b", "kind": "ends", "vocab": 128256, "hidden": 4096, "tokens": 2048, "rows": 1},
    ]


def _log_int(rng, lo, hi, step=1):
    """A multiple of `step` in [lo, hi], spread evenly over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi // step, max(-(-lo // step), int(round(v / step)))) * step


def _draw_dims(rng):
    d_h = rng.choice([64, 128, 128, 256])
    kv_heads = rng.choice([1, 2, 4, 8])
    group = rng.choice([1, 2, 4, 7])
    while kv_heads * group * d_h > 8192:
        group = max(1, group // 2)
    hidden = _log_int(rng, 1024, 5120, 128)
    return {"hidden": hidden, "q_heads": kv_heads * group, "kv_heads": kv_heads, "d_h": d_h,
            "ffn": max(1024, int(round(hidden * rng.uniform(2.5, 4.0) / 256)) * 256), "act": rng.choice(["silu", "gelu_tanh"])}


def draw(rng):
    kind = rng.choices(["linear", "block", "a8", "kv", "ends"], [3, 5, 2, 3, 1])[0]
    if kind == "linear":
        bits, group = rng.choice([(8, 0), (4, 32), (4, 0), (4, 128)])
        K = _log_int(rng, 512, 14336, {8: 32, 4: 128 if group == 128 else 64}[bits])
        N = _log_int(rng, 512, 16384, 8)
        M = _log_int(rng, 1, 2048)
        return {"kind": kind, "N": N, "K": K, "bits": bits, "group": group, "M": M}
    if kind == "block":
        M = _log_int(rng, 1, 2048)
        layers = rng.choice([1, 2, 3]) if M <= GRAPH_MAX_M else 1
        dims = rng.choice([GEMMA2_2B, LLAMA31_8B, None, None]) or _draw_dims(rng)
        if dims["hidden"] * dims["ffn"] > LLAMA31_8B["hidden"] * LLAMA31_8B["ffn"]:
            M = min(M, 1500)
        return {"kind": kind, **dims, "scheme": rng.choice(list(SCHEMES)), "M": M, "layers": layers}
    if kind == "a8":
        dims = rng.choice([GEMMA2_2B, LLAMA31_8B])
        decode = rng.random() < 0.5
        # a prompt in the integer form: the per-channel schemes, more than 128 tokens
        return {"kind": kind, **dims, "scheme": rng.choice(list(SCHEMES) if decode else ["q8", "844"]),
                "M": _log_int(rng, 1, 8) if decode else _log_int(rng, 129, 1024)}
    if kind == "kv":
        decode = rng.random() < 0.6
        heads, d_h = rng.choice([1, 2, 4, 8]), rng.choice([64, 128, 128, 256])
        group = rng.choice([1, 2, 4, 7, 8])
        cache = _log_int(rng, 256, 32768 if decode else 8192, 32)
        new = 1 if decode else _log_int(rng, 16, 256)
        return {"kind": kind, "heads": heads, "group": group, "d_h": d_h, "cache": cache, "filled": rng.randint(0, cache - new), "new": new,
                "layers": rng.choice([2, 4]) if decode else 1}
    return {"kind": kind, "vocab": _log_int(rng, 32000, 128256, 8), "hidden": _log_int(rng, 1024, 4096, 128), "tokens": _log_int(rng, 1, 2048), "rows": _log_int(rng, 1, 8)}


# ------------------------------------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device=DEVICE).half()


def _weights(g, N, K, bits, group):
    """Random integers over the full range and scales with which the product keeps the variance of its input."""
    lo, hi = (-8, 8) if bits == 4 else (-127, 128)
    q = torch.randint(lo, hi, (N, K), generator=g, device=DEVICE, dtype=torch.int8)
    rms = math.sqrt((hi - lo) ** 2 / 12.0)
    s = (torch.rand((N, K // group if group else 1), generator=g, device=DEVICE) + 0.5) / (rms * math.sqrt(K))
    return q, s.clamp_min(6.2e-5).half()


def _layer(g, N, K, bits, group):
    q, s = _weights(g, N, K, bits, group)
    return P.QLinear.from_weights(q.cpu().numpy(), s.cpu().numpy(), bits, group, device=DEVICE)


def _projections(case):
    """(name, N, K, bits, group) of a block's seven projections."""
    attn, ffn = SCHEMES[case["scheme"]]
    h, f = case["hidden"], case["ffn"]
    qd, kd = case["q_heads"] * case["d_h"], case["kv_heads"] * case["d_h"]
    return [("q", qd, h, *attn), ("k", kd, h, *attn), ("v", kd, h, *attn), ("o", h, qd, *attn), ("gate", f, h, *ffn), ("up", f, h, *ffn), ("down", h, f, *ffn)]


def _is_captured(case):
    """Whether a program would keep the step as a CUDA graph: the steps that generate tokens."""
    if case["kind"] == "kv":
        return case["new"] == 1
    return case["kind"] in ("block", "a8") and case["M"] <= GRAPH_MAX_M


def _captured(step):
    """The step as a CUDA graph, and the outputs that a replay fills."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = step()
    return graph, out


def _inputs(case, seed, layer, cache):
    """The state of a case; layer(g, N, K, bits, group) and cache(heads, positions, d_h) make what holds weights and keys."""
    g = _generator(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "linear":
        st["layer"] = layer(g, case["N"], case["K"], case["bits"], case["group"])
        st["x"] = _normal(g, case["M"], case["K"])
    elif kind in ("block", "a8"):
        st["blocks"] = [{n: layer(g, N, K, b, gr) for n, N, K, b, gr in _projections(case)} for _ in range(case.get("layers", 1))]
        M, h = case["M"], case["hidden"]
        st["x"] = _normal(g, M, h)
        if kind == "a8":
            st["attn"], st["inner"] = _normal(g, M, case["q_heads"] * case["d_h"]), _normal(g, M, case["ffn"])
        else:
            for b in st["blocks"]:
                b["norm1"], b["norm2"] = ((1.0 + 0.1 * torch.randn(h, generator=g, device=DEVICE)).half() for _ in range(2))
            n_pos, half = 4096, case["d_h"] // 2
            angle = torch.arange(n_pos, device=DEVICE, dtype=torch.float64)[:, None] * 10000.0 ** (-torch.arange(half, device=DEVICE, dtype=torch.float64) / half)
            st["cos"], st["sin"] = angle.cos().float().contiguous(), angle.sin().float().contiguous()
            # a decode step is one token of each user, a prompt is one user's consecutive tokens
            st["batch"] = M if M <= GRAPH_MAX_M else 1
            st["pos"] = (torch.randint(0, n_pos, (M,), generator=g, device=DEVICE) if M <= GRAPH_MAX_M else torch.arange(M, device=DEVICE)).int()
    elif kind == "kv":
        H, d, T, new = case["heads"], case["d_h"], case["cache"], case["new"]
        R = new * case["group"]
        st["layers"] = []
        for _ in range(case["layers"]):
            kv = cache(H, T, d)
            if case["filled"]:
                kv.append(_normal(g, H, case["filled"], d), _normal(g, H, case["filled"], d))
            # (the softmax between the two products is the caller's: its result is an input here)
            prob = torch.zeros((H, R, T), device=DEVICE, dtype=torch.float16)
            n = case["filled"] + new
            prob[:, :, :n] = torch.softmax(2.0 * torch.randn((H, R, n), generator=g, device=DEVICE), -1).half()
            st["layers"].append({"kv": kv, "k": _normal(g, H, new, d), "v": _normal(g, H, new, d), "q": _normal(g, H, R, d), "prob": prob})
    else:
        st["table"] = layer(g, case["vocab"], case["hidden"], 4, 32)
        st["ids"] = torch.randint(0, case["vocab"], (case["tokens"],), generator=g, device=DEVICE).int()
        st["x"] = _normal(g, case["rows"], case["hidden"])
        st["norm"] = (1.0 + 0.1 * torch.randn(case["hidden"], generator=g, device=DEVICE)).half()
    return st


def prepare(case, seed):
    st = _inputs(case, seed, _layer, lambda heads, positions, d_h: P.KVHeads(heads, positions, d_h, device=DEVICE))
    if _is_captured(case):
        st["graph"], st["out"] = _captured(lambda: _step(st))
    return st


# ------------------------------------------------------------------------------------------------ one pass
def _block_step(st):
    case, out = st["case"], []
    M, hq, hkv, d = case["M"], case["q_heads"], case["kv_heads"], case["d_h"]
    B, S = st["batch"], case["M"] // st["batch"]
    delta, h = st["x"], None
    for w in st["blocks"]:
        h, y = P.qlinear_residual_rmsnorm(delta, h, w["norm1"], 1e-5)
        q, k, v = P.qlinear_forward_group([w["q"], w["k"], w["v"]], y)
        q, k, v = P.qlinear_rope_qkv(q, k, v, st["pos"], st["cos"], st["sin"], B, S, hq, hkv, d)
        o = w["o"].forward(q.view(M, hq * d))
        h, y = P.qlinear_residual_rmsnorm(o, h, w["norm2"], 1e-5)
        delta = w["down"].forward(P.qlinear_forward_gated(w["gate"], w["up"], y, case["act"]))
        out += [k, v]
    return out + [h, delta]


def _kv_step(st):
    case, out = st["case"], []
    for layer in st["layers"]:
        kv = layer["kv"]
        kv.length = case["filled"]                       # the same positions in every pass
        kv.append(layer["k"], layer["v"])
        scores = kv.scores(layer["q"])
        if case["new"] * case["group"] <= 8:
            o = kv.output(layer["prob"])
        else:
            o = [head.output(layer["prob"][i]) for i, head in enumerate(kv.heads)]
        out += [scores, o]
    return out


def _step(st):
    kind = st["case"]["kind"]
    if kind == "linear":
        return st["layer"].forward(st["x"])
    if kind == "block":
        return _block_step(st)
    if kind == "a8":
        w = st["blocks"][0]
        return [w[n].forward_a8(st["attn"] if n == "o" else st["inner"] if n == "down" else st["x"]) for n in ("q", "k", "v", "o", "gate", "up", "down")]
    if kind == "kv":
        return _kv_step(st)
    rows = st["table"].embed(st["ids"])
    _, y = P.qlinear_residual_rmsnorm(st["x"], None, st["norm"], 1e-5, want_h=False)
    return [rows, st["table"].forward(y)]


def run(st):
    if "graph" in st:
        st["graph"].replay()
        return st["out"]
    return _step(st)


# ------------------------------------------------------------------------------------------------ what a pass cannot do without
def _weight_bytes(N, K, bits, group):
    return N * K * bits // 8 + 2 * N * (K // group if group else 1)


def work(case):
    kind = case["kind"]
    if kind == "linear":
        N, K, M = case["N"], case["K"], case["M"]
        return {"bytes": _weight_bytes(N, K, case["bits"], case["group"]) + 2 * M * (N + K), "flops": 2 * M * N * K}
    if kind in ("block", "a8"):
        proj, M, n = _projections(case), case["M"], case.get("layers", 1)
        weights = n * sum(_weight_bytes(*p[1:]) for p in proj)
        flops = n * sum(2 * M * p[1] * p[2] for p in proj)
        if kind == "a8":
            acts = 2 * M * (case["hidden"] + case["q_heads"] * case["d_h"] + case["ffn"] + sum(p[1] for p in proj))
        else:
            acts = 2 * M * (3 * case["hidden"] + n * 2 * case["kv_heads"] * case["d_h"]) + n * 4 * case["hidden"]
        return {"bytes": weights + acts, "flops": flops}
    if kind == "kv":
        H, d, T, new, n = case["heads"], case["d_h"], case["cache"], case["new"], case["layers"]
        R = new * case["group"]
        cache = H * (2 * T * d + 4 * T)                  # int8 keys and values, two fp16 scales per token
        acts = H * (2 * 2 * new * d + 2 * 2 * R * d + 2 * 2 * R * T)
        return {"bytes": n * (cache + acts), "flops": n * H * 4 * R * T * d}
    V, h, t, r = case["vocab"], case["hidden"], case["tokens"], case["rows"]
    return {"bytes": _weight_bytes(V, h, 4, 32) + t * (_weight_bytes(1, h, 4, 32) + 4 + 2 * h) + 2 * r * (2 * h + V), "flops": 2 * r * V * h}


def tolerance(case):
    # Four times the 2-norm distance from the same pass in 64 bits: one product and its fp16 rounding 2.8e-4; a block
    # rounds to fp16 after every operator, 1.6e-3 over two blocks; the value scales of a cache are folded into fp16
    # probabilities, whose product is subnormal over long caches, 1.1e-3.
    return {"rel": {"linear": 1.2e-3, "block": 6.4e-3, "a8": 1.2e-3, "kv": 4.5e-3, "ends": 1.2e-3}[case["kind"]]}


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _weights64(g, N, K, bits, group):
    q, s = _weights(g, N, K, bits, group)
    return lambda: (q.double().view(N, -1, group or K) * s.double()[:, :, None]).view(N, K)


class _Cache64:
    """Keys and values quantised to int8 with one fp16 scale per token (decided in fp32, as the cache defines it)."""

    def __init__(self, heads, positions, d_h):
        self.k, self.v = (torch.zeros((heads, positions, d_h), device=DEVICE, dtype=torch.float64) for _ in range(2))
        self.length = 0

    def append(self, k, v):
        at = slice(self.length, self.length + k.shape[1])
        for store, x in ((self.k, k.float()), (self.v, v.float())):
            s = (x.abs().amax(-1, keepdim=True) / 127.0).half().float()
            store[:, at] = (torch.round(x / s).clamp(-127, 127) * s).double()
        self.length = at.stop


def _norm64(h, gamma):
    return h / (h.square().mean(-1, keepdim=True) + 1e-5).sqrt() * gamma.double()


def _block64(st):
    case, out = st["case"], []
    M, hq, hkv, d = case["M"], case["q_heads"], case["kv_heads"], case["d_h"]
    B, S, gq = st["batch"], case["M"] // st["batch"], case["q_heads"] // case["kv_heads"]
    cos, sin = (st[n].double()[st["pos"].long()][:, None, :] for n in ("cos", "sin"))

    def rotate(x, heads):
        lo, hi = x.view(M, heads, d).split(d // 2, -1)
        return torch.cat([lo * cos - hi * sin, hi * cos + lo * sin], -1)

    def per_kv_head(x, n):                               # [B S, h_kv n, d] -> [B h_kv, S n, d]
        return x.reshape(B, S, hkv, n, d).permute(0, 2, 1, 3, 4).reshape(B * hkv, S * n, d)
    h, delta = 0.0, st["x"].double()
    for w in st["blocks"]:
        h = h + delta
        y = _norm64(h, w["norm1"])
        q, k, v = (y @ w[n]().T for n in "qkv")
        out += [per_kv_head(rotate(k, hkv), 1), per_kv_head(v.view(M, hkv, d), 1)]
        h = h + per_kv_head(rotate(q, hq), gq).reshape(M, hq * d) @ w["o"]().T
        y = _norm64(h, w["norm2"])
        gate = y @ w["gate"]().T
        gate = torch.nn.functional.silu(gate) if case["act"] == "silu" else torch.nn.functional.gelu(gate, approximate="tanh")
        delta = (gate * (y @ w["up"]().T)) @ w["down"]().T
    return out + [h, delta]


def _a8_64(x, w):
    """Activations quantised per token (decided in fp32, as the call defines it), then the product."""
    amax = x.float().abs().amax(-1, keepdim=True)
    xq = torch.round(x.float() * (127.0 / amax)).clamp(-127, 127)
    return (xq.double() @ w.T) * (amax / 127.0).double()


def exact(case, seed):
    st = _inputs(case, seed, _weights64, _Cache64)
    kind, out = case["kind"], []
    if kind == "linear":
        return st["x"].double() @ st["layer"]().T
    if kind == "block":
        return _block64(st)
    if kind == "a8":
        w = st["blocks"][0]
        return [_a8_64(st["attn"] if n == "o" else st["inner"] if n == "down" else st["x"], w[n]()) for n in ("q", "k", "v", "o", "gate", "up", "down")]
    if kind == "kv":
        for layer in st["layers"]:
            kv, prob = layer["kv"], layer["prob"].double()
            kv.append(layer["k"], layer["v"])
            o = prob @ kv.v
            out += [layer["q"].double() @ kv.k.transpose(1, 2), o if case["new"] * case["group"] <= 8 else list(o)]
        return out
    table = st["table"]()
    return [table[st["ids"].long()], _norm64(st["x"].double(), st["norm"]) @ table.T]
