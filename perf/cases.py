"""The work whose speed is measured: calls that a program using this package makes.

Five families, each through the package's public entry points:

  linear    the projections of `layers` decoder layers (and the lm_head) in
            decoder order, as one sq_linear_chain: a draft pass (INT4 or FP8
            weights, one row per sequence), a verify pass (FP16 weights, K + 1
            rows per sequence) or a prefill pass (up to 256 rows).  Programs
            capture such a pass into a CUDA graph and replay it, as
            generate.Generator and bench.py do; `graph: False` is the plain
            call.  Every layer reads a resident N(0, 1) hidden state and the
            `o` projection reads the head of the q/k/v output (the wiring of
            stack.pass_ops), but each keeps its own outputs, so all come back.
  attention the new tokens' keys and values into the cache, then grouped-query
            attention over it (in one launch at one new token, as
            stack.decoder_pass does).
  accept    the accept / resample step from logits, or (K = 0) sampling one
            token per sequence.
  quantize  deriving an INT4 or FP8 variant from an FP16 matrix.
  decoder   a whole decoder pass from token ids to logits, replayed as a graph.

Sizes are those of shapes.STACKS, or generic.
"""
from __future__ import annotations

import math

import torch

import paper_2609_21704_gb300 as sq
from paper_2609_21704_gb300.shapes import STACKS, StackShape
from paper_2609_21704_gb300.stack import DecoderState, LinearStack, decoder_pass

HEAD_DIM = 128
THETA = 1e6
RMS_EPS = 1e-6
WKIND = {"fp16": sq.SQ_W_FP16, "int4": sq.SQ_W_INT4, "fp8": sq.SQ_W_FP8}
WEIGHT_BYTES = {"fp16": 2.0, "int4": 0.5 + 2.0 / 128.0, "fp8": 1.0}
# rates behind the cost bound of drawn cases (bytes/s, flop/s); only their
# ratio matters
COST_BYTES, COST_FLOPS = 6.8e12, 1.7e15


# ---- cases ---------------------------------------------------------------------

def _linear(name, stack, variant, rows, layers, head, graph=True):
    s = STACKS[stack]
    return {"name": name, "family": "linear", "hidden": s.hidden, "q_heads": s.q_heads,
            "kv_heads": s.kv_heads, "inter": s.intermediate, "vocab": s.vocab, "layers": layers,
            "head": head, "attn_proj": True, "variant": variant, "rows": rows, "graph": graph}


def listed():
    mlp = _linear("mlp_0p5b_int4_1row", "qwen2.5-0.5b-mlp", "int4", 1, 1, False, graph=False)
    mlp["attn_proj"] = False
    return [
        # the smallest draft step: one MLP block of the 0.5B shape, one row,
        # called eagerly (two launches of a few microseconds)
        mlp,
        # a whole INT4 draft pass of the 1.5B stack at batch 1 (113 launches)
        _linear("draft_1p5b_int4_1row", "qwen2.5-1.5b", "int4", 1, 28, True),
        # the headline's draft pass: 14B layers and lm_head, INT4, batch 1
        _linear("draft_14b_int4_1row", "qwen2.5-14b", "int4", 1, 4, True),
        # an FP8 draft at batch 8
        _linear("draft_7b_fp8_8rows", "qwen2.5-7b", "fp8", 8, 4, True),
        # an INT4 draft at batch 16
        _linear("draft_14b_int4_16rows", "qwen2.5-14b", "int4", 16, 4, True),
        # the parent verifies 16 sequences of 4 drafts: 80 rows
        _linear("verify_14b_fp16_80rows", "qwen2.5-14b", "fp16", 80, 4, True),
        # the largest pass one call takes: 256 prompt rows through the parent
        # (a prefill pass that only fills the cache runs no lm_head)
        _linear("prefill_14b_fp16_256rows", "qwen2.5-14b", "fp16", 256, 4, False),
        # decode attention of the 14B heads: 4 sequences, 8000 tokens each, in
        # caches of 16384
        {"name": "attention_decode_8k", "family": "attention", "B": 4, "T": 1, "q_heads": 40,
         "kv_heads": 8, "ctx": 8000, "max_ctx": 16384},
        # one prefill chunk of the 7B heads (28 tokens, the most a call takes)
        # behind 2000 tokens
        {"name": "attention_prefill_28", "family": "attention", "B": 4, "T": 28, "q_heads": 28,
         "kv_heads": 4, "ctx": 2000, "max_ctx": 4096},
        # the accept step of 16 sequences of 8 drafts, from the lm_heads' logits
        {"name": "accept_b16_k8", "family": "accept", "B": 16, "K": 8, "vocab": 152064,
         "mode": "sample", "temperature": 1.0},
        # deriving the INT4 variant of the 14B fused gate/up matrix
        {"name": "quantize_int4_14b_gate_up", "family": "quantize", "N": 27648, "K": 5120,
         "variant": "int4"},
        # the parent's whole verify pass over five tokens behind 1000 (1.5B)
        _decoder("decoder_verify_1p5b", "qwen2.5-1.5b", "fp16", 1, 5, 28, 1000, 2048),
    ]


def _decoder(name, stack, variant, B, T, layers, ctx, max_ctx):
    s = STACKS[stack]
    return {"name": name, "family": "decoder", "hidden": s.hidden, "q_heads": s.q_heads,
            "kv_heads": s.kv_heads, "inter": s.intermediate, "vocab": s.vocab, "layers": layers,
            "variant": variant, "B": B, "T": T, "ctx": ctx, "max_ctx": max_ctx}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost(case):
    w = work(case)
    return w["bytes"] / COST_BYTES + w["flops"] / COST_FLOPS


def draw(rng):
    cap = max(_cost(c) for c in listed())
    case = None
    while case is None or _cost(case) > cap:
        case = _draw_any(rng)
    return case


def _draw_any(rng):
    family = rng.choice(["linear"] * 6 + ["attention"] * 3 + ["accept", "quantize", "decoder"])
    if family == "linear":
        variant = rng.choice(["int4", "int4", "fp8", "fp16"])
        stack = rng.choice(list(STACKS) + ["generic"])
        if stack == "generic":  # ragged sizes: each weight format's own granularity of K
            gran = {"int4": 128, "fp8": 16, "fp16": 8}[variant]
            kv = rng.choice([1, 2, 3, 5])
            case = {"family": "linear", "hidden": gran * _log_int(rng, 512 // gran, 6144 // gran),
                    "q_heads": kv * rng.choice([1, 3, 6]), "kv_heads": kv,
                    "inter": gran * _log_int(rng, 512 // gran, 16384 // gran),
                    "vocab": _log_int(rng, 1001, 160001), "attn_proj": True}
        else:
            case = _linear("", stack, "int4", 1, 1, False)
            del case["name"]
            case["attn_proj"] = stack != "qwen2.5-0.5b-mlp"
        case["variant"] = variant
        case["rows"] = _log_int(rng, 1, 256)
        case["layers"] = rng.randint(1, 4)
        case["head"] = rng.random() < 0.5
        case["graph"] = rng.random() < 0.75
        return case
    if family == "attention":
        kv = rng.choice([1, 2, 4, 8])
        g = rng.choice([1, 2, 5, 6, 7, 8])
        T = rng.choice([1, 1, 2, _log_int(rng, 2, min(32, 200 // g)), min(32, 200 // g)])
        ctx = _log_int(rng, 1, 16000)
        return {"family": "attention", "B": _log_int(rng, 1, 16), "T": T, "q_heads": kv * g,
                "kv_heads": kv, "ctx": ctx, "max_ctx": int((ctx + T) * rng.choice([1.0, 1.3, 4.0]))}
    if family == "accept":
        vocab = rng.choice([32000, 151936, 152064, _log_int(rng, 1000, 200000)])
        return {"family": "accept", "B": _log_int(rng, 1, 16), "K": rng.choice([0, 1, 2, 4, 5, 8]),
                "vocab": vocab, "mode": rng.choice(["sample", "greedy"]),
                "temperature": rng.choice([0.7, 1.0])}
    if family == "quantize":
        gran = rng.choice([128, 16])
        return {"family": "quantize", "N": _log_int(rng, 1000, 40000),
                "K": gran * _log_int(rng, 512 // gran, 19000 // gran),
                "variant": "int4" if gran == 128 else "fp8"}
    ctx = _log_int(rng, 16, 4000)
    stack = rng.choice(["qwen2.5-1.5b", "qwen2.5-7b", "qwen2.5-14b"])
    T = rng.randint(1, 9)
    case = _decoder("", stack, rng.choice(["int4", "fp8", "fp16"]), _log_int(rng, 1, 8), T,
                    rng.randint(1, 6), ctx, ctx + T + rng.choice([0, 500]))
    del case["name"]
    return case


# ---- inputs --------------------------------------------------------------------

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _normal(seed, shape, std=1.0, dtype=torch.float16):
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    return torch.empty(shape, dtype=dtype, device=_device()).normal_(0.0, std, generator=g)


def _weight_seed(seed, index):
    """The seed of a LinearStack's index-th projection (decoder order, then
    the lm_head, then the embedding)."""
    return (seed + index) * 7919 + 17


def _shape(case):
    return StackShape("case", case["hidden"], case["q_heads"], case["kv_heads"], case["inter"],
                      case["vocab"], case["layers"])


def _dims(case):
    """(name, output columns, weight rows, K) of one layer's projections."""
    q, kv = case["q_heads"] * HEAD_DIM, case["kv_heads"] * HEAD_DIM
    h, i = case["hidden"], case["inter"]
    return [("qkv", q + 2 * kv, q + 2 * kv, h), ("o", h, h, q), ("gate_up", i, 2 * i, h), ("down", h, h, i)]


def _linear_dims(case):
    return _dims(case) if case["attn_proj"] else _dims(case)[2:]


def _uniforms(seed, shape):
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    m = torch.randint(0, 1 << 24, shape, device=_device(), generator=g)
    return m.to(torch.float64).mul_(2.0 ** -24).to(torch.float32)


def _capture(fn):
    """fn run once on a side stream, then captured there as a graph."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        fn(s)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        fn(s)
    return g


def prepare(case, seed):
    return {"linear": _prepare_linear, "attention": _prepare_attention, "accept": _prepare_accept,
            "quantize": _prepare_quantize, "decoder": _prepare_decoder}[case["family"]](case, seed)


def run(state):
    if "graph" in state:
        state["graph"].replay()
    else:
        state["call"]()
    return state["out"]


def _stack_seed(seed):
    return 1000 * (seed % 100003)


def _x_seed(seed):
    return _stack_seed(seed) + 500_000_019


def _linear_x(case, seed):
    return _normal(_x_seed(seed), (case["rows"], case["hidden"]))


def _prepare_linear(case, seed):
    variant, M = case["variant"], case["rows"]
    stack = LinearStack(_shape(case), _device(), seed=_stack_seed(seed),
                        variants=() if variant == "fp16" else (variant,), with_lm_head=case["head"])
    x = _linear_x(case, seed)
    wk, ops = WKIND[variant], []

    def new(*shape):
        return torch.empty(shape, dtype=torch.float16, device=_device())

    # one output tensor per projection: [layers, rows, columns]
    y = {name: new(case["layers"], M, cols) for name, cols, _, _ in _linear_dims(case)}
    for li, layer in enumerate(stack.layers):
        p = {proj.name: proj.weight(variant) for proj in layer}
        if case["attn_proj"]:
            q_out = case["q_heads"] * HEAD_DIM
            qkv, o = y["qkv"][li], y["o"][li]
            attn = qkv.view(-1)[: M * q_out].view(M, q_out)
            ops.append((wk, x, *p["qkv"], None, None, sq.SQ_EPI_NONE, qkv))
            ops.append((wk, attn, *p["o"], None, None, sq.SQ_EPI_NONE, o))
        h, d = y["gate_up"][li], y["down"][li]
        ops.append((wk, x, *p["gate_up"], None, None, sq.SQ_EPI_SILU_GATE, h))
        ops.append((wk, h, *p["down"], None, None, sq.SQ_EPI_NONE, d))
    out = list(y.values())
    if case["head"]:
        out.append(new(M, case["vocab"]))
        ops.append((wk, x, *stack.lm_head.weight(variant), None, None, sq.SQ_EPI_NONE, out[-1]))
    state = {"stack": stack, "x": x, "out": out}
    if case["graph"]:
        state["graph"] = _capture(lambda s: sq.sq_linear_chain(ops, s))
    else:
        state["call"] = lambda: sq.sq_linear_chain(ops)
    return state


def _attention_inputs(case, seed):
    B, T, Hq, Hkv = case["B"], case["T"], case["q_heads"], case["kv_heads"]
    width = (Hq + 2 * Hkv) * HEAD_DIM
    cache = (B, Hkv, case["max_ctx"], HEAD_DIM)
    qkv = _normal(_x_seed(seed), (B * T, width))
    k, v = _normal(_x_seed(seed) + 1, cache), _normal(_x_seed(seed) + 2, cache)
    # sequences of a batch differ in length: `ctx` and a few tokens less
    pos0 = torch.tensor([max(0, case["ctx"] - 7 * b) for b in range(B)], dtype=torch.int32, device=_device())
    return qkv, k, v, pos0


def _prepare_attention(case, seed):
    B, T, Hq, Hkv = case["B"], case["T"], case["q_heads"], case["kv_heads"]
    qkv, k, v, pos0 = _attention_inputs(case, seed)
    out = torch.empty((B * T, Hq * HEAD_DIM), dtype=torch.float16, device=_device())
    ws = torch.empty(sq.sq_attention_workspace_bytes(B, T, Hq, Hkv, case["max_ctx"]), dtype=torch.uint8,
                     device=_device())

    def call():
        if T == 1:
            sq.sq_attention_append(qkv, B, T, Hq, Hkv, pos0, THETA, k, v, out, ws)
        else:
            sq.sq_kv_append(qkv, B, T, Hq, Hkv, pos0, THETA, k, v)
            sq.sq_attention(qkv, B, T, Hq, Hkv, pos0, THETA, k, v, out, ws)

    return {"call": call, "out": [out, k, v]}


def _prepare_accept(case, seed):
    B, K, V = case["B"], case["K"], case["vocab"]
    dev, s = _device(), _x_seed(seed)
    zp = _normal(s, (B, K + 1, V), 2.0)
    u = _uniforms(s + 3, (B, K + 1))
    n = torch.empty((B,), dtype=torch.int32, device=dev)
    tok = torch.empty((B, K + 1), dtype=torch.int32, device=dev)
    ws = torch.zeros(sq.sq_accept_logits_workspace_bytes(B, K, V), dtype=torch.uint8, device=dev)
    mode = sq.SQ_ACCEPT_GREEDY if case["mode"] == "greedy" else sq.SQ_ACCEPT_SAMPLE
    T = case["temperature"]
    if K == 0 and case["mode"] == "sample":
        z = zp.view(B, V)
        return {"call": lambda: sq.sq_sample_logits(z, u, T, tok, ws), "out": [tok]}
    zq, draft = None, None
    if K > 0:  # the draft's logits are the parent's with noise; its tokens are drawn from them
        zq = (zp[:, :K].transpose(0, 1).float() + _normal(s + 1, (K, B, V), 0.5, torch.float32)).half()
        zq = zq.contiguous()
        g = torch.Generator(device=dev)
        g.manual_seed(s + 2)
        p = torch.softmax(zq.float() / T, dim=-1).view(K * B, V)
        draft = torch.multinomial(p, 1, generator=g).view(K, B).t().contiguous().to(torch.int32)
    return {"call": lambda: sq.sq_accept_logits(zp, zq, draft, u, T, mode, n, tok, ws), "out": [n, tok]}


def _prepare_quantize(case, seed):
    N, K = case["N"], case["K"]
    w = _normal(_x_seed(seed), (N, K), 0.02)
    kind = sq.SQ_INT4_G128 if case["variant"] == "int4" else sq.SQ_FP8_E4M3_ROW
    cb, _ = sq.sq_quantized_bytes(kind, N, K)
    codes = torch.empty((N, cb // N), dtype=torch.uint8, device=_device())
    if case["variant"] == "int4":
        scales = torch.empty((N, K // 128), dtype=torch.float16, device=_device())
    else:
        scales = torch.empty((N,), dtype=torch.float32, device=_device())
    return {"call": lambda: sq.sq_quantize(w, kind, codes, scales), "out": [codes, scales]}


def _decoder_inputs(case, seed):
    """Gains, cached keys and values per layer, token ids, positions."""
    nl, B, T = case["layers"], case["B"], case["T"]
    s = _x_seed(seed)
    gains = [(1.0 + _normal(s + 10 + i, (case["hidden"],), 0.05).float()).half() for i in range(2 * nl + 1)]
    cache = (nl, B, case["kv_heads"], case["max_ctx"], HEAD_DIM)
    ks, vs = _normal(s + 1000, cache), _normal(s + 2000, cache)
    g = torch.Generator(device=_device())
    g.manual_seed(s + 3)
    ids = torch.randint(0, case["vocab"], (B * T,), device=_device(), generator=g).to(torch.int32)
    pos0 = torch.tensor([max(0, case["ctx"] - 5 * b) for b in range(B)], dtype=torch.int32, device=_device())
    table = _normal(s + 4, (case["vocab"], case["hidden"]))
    return gains, ks, vs, ids, pos0, table


def _prepare_decoder(case, seed):
    variant, B, T = case["variant"], case["B"], case["T"]
    stack = LinearStack(_shape(case), _device(), seed=_stack_seed(seed),
                        variants=() if variant == "fp16" else (variant,))
    st = DecoderState(stack, B, T, case["max_ctx"])
    st.gamma, ks, vs, ids, pos0, table = _decoder_inputs(case, seed)
    st.k, st.v = list(ks), list(vs)

    def step(s):
        sq.sq_embed(ids, table, st.x, s)
        decoder_pass(stack, variant, st, s, pos0=pos0)

    return {"graph": _capture(step), "out": [st.logits, st.x, ks, vs], "keep": (stack, st, ids, pos0, table)}


# ---- work and tolerances ---------------------------------------------------------

def _linear_work(dims, rows, wb):
    b = sum(wb * n * k + 2 * rows * (k + cols) for _, cols, n, k in dims)
    return {"bytes": b, "flops": sum(2 * rows * n * k for _, _, n, k in dims)}


def work(case):
    f = case["family"]
    if f in ("linear", "decoder"):
        dims = (_linear_dims(case) if f == "linear" else _dims(case)) * case["layers"]
        if f == "decoder" or case["head"]:
            dims = dims + [("lm_head", case["vocab"], case["vocab"], case["hidden"])]
        rows = case["rows"] if f == "linear" else case["B"] * case["T"]
        w = _linear_work(dims, rows, WEIGHT_BYTES[case["variant"]])
        if f == "decoder":
            a = _attention_work(case)
            w = {key: w[key] + case["layers"] * a[key] for key in w}
        return w
    if f == "attention":
        return _attention_work(case)
    if f == "accept":
        # every logit row is needed for its normaliser
        rows = case["B"] * (2 * case["K"] + 1)
        return {"bytes": 2 * rows * case["vocab"], "flops": 2 * rows * case["vocab"]}
    n = case["N"] * case["K"]
    return {"bytes": (2 + WEIGHT_BYTES[case["variant"]]) * n, "flops": 2 * n}


def _attention_work(case):
    B, T, Hq, Hkv = case["B"], case["T"], case["q_heads"], case["kv_heads"]
    L = case["ctx"] + T
    return {"bytes": 4 * B * Hkv * HEAD_DIM * L + 2 * B * T * (2 * Hq + 4 * Hkv) * HEAD_DIM,
            "flops": 4 * B * T * Hq * HEAD_DIM * L}


def tolerance(case):
    f = case["family"]
    if f in ("accept", "quantize"):
        return "exact"  # whole numbers, codes and their scales
    if f == "decoder":
        # fp16 activations rounded between the layers of a whole model (2.8e-3
        # against exact() after 28 layers)
        return {"rel": 1.2e-2}
    if f == "attention":
        return {"rel": 1e-3}  # fp32 sums, one fp16 rounding (2.1e-4)
    # one or two chained products, fp32 sums, fp16 results: 2.1e-4 to 3.4e-4,
    # and 4.2e-4 where an INT4 weight is rounded once to fp16
    return {"rel": 1.7e-3}


# ---- the same in 64 bits -----------------------------------------------------------

def exact(case, seed):
    with torch.no_grad():
        return {"linear": _exact_linear, "attention": _exact_attention, "accept": lambda c, s: None,
                "quantize": _exact_quantize, "decoder": _exact_decoder}[case["family"]](case, seed)


def _divide(a, b):
    """a / b with one rounding (a scalar divisor would be taken as a product
    with its reciprocal)."""
    return a / torch.full_like(a, b)


def _quantized(w, variant):
    """(codes, scales) of the definitions in the header: IEEE fp32 divides."""
    n, k = w.shape
    wf = w.float()
    if variant == "int4":
        g = wf.view(n, k // 128, 128)
        amax = g.abs().amax(dim=-1)
        s = _divide(amax, 7.0).half()
        s = torch.where((amax > 0) & (s == 0), torch.full_like(s, 2.0 ** -24), s)
        sf = s.float().unsqueeze(-1)
        c = torch.where(sf != 0, torch.round(g / torch.where(sf != 0, sf, torch.ones_like(sf))), 0.0 * g)
        return c.clamp(-8, 7).view(n, k), s
    s = _divide(wf.abs().amax(dim=-1), 448.0)
    sf = s.unsqueeze(-1)
    c = torch.where(sf != 0, wf / torch.where(sf != 0, sf, torch.ones_like(sf)), 0.0 * wf)
    return c.clamp(-448, 448).to(torch.float8_e4m3fn), s


def _dequantized(w, variant):
    """The weights a variant stands for, in 64 bits."""
    if variant == "fp16":
        return w.double()
    c, s = _quantized(w, variant)
    if variant == "int4":
        n, k = w.shape
        return (c.view(n, k // 128, 128).double() * s.double().unsqueeze(-1)).view(n, k)
    return c.float().double() * s.double().unsqueeze(-1)


def _matmul(x, seed, n, k, variant):
    """x W'^T in 64 bits, a slice of the output rows at a time."""
    w = _normal(seed, (n, k), 0.02)
    step = max(1, (1 << 26) // k)
    return torch.cat([x @ _dequantized(w[i:i + step], variant).t() for i in range(0, n, step)], dim=1)


def _silu_gate(y):
    g, u = y.chunk(2, dim=1)
    return g * torch.sigmoid(g) * u


def _exact_linear(case, seed):
    variant, M, s0 = case["variant"], case["rows"], _stack_seed(seed)
    x = _linear_x(case, seed).double()
    ys, i = {name: [] for name, _, _, _ in _linear_dims(case)}, 0
    for _ in range(case["layers"]):
        for name, _, n, k in _dims(case):
            ws = _weight_seed(s0, i)
            i += 1
            if name not in ys:
                continue
            if name == "o":
                y = _matmul(ys["qkv"][-1].reshape(-1)[: M * k].view(M, k), ws, n, k, variant)
            elif name == "gate_up":
                y = _silu_gate(_matmul(x, ws, n, k, variant))
            else:
                y = _matmul(ys["gate_up"][-1] if name == "down" else x, ws, n, k, variant)
            ys[name].append(y)
    out = [torch.stack(y) for y in ys.values()]
    if case["head"]:
        out.append(_matmul(x, _weight_seed(s0, i), case["vocab"], case["hidden"], variant))
    return out


def _rotate(x, pos):
    """x [T, heads, 128] rotated at positions pos [T]: pairs (d, d + 64)."""
    d = torch.arange(HEAD_DIM // 2, dtype=torch.float64, device=x.device)
    a = pos.double().view(-1, 1, 1) * float(torch.tensor(THETA, dtype=torch.float32)) ** (-2.0 * d / HEAD_DIM)
    x1, x2 = x[..., : HEAD_DIM // 2], x[..., HEAD_DIM // 2:]
    return torch.cat([x1 * a.cos() - x2 * a.sin(), x2 * a.cos() + x1 * a.sin()], dim=-1)


def _attend(qkv, B, T, Hq, Hkv, pos0, k, v):
    """Appends to k, v (64-bit [B, Hkv, ctx, 128]) in place; the attention rows."""
    rows = qkv.view(B, T, Hq + 2 * Hkv, HEAD_DIM)
    out = torch.empty((B, T, Hq, HEAD_DIM), dtype=torch.float64, device=qkv.device)
    G = Hq // Hkv
    for b in range(B):
        p0 = int(pos0[b])
        L = p0 + T
        pos = torch.arange(p0, L, device=qkv.device)
        q = _rotate(rows[b, :, :Hq], pos)
        k[b, :, p0:L] = _rotate(rows[b, :, Hq:Hq + Hkv], pos).transpose(0, 1)
        v[b, :, p0:L] = rows[b, :, Hq + Hkv:].transpose(0, 1)
        mask = torch.arange(L, device=qkv.device).view(1, 1, L) <= pos.view(T, 1, 1)
        for h in range(Hkv):
            sc = (q[:, h * G:(h + 1) * G] @ k[b, h, :L].t()) / math.sqrt(HEAD_DIM)
            out[b, :, h * G:(h + 1) * G] = sc.masked_fill(~mask, -math.inf).softmax(dim=-1) @ v[b, h, :L]
    return out.view(B * T, Hq * HEAD_DIM)


def _exact_attention(case, seed):
    qkv, k, v, pos0 = _attention_inputs(case, seed)
    k, v = k.double(), v.double()
    out = _attend(qkv.double(), case["B"], case["T"], case["q_heads"], case["kv_heads"], pos0, k, v)
    return [out, k, v]


def _exact_quantize(case, seed):
    w = _normal(_x_seed(seed), (case["N"], case["K"]), 0.02)
    codes, scales = [], []
    step = max(1, (1 << 26) // case["K"])
    for i in range(0, case["N"], step):
        c, s = _quantized(w[i:i + step], case["variant"])
        if case["variant"] == "int4":
            n = (c + 8).to(torch.uint8)
            codes.append(n[:, 0::2] | (n[:, 1::2] << 4))
        else:
            codes.append(c.view(torch.uint8))
        scales.append(s)
    return [torch.cat(codes), torch.cat(scales)]


def _exact_decoder(case, seed):
    gains, ks, vs, ids, pos0, table = _decoder_inputs(case, seed)
    ks, vs = ks.double(), vs.double()
    variant, s0 = case["variant"], _stack_seed(seed)
    B, T, Hq, Hkv = case["B"], case["T"], case["q_heads"], case["kv_heads"]

    def norm(x, g):
        return x / torch.sqrt(x.square().mean(dim=-1, keepdim=True) + RMS_EPS) * g.double()

    x = table[ids.long()].double()
    for li in range(case["layers"]):
        (_, _, nq, kq), (_, _, no, ko), (_, _, ng, kg), (_, _, nd, kd) = _dims(case)
        ws = [_weight_seed(s0, 4 * li + j) for j in range(4)]
        qkv = _matmul(norm(x, gains[2 * li]), ws[0], nq, kq, variant)
        a = _attend(qkv, B, T, Hq, Hkv, pos0, ks[li], vs[li])
        x = x + _matmul(a, ws[1], no, ko, variant)
        h = _silu_gate(_matmul(norm(x, gains[2 * li + 1]), ws[2], ng, kg, variant))
        x = x + _matmul(h, ws[3], nd, kd, variant)
    logits = _matmul(norm(x, gains[-1]), _weight_seed(s0, 4 * case["layers"]), case["vocab"], case["hidden"],
                     variant)
    return [logits, x, ks, vs]
