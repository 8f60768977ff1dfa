"""The work that users of this library have it do, as cases that can be timed and compared.

Every case goes through the public Python entry points of ``paper_2604_16498_b200.binding`` with the buffers that a
serving or evaluation program keeps: output tensors, the decode workspace, weights.  Inputs are unit-variance normals
(weights have standard deviation 1 / sqrt(fan-in), so that every pre-activation has unit variance too); cached or padded
lengths are uniform.  Shapes are those of the library's own workloads and tests: a GPT-2-small-shaped model (12 heads of
64, width 768, MLP 3072), a 1B-class one (32 query and 8 KV heads of 64, width 2048, MLP 8192) and an 8B-class one (32
query and 8 KV heads of 128, width 4096, MLP 14336).

``listed()`` has one case per kind of use; ``draw()`` spreads sizes, data types and options over the same kinds.
"""
import math

import torch

from paper_2604_16498_b200 import binding as forge

NONE, CAUSAL, PADDING, CAUSAL_PADDING = forge.MASK_NONE, forge.MASK_CAUSAL, forge.MASK_PADDING, forge.MASK_CAUSAL_PADDING
_DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}


# ---------------------------------------------------------------------------------------------------------- cases
def _attention(dtype, B, Hq, Hkv, Sq, Skv, D, mask, min_len=0, bias_heads=0):
    """min_len: valid lengths are uniform in [min_len, Skv] where the mask has padding; bias_heads: 0 without an additive
    mask tensor, 1 for one shared by all heads, Hq for one per head."""
    return dict(kind="attention", dtype=dtype, B=B, Hq=Hq, Hkv=Hkv, Sq=Sq, Skv=Skv, D=D, mask=mask, min_len=min_len,
                bias_heads=bias_heads)


def _decode(dtype, B, Hq, Hkv, Smax, D, min_len, splits):
    return dict(kind="decode", dtype=dtype, B=B, Hq=Hq, Hkv=Hkv, Smax=Smax, D=D, min_len=min_len, splits=splits)


def _linear(dtype, M, N, K, act, layout, bias=True, residual=False):
    """dtype "w8": int8 weights with fp16 activations.  act "swiglu": the gated MLP input with a second weight matrix."""
    return dict(kind="linear", dtype=dtype, M=M, N=N, K=K, act=act, layout=layout, bias=bias, residual=residual)


def _layer(B, S, Hq, Hkv, D, F, mlp, layout, bias):
    return dict(kind="layer", B=B, S=S, Hq=Hq, Hkv=Hkv, D=D, F=F, mlp=mlp, layout=layout, bias=bias)


def listed():
    return [
        # The smallest call: one 128-token prompt of a GPT-2-small-shaped model evaluated in fp32 (latency).
        dict(_attention("f32", 1, 12, 12, 128, 128, 64, CAUSAL), name="attn_f32_b1_s128"),
        # Sentence classification in batches: short sequences of mixed length, padded to 128 (launch and copies).
        dict(_attention("bf16", 32, 12, 12, 128, 128, 64, PADDING, min_len=16), name="attn_encoder_b32_s128"),
        # Perplexity evaluation of a GPT-2-small-shaped model over full contexts.
        dict(_attention("bf16", 8, 12, 12, 1024, 1024, 64, CAUSAL), name="attn_d64_b8_s1024"),
        # Prompt processing of an 8B-class model: the largest attention of the benchmark.
        dict(_attention("bf16", 4, 32, 8, 2048, 2048, 128, CAUSAL), name="attn_gqa_b4_s2048"),
        # Chunked prefill in fp16: an odd chunk of queries behind a cached prefix of uneven length, 7 query heads per KV head.
        dict(_attention("f16", 3, 28, 4, 777, 1801, 128, CAUSAL_PADDING, min_len=1024), name="attn_f16_chunk_777_1801"),
        # Token generation for a batch of 16 conversations of an 8B-class model.
        dict(_decode("bf16", 16, 32, 8, 4096, 128, 1024, 16), name="decode_b16_4096"),
        # Token generation at the end of one long document (the workspace and splits that the header recommends for it).
        dict(_decode("f16", 1, 32, 8, 32768, 128, 32768, 128), name="decode_f16_b1_32768"),
        # The first MLP projection of a GPT-2-small-shaped model over a large batch of tokens.
        dict(_linear("bf16", 8192, 3072, 768, "gelu_tanh", "kn"), name="linear_gelu_8192"),
        # A down projection with its residual while 16 conversations generate tokens (the weights are streamed once).
        dict(_linear("bf16", 16, 4096, 14336, "none", "nk", bias=False, residual=True), name="linear_add_m16"),
        # Weight-only int8, 128-token prompt: the largest model's setting in the evaluation.
        dict(_linear("w8", 128, 14336, 4096, "silu", "nk", bias=False), name="linear_w8_m128"),
        # A whole GPT-2-small-shaped layer for one 128-token prompt (five dependent small operators).
        dict(_layer(1, 128, 12, 12, 64, 3072, "gelu", "kn", True), name="layer_gpt2_b1_s128"),
        # A whole 8B-class layer for 8192 prompt tokens: the largest case.
        dict(_layer(4, 2048, 32, 8, 128, 14336, "swiglu", "nk", False), name="layer_8b_b4_s2048"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_attention(rng):
    dtype = rng.choice(["bf16", "bf16", "f16"])
    Hq, Hkv = rng.choice([(12, 12), (32, 8), (28, 4), (16, 4), (16, 16)])
    D = rng.choice([64, 64, 80, 96, 128, 128, 128, 256])
    Sq = _log_int(rng, 16, 4096)
    Skv = Sq + rng.choice([0, 0, 0, _log_int(rng, 1, 2048)])
    mask = rng.choice([CAUSAL, CAUSAL, PADDING, CAUSAL_PADDING, NONE])
    B = max(1, min(_log_int(rng, 1, 64), 16384 // Skv))
    bias = 0
    if dtype == "bf16" and D <= 128 and rng.random() < 0.2:
        bias = rng.choice([1, Hq])
        B = max(1, min(B, (64 << 20) // (bias * Sq * Skv)))
    return _attention(dtype, B, Hq, Hkv, Sq, Skv, D, mask, min_len=max(1, Skv // 8), bias_heads=bias)


def _draw_decode(rng):
    B = _log_int(rng, 1, 64)
    Hq, Hkv = rng.choice([(32, 8), (32, 8), (12, 12), (28, 4)])
    D = 64 if Hq == 12 else rng.choice([64, 128, 128])
    Smax = min(_log_int(rng, 64, 32768), (1 << 20) // (B * Hkv // 4))
    # splits: what the header recommends for few (sequence, head) pairs, else the benchmark's 16
    splits = max(16, min(256, 7 * 148 // (B * Hkv)))
    return _decode(rng.choice(["bf16", "f16"]), B, Hq, Hkv, Smax, D, max(1, Smax // 4), splits)


def _draw_linear(rng):
    M = _log_int(rng, 1, 8192)
    width, mlp = rng.choice([(768, 3072), (2048, 8192), (4096, 14336), (8 * _log_int(rng, 32, 512), 8 * _log_int(rng, 32, 1536))])
    N, K = rng.choice([(width, width), (mlp, width), (width, mlp)])
    dtype = rng.choice(["bf16", "bf16", "f16", "w8"])
    if dtype == "w8":
        K = (K + 15) // 16 * 16
    return _linear(dtype, M, N, K, rng.choice(["none", "gelu_tanh", "silu", "relu", "gelu_erf"]),
                   "nk" if dtype == "w8" else rng.choice(["kn", "nk"]), bias=rng.random() < 0.5, residual=rng.random() < 0.3)


def _draw_swiglu(rng):
    width, mlp = rng.choice([(2048, 8192), (4096, 14336)])
    return _linear("bf16", _log_int(rng, 1, 8192), mlp, width, "swiglu", rng.choice(["kn", "nk"]), bias=False)


def _draw_layer(rng):
    S = _log_int(rng, 16, 2048)
    B = max(1, min(_log_int(rng, 1, 16), 8192 // S))
    model = rng.choice(["gpt2", "1b", "8b"])
    if model == "gpt2":
        return _layer(B, min(S, 1024), 12, 12, 64, 3072, "gelu", "kn", True)
    if model == "1b":
        return _layer(B, S, 32, 8, 64, 8192, "swiglu", "nk", False)
    return _layer(B, S, 32, 8, 128, 14336, "swiglu", "nk", False)


def draw(rng):
    kind = rng.choice(["attention", "attention", "attention", "attention_f32", "decode", "decode", "linear", "linear", "linear",
                       "swiglu", "layer"])
    if kind == "attention":
        return _draw_attention(rng)
    if kind == "attention_f32":
        S = _log_int(rng, 8, 512)
        return _attention("f32", rng.randint(1, 8), 12, 12, S, S, rng.choice([64, 64, 128]), rng.choice([CAUSAL, CAUSAL, PADDING]),
                          min_len=max(1, S // 8))
    return {"decode": _draw_decode, "linear": _draw_linear, "swiglu": _draw_swiglu, "layer": _draw_layer}[kind](rng)


# ---------------------------------------------------------------------------------------------------------- inputs
class _Draws:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, shape, dtype, std=1.0):
        return torch.randn(shape, generator=self.g, device="cuda").mul_(std).to(dtype)

    def lens(self, B, lo, hi):
        return torch.randint(lo, hi + 1, (B,), generator=self.g, device="cuda", dtype=torch.int32)


_ACTS = {"gelu_tanh": forge.ACT_GELU_TANH, "gelu_erf": forge.ACT_GELU_ERF, "relu": forge.ACT_RELU, "silu": forge.ACT_SILU,
         "none": forge.ACT_NONE}
_LAYOUTS = {"kn": forge.W_KN, "nk": forge.W_NK}


def prepare(case, seed):
    r = _Draws(seed)
    s = {"case": case}
    kind = case["kind"]
    if kind == "attention":
        B, Hq, Hkv, Sq, Skv, D = (case[k] for k in ("B", "Hq", "Hkv", "Sq", "Skv", "D"))
        dt = _DTYPES[case["dtype"]]
        s["q"] = r.normal((B, Hq, Sq, D), dt)
        s["k"] = r.normal((B, Hkv, Skv, D), dt)
        s["v"] = r.normal((B, Hkv, Skv, D), dt)
        s["lens"] = r.lens(B, case["min_len"], Skv) if case["mask"] & PADDING else None
        if case["bias_heads"]:
            s["bias"] = r.normal((B, case["bias_heads"], Sq, Skv), torch.float32)
        s["out"] = torch.empty_like(s["q"])
    elif kind == "decode":
        B, Hq, Hkv, Smax, D = (case[k] for k in ("B", "Hq", "Hkv", "Smax", "D"))
        dt = _DTYPES[case["dtype"]]
        s["q"] = r.normal((B, Hq, D), dt)
        s["k"] = r.normal((B, Hkv, Smax, D), dt)
        s["v"] = r.normal((B, Hkv, Smax, D), dt)
        s["lens"] = r.lens(B, case["min_len"], Smax)
        s["out"] = torch.empty_like(s["q"])
        s["workspace"] = torch.empty(forge.attn_decode_workspace_bytes(B, Hq, D, case["splits"]), dtype=torch.uint8, device="cuda")
        forge.attn_decode_workspace_init(s["workspace"])
    elif kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float16
        s["x"] = r.normal((M, K), dt)
        wshape = (K, N) if case["layout"] == "kn" else (N, K)
        if case["dtype"] == "w8":  # symmetric per-channel quantisation of weights with standard deviation 1 / sqrt(K)
            s["w"] = r.normal((N, K), torch.float32, 32.0).round_().clamp_(-127, 127).to(torch.int8)
            s["scale"] = (torch.rand((N,), generator=r.g, device="cuda") + 0.5) / (32.0 * math.sqrt(K))
        else:
            s["w"] = r.normal(wshape, dt, K ** -0.5)
        if case["act"] == "swiglu":
            s["w_up"] = r.normal(wshape, dt, K ** -0.5)
        s["b"] = r.normal((N,), dt, 0.02) if case["bias"] else None
        s["residual"] = r.normal((M, N), dt) if case["residual"] else None
        s["out"] = torch.empty((M, N), dtype=dt, device="cuda")
    else:
        B, S, Hq, Hkv, D, F = (case[k] for k in ("B", "S", "Hq", "Hkv", "D", "F"))
        H, bf = Hq * D, torch.bfloat16

        def weight(fan_in, fan_out):
            return r.normal((fan_in, fan_out) if case["layout"] == "kn" else (fan_out, fan_in), bf, fan_in ** -0.5)

        w = {"w_qkv": weight(H, (Hq + 2 * Hkv) * D), "w_o": weight(H, H), "w_up": weight(H, F), "w_down": weight(F, H)}
        if case["mlp"] == "swiglu":
            w["w_gate"] = weight(H, F)
        if case["bias"]:
            for name, n in (("b_qkv", (Hq + 2 * Hkv) * D), ("b_o", H), ("b_up", F), ("b_down", H)):
                w[name] = r.normal((n,), bf, 0.02)
        s["weights"] = w
        s["x"] = r.normal((B * S, H), bf)
        s["out"] = torch.empty_like(s["x"])
        plan = forge.decoder_layer_plan(B, S, Hq, Hkv, D, F, forge.MLP_SWIGLU if case["mlp"] == "swiglu" else forge.MLP_GELU)
        s["workspace"] = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "attention":
        if c["bias_heads"]:
            return forge.attn_fused_bias(s["q"], s["k"], s["v"], s["bias"], c["mask"], s["lens"], out=s["out"])
        fn = {"bf16": forge.attn_fused, "f16": forge.attn_fused_f16, "f32": forge.attn_fused_f32}[c["dtype"]]
        return fn(s["q"], s["k"], s["v"], c["mask"], s["lens"], out=s["out"])
    if kind == "decode":
        return forge.attn_decode_splitkv(s["q"], s["k"], s["v"], s["lens"], c["splits"], out=s["out"], workspace=s["workspace"])
    if kind == "linear":
        if c["act"] == "swiglu":
            return forge.linear_swiglu(s["x"], s["w"], s["w_up"], _LAYOUTS[c["layout"]], out=s["out"])
        if c["dtype"] == "w8":
            return forge.linear_act_w8a16(s["x"], s["w"], s["scale"], s["b"], s["residual"], _ACTS[c["act"]], out=s["out"])
        return forge.linear_act(s["x"], s["w"], s["b"], s["residual"], _ACTS[c["act"]], _LAYOUTS[c["layout"]], out=s["out"])
    return forge.decoder_layer(s["x"], s["weights"], c["B"], c["S"], c["Hq"], c["Hkv"], c["D"], c["F"],
                               forge.MLP_SWIGLU if c["mlp"] == "swiglu" else forge.MLP_GELU, _LAYOUTS[c["layout"]], CAUSAL,
                               out=s["out"], workspace=s["workspace"])


# ---------------------------------------------------------------------------------------------------------- work
def _visible(Sq, Skv, mask, kv_len):
    """(query, key) pairs of one head with kv_len valid keys."""
    if not mask & CAUSAL:
        return Sq * kv_len
    off = Skv - Sq  # query i sees keys up to i + off
    full = max(0, min(Sq, Sq - (kv_len - off)))  # queries that see all kv_len keys
    part = Sq - full
    return part * off + part * (part + 1) // 2 + full * kv_len


def work(case):
    """Lengths drawn from the seed count with their mean."""
    kind = case["kind"]
    if kind == "attention":
        B, Hq, Hkv, Sq, Skv, D = (case[k] for k in ("B", "Hq", "Hkv", "Sq", "Skv", "D"))
        es = 4 if case["dtype"] == "f32" else 2
        kv = (case["min_len"] + Skv) // 2 if case["mask"] & PADDING else Skv
        pairs = B * Hq * _visible(Sq, Skv, case["mask"], kv)
        by = es * D * (2 * B * Hq * Sq + 2 * B * Hkv * kv)
        if case["bias_heads"]:
            by += 4 * B * case["bias_heads"] * _visible(Sq, Skv, case["mask"], kv)
        return {"bytes": by, "flops": 4 * D * pairs}
    if kind == "decode":
        B, Hq, Hkv, D = case["B"], case["Hq"], case["Hkv"], case["D"]
        tokens = B * (case["min_len"] + case["Smax"]) // 2
        return {"bytes": 4 * Hkv * D * tokens + 4 * B * Hq * D, "flops": 4 * D * Hq * tokens}
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        mats = 2 if case["act"] == "swiglu" else 1
        wb = 1 if case["dtype"] == "w8" else 2
        by = 2 * M * K + mats * wb * N * K + 2 * M * N * (2 if case["residual"] else 1) + 2 * N * int(case["bias"])
        return {"bytes": by, "flops": 2 * mats * M * N * K}
    B, S, Hq, Hkv, D, F = (case[k] for k in ("B", "S", "Hq", "Hkv", "D", "F"))
    H, T = Hq * D, B * S
    params = H * (Hq + 2 * Hkv) * D + H * H + H * F * (3 if case["mlp"] == "swiglu" else 2)
    return {"bytes": 2 * params + 4 * T * H, "flops": 2 * T * params + 4 * D * B * Hq * _visible(S, S, CAUSAL, S)}


def tolerance(case):
    """About four times the relative error measured against an fp64 evaluation of the same operator: 2e-7 .. 3.4e-7 for fp32
    attention; 1.9e-3 .. 2.6e-3 for bf16 attention, decode and layers (probabilities and outputs are rounded to bf16) and
    1.66e-3 for bf16 linears (outputs rounded once); 2.3e-4 .. 2.9e-4 for fp16 attention and 2.1e-4 for fp16 linears."""
    dtype = case.get("dtype", "bf16")
    if dtype == "f32":
        return {"rel": 1.5e-6}
    if case["kind"] == "linear":
        return {"rel": 7e-3 if dtype == "bf16" else 9e-4}
    return {"rel": 1e-2 if dtype == "bf16" else 1.2e-3}
