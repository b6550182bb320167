"""The calls that a serving program makes of this library, at the sizes it makes them with.

listed() names twelve of them: the smallest linear, the linears of one layer at
decode and prefill sizes (NVFP4 and MXFP4), the fused MLP, decode attention
over long and ragged caches, a prompt's K/V append, a decode step of a layer's
whole attention block, and the quantization of a weight at load time.  draw()
gives more cases of the same ranges.  Shapes are those of
paper_2606_15682_gb300/synth.py and the tests, or generic.

Decode-sized calls run as a CUDA graph that the program captured once, as a
serving loop does; prefill-sized ones are called directly.
"""
import math

import torch

from paper_2606_15682_gb300 import nvfp4 as N

DEV = "cuda"
HEAD_DIM = 128


# ------------------------------------------------------------------ cases ---

def listed():
    return [
        # One small projection for a handful of sequences: latency only.
        dict(name="linear_m16", kind="dyn", M=16, N=1536, K=1536),
        # A 14B layer's four linears for a single sequence: every weight byte streamed for one token.
        dict(name="linears_14b_m1", kind="linears", fmt="nvfp4", M=1, hidden=5120, qkv=7168, o_in=5120, inter=13824),
        # The same layer at the deployment's decode batch.
        dict(name="linears_14b_m256", kind="linears", fmt="nvfp4", M=256, hidden=5120, qkv=7168, o_in=5120, inter=13824),
        # Prefill of a small model: short K, where per-tile and per-launch costs count.
        dict(name="linears_1.5b_m2048", kind="linears", fmt="nvfp4", M=2048, hidden=1536, qkv=2048, o_in=1536, inter=8960),
        # Prefill of a large model: the compute-bound end.
        dict(name="linears_32b_m8192", kind="linears", fmt="nvfp4", M=8192, hidden=5120, qkv=10240, o_in=8192, inter=27648),
        # The MXFP4 variant with its block rotation, one ragged prompt.
        dict(name="mx_linears_m1000", kind="linears", fmt="mxfp4_rot", M=1000, hidden=5120, qkv=7168, o_in=5120,
             inter=13824),
        # The MLP with SwiGLU and the down projection's quantization in the epilogue, a ragged prompt.
        dict(name="mlp_14b_m777", kind="mlp", fmt="nvfp4", M=777, hidden=5120, inter=13824),
        # Decode attention at the long-reasoning end: 64 sequences of 16384 tokens.
        dict(name="attn_b64_t16384", kind="attention", kv="e2m1", batch=64, heads=40, kv_heads=8, capacity=16384,
             ragged=False),
        # Decode attention for a few sequences of different lengths, the QAT runs' E1M2 elements.
        dict(name="attn_e1m2_b3_ragged", kind="attention", kv="e1m2", batch=3, heads=40, kv_heads=8, capacity=8000,
             ragged=True),
        # One prompt's keys and values: RoPE, shift, quantize, append.
        dict(name="append_rope_t4093", kind="append", kv="e2m1", batch=1, kv_heads=8, tokens=4093, rope=True),
        # A decode step of a 14B layer's attention block, from its input to the o projection's output, 32 sequences of
        # different lengths.
        dict(name="block_14b_b32", kind="block", kv="e2m1", batch=32, hidden=5120, heads=40, kv_heads=8, capacity=4096),
        # A weight at load time: tensor scale, then codes and scales.
        dict(name="weight_13824x5120", kind="weight", rows=13824, cols=5120),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(rng, lo, hi, m):
    return max(1, round(_log(rng, lo, hi) / m)) * m


MOST_FLOPS = 8e12


def draw(rng):
    kind = rng.choice(["dyn", "linears", "linears", "linears", "mlp", "attention", "attention", "append", "block",
                       "weight"])
    if kind == "dyn":
        return dict(kind=kind, M=rng.randint(1, 32), N=_mult(rng, 256, 10240, 16), K=256 * rng.randint(1, 6))
    if kind in ("linears", "mlp"):
        M = _log(rng, 1, 8192)
        hidden, inter = _mult(rng, 1024, 8192, 256), _mult(rng, 2048, 27648, 256)
        while 6.0 * M * hidden * inter * (4 / 3) > MOST_FLOPS:
            M = max(1, M * 2 // 3)
        if kind == "mlp":
            return dict(kind=kind, fmt=rng.choice(["nvfp4", "mxfp4", "mxfp4_rot"]), M=M, hidden=hidden, inter=inter)
        o_in = _mult(rng, 1024, 8192, 256)
        return dict(kind=kind, fmt=rng.choice(["nvfp4", "nvfp4", "mxfp4", "mxfp4_rot"]), M=M, hidden=hidden,
                    qkv=_mult(rng, 1024, 10240, 128), o_in=o_in, inter=inter)
    if kind == "attention":
        kv_heads = rng.randint(1, 8)
        batch, capacity = _log(rng, 1, 64), 2 * _log(rng, 64, 8192)
        return dict(kind=kind, kv=rng.choice(["e2m1", "e2m1", "e1m2"]), batch=batch, heads=kv_heads * rng.randint(1, 8),
                    kv_heads=kv_heads, capacity=capacity, ragged=rng.random() < 0.7)
    if kind == "append":
        return dict(kind=kind, kv=rng.choice(["e2m1", "e2m1", "e1m2"]), batch=rng.choice([1, 1, 3, 16]),
                    kv_heads=rng.randint(1, 8), tokens=_log(rng, 1, 16384), rope=rng.random() < 0.7)
    if kind == "block":
        kv_heads = rng.choice([2, 4, 8])
        return dict(kind=kind, kv="e2m1", batch=_log(rng, 1, 128), hidden=_mult(rng, 1024, 5120, 256),
                    heads=kv_heads * rng.choice([2, 4, 6, 8]), kv_heads=kv_heads, capacity=2 * _log(rng, 64, 4096))
    return dict(kind=kind, rows=_log(rng, 100, 30000), cols=_mult(rng, 1024, 13824, 64))


# ----------------------------------------------------------------- inputs ---

def _gen(seed, i):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1009 + i)
    return g


def _activation(rows, cols, seed, i):
    """N(0, 1) with 1 % of the channels 30 times as large, as decoder activations have them."""
    g = _gen(seed, i)
    x = torch.randn(rows, cols, generator=g, device=DEV)
    n = max(1, round(0.01 * cols))
    x[:, torch.randperm(cols, generator=g, device=DEV)[:n]] *= 30.0
    return x.to(torch.bfloat16)


def _weight(rows, cols, seed, i):
    g = _gen(seed, i)
    return (torch.randn(rows, cols, generator=g, device=DEV) * 0.02).to(torch.bfloat16)


def _kv(tokens, heads, seed, i):
    """Keys or values [tokens, heads, 128] with a lognormal spread over channels."""
    g = _gen(seed, i)
    spread = torch.exp(0.5 * torch.randn(heads, HEAD_DIM, generator=g, device=DEV))
    return (torch.randn(tokens, heads, HEAD_DIM, generator=g, device=DEV) * spread).to(torch.bfloat16)


def _queries(batch, heads, seed, i):
    return torch.randn(batch, heads, HEAD_DIM, generator=_gen(seed, i), device=DEV).to(torch.bfloat16)


def _lens(batch, capacity, ragged):
    """Cached tokens of each sequence: all of the capacity, or spread from an eighth of it up."""
    if not ragged:
        return [capacity] * batch
    return [max(1, capacity - (b * 7919) % max(1, capacity * 7 // 8)) for b in range(batch)]


def _rope_table(n):
    """(cos, sin) of p * 1e6^(-2i/128), rounded once."""
    inv = 1.0e6 ** (-torch.arange(0, HEAD_DIM, 2, dtype=torch.float64, device=DEV) / HEAD_DIM)
    ang = torch.arange(n, dtype=torch.float64, device=DEV)[:, None] * inv[None]
    return torch.stack([ang.cos(), ang.sin()], dim=-1).float().contiguous()


#: Static tensor scales of a calibrated deployment: the largest magnitude each tensor is expected to reach, over 6 * 448.
KV_G = 40.0 / 2688
O_G, ACT_G = 8.0 / 2688, 400.0 / 2688
SOFTMAX = 1.0 / math.sqrt(HEAD_DIM)


# --------------------------------------------------------------- the calls ---

def _empty(*shape, dtype=torch.uint8):
    return torch.empty(*shape, dtype=dtype, device=DEV)


def _scales(rows, cols, fmt):
    size = N.nvfp4_scales_bytes if fmt == "nvfp4" else N.mxfp4_scales_bytes
    return _empty(size(rows, cols, N.SCALES_MMA))


def _operand(rows, cols, fmt):
    """Buffers of one quantized operand: codes, scales, tensor scale."""
    return dict(codes=_empty(rows, cols // 2), scales=_scales(rows, cols, fmt), g=_empty(1, dtype=torch.float32))


def _quantize_weight(w, fmt):
    q = _operand(*w.shape, fmt)
    if fmt == "nvfp4":
        N.nvfp4_tensor_scale(w, q["g"])
        N.nvfp4_quantize(w, q["g"], q["codes"], q["scales"])
    else:
        N.mxfp4_quantize(w, q["codes"], q["scales"], rotate=fmt == "mxfp4_rot")
    return q


def _quantize(x, q, fmt, state):
    if fmt == "nvfp4":
        N.nvfp4_quantize_dynamic(x, state, q["g"], q["codes"], q["scales"])
    else:
        N.mxfp4_quantize(x, q["codes"], q["scales"], rotate=fmt == "mxfp4_rot")


def _linear(a, w, out, fmt):
    M, Nn = out.shape
    K = w["codes"].shape[1] * 2
    if fmt == "nvfp4":
        N.nvfp4_linear(a["codes"], a["scales"], a["g"], w["codes"], w["scales"], w["g"], out, M, Nn, K)
    else:
        N.mxfp4_linear(a["codes"], a["scales"], w["codes"], w["scales"], out, M, Nn, K)


def _swiglu(a, w, M, inter, K, h, fmt):
    if fmt == "nvfp4":
        N.nvfp4_linear_swiglu_quantize(a["codes"], a["scales"], a["g"], w["codes"], w["scales"], w["g"], M, inter, K,
                                       h["g"], h["codes"], h["scales"])
    else:
        N.mxfp4_linear_swiglu_quantize(a["codes"], a["scales"], w["codes"], w["scales"], M, inter, K, h["codes"],
                                       h["scales"], rotate=fmt == "mxfp4_rot")


def _gate_up(gate, up, fmt):
    w = torch.empty(2 * gate.shape[0], gate.shape[1], dtype=gate.dtype, device=DEV)
    N.nvfp4_interleave_gate_up(gate, up, w)
    return _quantize_weight(w, fmt)


def _bf16(*shape):
    return _empty(*shape, dtype=torch.bfloat16)


def _state_buffer():
    return torch.zeros(N.DYNAMIC_STATE_BYTES, dtype=torch.uint8, device=DEV)


def _weights(case, seed):
    """(name, N, K) of a layer's linears."""
    h = case["hidden"]
    return [("qkv", case["qkv"], h), ("o", h, case["o_in"]), ("gate_up", 2 * case["inter"], h),
            ("down", h, case["inter"])]


def _by_graph(case):
    """Decode-sized work is replayed from a graph; prompts are called directly."""
    kind = case["kind"]
    return kind in ("dyn", "attention", "block") or (kind in ("linears", "mlp") and case["M"] <= 512)


def prepare(case, seed):
    s = _prepare(case, seed)
    s["case"] = case
    torch.cuda.synchronize()
    if _by_graph(case):
        _pass(s)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            s["out"] = _pass(s)
        s["graph"] = graph
    return s


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["out"]
    return _pass(state)


def _prepare(case, seed):
    kind = case["kind"]
    if kind == "dyn":
        M, Nn, K = case["M"], case["N"], case["K"]
        return dict(x=_activation(M, K, seed, 0), w=_quantize_weight(_weight(Nn, K, seed, 1), "nvfp4"),
                    y=_bf16(M, Nn), g=_empty(1, dtype=torch.float32))
    if kind == "linears":
        M, fmt = case["M"], case["fmt"]
        return dict(state=_state_buffer(), linears=[
            dict(name=name, x=_activation(M, K, seed, 2 * i), w=_quantize_weight(_weight(Nn, K, seed, 2 * i + 1), fmt),
                 a=_operand(M, K, fmt), out=_bf16(M, Nn)) for i, (name, Nn, K) in enumerate(_weights(case, seed))])
    if kind == "mlp":
        M, fmt, h, I = case["M"], case["fmt"], case["hidden"], case["inter"]
        act = _operand(M, I, fmt)
        act["g"].fill_(ACT_G)
        return dict(state=_state_buffer(), x=_activation(M, h, seed, 0),
                    gate_up=_gate_up(_weight(I, h, seed, 1), _weight(I, h, seed, 2), fmt),
                    down=_quantize_weight(_weight(h, I, seed, 3), fmt), a=_operand(M, h, fmt), act=act, y=_bf16(M, h))
    if kind == "attention":
        cache = _filled_cache(case, seed, _lens(case["batch"], case["capacity"], case["ragged"]))
        B, H = case["batch"], case["heads"]
        return dict(cache=cache, q=_queries(B, H, seed, 1), y=_bf16(B, H, HEAD_DIM),
                    ws=_empty(max(16, N.decode_attention_nvfp4_workspace_size(B, H, case["capacity"]))))
    if kind == "append":
        B, H, T = case["batch"], case["kv_heads"], case["tokens"]
        return dict(cache=_cache(case, B, T + T % 2), k=_kv(B * T, H, seed, 0), v=_kv(B * T, H, seed, 1),
                    shift=torch.randn(H, HEAD_DIM, generator=_gen(seed, 2), device=DEV),
                    seq=torch.arange(B, dtype=torch.int32, device=DEV).repeat_interleave(T),
                    pos=torch.arange(T, dtype=torch.int32, device=DEV).repeat(B), table=_rope_table(T + T % 2))
    if kind == "block":
        return _prepare_block(case, seed)
    return dict(w=_weight(case["rows"], case["cols"], seed, 0), q=_operand(case["rows"], case["cols"], "nvfp4"))


def _cache(case, batch, capacity):
    return N.KVCache(batch, case["kv_heads"], capacity, KV_G, KV_G, device=DEV,
                     kv_format=N.KV_E1M2 if case["kv"] == "e1m2" else N.KV_E2M1)


def _filled_cache(case, seed, lens):
    """A cache whose sequences hold lens tokens each, put there by the append call."""
    cache = _cache(case, case["batch"], case["capacity"])
    for b, n in enumerate(lens):
        k, v = _kv(n, case["kv_heads"], seed, 100 + 2 * b), _kv(n, case["kv_heads"], seed, 101 + 2 * b)
        N.kv_append_nvfp4(cache, k, v, torch.full((n,), b, dtype=torch.int32, device=DEV),
                          torch.arange(n, dtype=torch.int32, device=DEV))
    cache.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
    return cache


def _block_lens(case):
    """Tokens of each sequence after the step: the new one is the last."""
    return _lens(case["batch"], case["capacity"], True)


def _prepare_block(case, seed):
    B, h, H, HK = (case[k] for k in ("batch", "hidden", "heads", "kv_heads"))
    lens = _block_lens(case)
    qkv_n = (H + 2 * HK) * HEAD_DIM
    cache = _filled_cache(case, seed, [max(1, n - 1) for n in lens])
    cache.seq_lens.copy_(torch.tensor(lens, dtype=torch.int32))
    att = _operand(B, H * HEAD_DIM, "nvfp4")
    att["g"].fill_(O_G)
    pos = torch.tensor([n - 1 for n in lens], dtype=torch.int32, device=DEV)
    table = _rope_table(case["capacity"])
    return dict(cache=cache, state=_state_buffer(), x=_activation(B, h, seed, 0), a=_operand(B, h, "nvfp4"), att=att,
                qkv=_bf16(B, qkv_n), y=_bf16(B, h), w_qkv=_quantize_weight(_weight(qkv_n, h, seed, 1), "nvfp4"),
                w_o=_quantize_weight(_weight(h, H * HEAD_DIM, seed, 2), "nvfp4"), table=table, pos=pos,
                cs=table[pos.long()][:, None], seq=torch.arange(B, dtype=torch.int32, device=DEV),
                ws=_empty(max(16, N.decode_attention_nvfp4_workspace_size(B, H, case["capacity"]))))


def _pass(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "dyn":
        w = s["w"]
        N.nvfp4_linear_dynamic(s["x"], w["codes"], w["scales"], w["g"], s["y"], case["N"], g_a=s["g"])
        return dict(out=s["y"], g=s["g"])
    if kind == "linears":
        got = {}
        for t in s["linears"]:
            _quantize(t["x"], t["a"], case["fmt"], s["state"])
            _linear(t["a"], t["w"], t["out"], case["fmt"])
            got[t["name"]] = dict(out=t["out"], codes=t["a"]["codes"], scales=t["a"]["scales"])
        return got
    if kind == "mlp":
        fmt, M = case["fmt"], case["M"]
        _quantize(s["x"], s["a"], fmt, s["state"])
        _swiglu(s["a"], s["gate_up"], M, case["inter"], case["hidden"], s["act"], fmt)
        _linear(s["act"], s["down"], s["y"], fmt)
        return dict(y=s["y"], act_codes=s["act"]["codes"], act_scales=s["act"]["scales"])
    if kind == "attention":
        N.decode_attention_nvfp4(s["cache"], s["q"], SOFTMAX, s["y"], s["ws"])
        return dict(out=s["y"])
    if kind == "append":
        c = s["cache"]
        if case["rope"]:
            N.kv_append_rope_nvfp4(c, s["k"], s["v"], s["seq"], s["pos"], s["table"], k_shift=s["shift"])
        else:
            N.kv_append_nvfp4(c, s["k"], s["v"], s["seq"], s["pos"])
        return dict(k_codes=c.k_codes, k_scales=c.k_scales, v_codes=c.v_codes, v_scales=c.v_scales)
    if kind == "block":
        return _block_pass(s, case)
    q = s["q"]
    N.nvfp4_tensor_scale(s["w"], q["g"])
    N.nvfp4_quantize(s["w"], q["g"], q["codes"], q["scales"])
    return q


def _rope_f32(x, cs):
    c, d, half = cs[..., 0], cs[..., 1], HEAD_DIM // 2
    a, b = x[..., :half].float(), x[..., half:].float()
    return torch.cat([a * c - b * d, a * d + b * c], dim=-1)


def _block_pass(s, case):
    B, H, HK = case["batch"], case["heads"], case["kv_heads"]
    _quantize(s["x"], s["a"], "nvfp4", s["state"])
    _linear(s["a"], s["w_qkv"], s["qkv"], "nvfp4")
    q, k, v = s["qkv"].view(B, H + 2 * HK, HEAD_DIM).split([H, HK, HK], dim=1)
    N.kv_append_rope_nvfp4(s["cache"], k.contiguous(), v.contiguous(), s["seq"], s["pos"], s["table"])
    q = _rope_f32(q, s["cs"]).to(torch.bfloat16)
    N.decode_attention_nvfp4_quantize(s["cache"], q, SOFTMAX, s["att"]["g"], s["att"]["codes"], s["att"]["scales"],
                                      s["ws"])
    _linear(s["att"], s["w_o"], s["y"], "nvfp4")
    return dict(y=s["y"], qkv=s["qkv"])


# ------------------------------------------------------------------- work ---

FP4 = 0.5 + 1 / 16  # bytes of an element: half a byte of code, a scale byte per 16


def work(case):
    kind = case["kind"]
    if kind == "dyn":
        M, Nn, K = case["M"], case["N"], case["K"]
        return dict(bytes=2 * M * K + FP4 * Nn * K + 2 * M * Nn, flops=2 * M * Nn * K)
    if kind == "linears":
        M, ws = case["M"], _weights(case, 0)
        return dict(bytes=sum((2 + FP4) * M * K + FP4 * Nn * K + 2 * M * Nn for _, Nn, K in ws),
                    flops=sum(2 * M * Nn * K for _, Nn, K in ws))
    if kind == "mlp":
        M, h, I = case["M"], case["hidden"], case["inter"]
        return dict(bytes=4 * M * h + FP4 * (3 * h * I + M * I), flops=6 * M * h * I)
    if kind == "attention":
        t = sum(_lens(case["batch"], case["capacity"], case["ragged"]))
        return dict(bytes=2 * t * case["kv_heads"] * HEAD_DIM * FP4 + 4 * case["batch"] * case["heads"] * HEAD_DIM,
                    flops=4 * t * case["heads"] * HEAD_DIM)
    if kind == "append":
        n = case["batch"] * case["tokens"]
        return dict(bytes=2 * n * case["kv_heads"] * HEAD_DIM * (2 + FP4) + (case["tokens"] * 512 if case["rope"] else 0),
                    flops=0)
    if kind == "block":
        B, h, H, HK = (case[k] for k in ("batch", "hidden", "heads", "kv_heads"))
        t, d = sum(_block_lens(case)), HEAD_DIM
        params = h * (2 * H + 2 * HK) * d
        return dict(bytes=FP4 * params + 2 * t * HK * d * FP4 + B * (4 * h + 2 * (H + 2 * HK) * d),
                    flops=2 * B * params + 4 * t * H * d)
    n = case["rows"] * case["cols"]
    return dict(bytes=(2 + FP4) * n, flops=0)


def tolerance(case):
    kind = case["kind"]
    if kind in ("append", "weight"):
        return "exact"
    if kind in ("dyn", "linears"):
        # bf16 outputs of one rounding after a sum in 32 bits: 1.7e-3 from the exact sums.  Codes stay the same.
        return dict(rel=7e-3, max=0.03)
    if kind == "attention":
        # bf16 outputs; weights and the values' products go through 16-bit tensor-core operands.
        return dict(rel=8e-3, max=0.06)
    if kind == "mlp":
        # The activation's codes move where it sits on a rounding edge.
        return dict(rel=1.5e-2, max=0.2, differ=0.01)
    # block: a change of rounding in the attention moves codes of the o projection's input.
    return dict(rel=0.01, max=0.3)


# ------------------------------------------------------- the same in 64 bits ---

E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _e2m1(v):
    """Nearest E2M1 value, ties to the even code, saturating."""
    a = v.abs()
    code = ((a > 0.25).to(torch.uint8) + (a >= 0.75) + (a > 1.25) + (a >= 1.75) + (a > 2.5) + (a >= 3.5) + (a > 5.0))
    return torch.tensor(E2M1, device=v.device)[code.long()] * torch.sign(v)


def _fp4(x, g):
    """NVFP4 values of x along its last axis, without the tensor scale, in 32 bits (exact)."""
    b = x.float().reshape(*x.shape[:-1], -1, 16)
    g = torch.as_tensor(g, dtype=torch.float32, device=x.device)
    s = (b.abs().amax(-1, keepdim=True) / (g * 6.0)).clamp(max=448.0).to(torch.float8_e4m3fn).float()
    m = torch.where(s > 0, torch.reciprocal(s * g), torch.zeros_like(s))
    return (_e2m1(b * m) * s).reshape(x.shape)


def _e1m2(x, g):
    b = x.float().reshape(*x.shape[:-1], -1, 16)
    g = torch.as_tensor(g, dtype=torch.float32, device=x.device)
    s = (b.abs().amax(-1, keepdim=True) / (g * 3.5)).clamp(max=448.0).to(torch.float8_e4m3fn).float()
    m = torch.where(s > 0, torch.reciprocal(s * g), torch.zeros_like(s))
    k = torch.round(b.abs() * m * 2).clamp(max=7.0) * 0.5 * torch.sign(b)
    return (k * s).reshape(x.shape)


def _hadamard32(b):
    for step in (1, 2, 4, 8, 16):
        v = b.reshape(*b.shape[:-1], -1, 2, step)
        b = torch.stack([v[..., 0, :] + v[..., 1, :], v[..., 0, :] - v[..., 1, :]], dim=-2).reshape(b.shape)
    return b * torch.tensor(1 / math.sqrt(32), dtype=torch.float32, device=b.device).to(b.dtype)


def _mx(x, rotate):
    """MXFP4 values of x along its last axis."""
    b = x.float().reshape(*x.shape[:-1], -1, 32)
    if rotate:
        b = _hadamard32(b)
    amax = b.abs().amax(-1, keepdim=True)
    e = torch.where(amax > 0, torch.frexp(amax)[1] - 3, torch.full_like(amax, -127.0).int()).clamp(-127, 127)
    e = torch.ldexp(torch.ones_like(amax, dtype=torch.float64), e)
    return (_e2m1((b.double() / e).float()).double() * e).float().reshape(x.shape)


def _scale(x):
    # A tensor divisor: torch turns a division by a number into a product with its reciprocal.
    return x.float().abs().max() / torch.tensor(2688.0, device=x.device)


def _values(x, fmt, g=None):
    """(values without the tensor scale, tensor scale) of a quantized operand."""
    if fmt == "nvfp4":
        g = _scale(x) if g is None else torch.as_tensor(g, dtype=torch.float32, device=DEV)
        return _fp4(x, g), g
    return _mx(x, fmt == "mxfp4_rot"), torch.ones((), device=DEV)


def _product(a, w, rows=2048):
    """a wT in 64 bits, with the tensor scales' 32-bit product."""
    scale = (a[1] * w[1]).double()
    out = torch.empty(a[0].shape[0], w[0].shape[0], dtype=torch.float64, device=DEV)
    wd = w[0].double()
    for i in range(0, out.shape[0], rows):
        out[i:i + rows] = a[0][i:i + rows].double() @ wd.T
    return out.mul_(scale)


def _attend(q, k, v, k_g, v_g):
    """q [H, 128] over values k, v [T, HK, 128] of one sequence."""
    T, HK, d = k.shape
    kd, vd = k.double().permute(1, 0, 2) * k_g, v.double().permute(1, 0, 2) * v_g
    qd = q.double().view(HK, -1, d)
    p = torch.softmax(qd @ kd.transpose(1, 2) * SOFTMAX, dim=-1)
    return (p @ vd).reshape(-1, d)


def exact(case, seed):
    kind = case["kind"]
    if kind == "dyn":
        M, Nn, K = case["M"], case["N"], case["K"]
        a = _values(_activation(M, K, seed, 0), "nvfp4")
        return dict(out=_product(a, _values(_weight(Nn, K, seed, 1), "nvfp4")), g=None)
    if kind == "linears":
        got = {}
        for i, (name, Nn, K) in enumerate(_weights(case, seed)):
            a = _values(_activation(case["M"], K, seed, 2 * i), case["fmt"])
            w = _values(_weight(Nn, K, seed, 2 * i + 1), case["fmt"])
            got[name] = dict(out=_product(a, w), codes=None, scales=None)
        return got
    if kind == "mlp":
        fmt, h, I = case["fmt"], case["hidden"], case["inter"]
        a = _values(_activation(case["M"], h, seed, 0), fmt)
        y = _mlp(a, [_weight(I, h, seed, 1), _weight(I, h, seed, 2)], _weight(h, I, seed, 3), fmt)
        return dict(y=y, act_codes=None, act_scales=None)
    if kind == "attention":
        B, HK = case["batch"], case["kv_heads"]
        q, g = _queries(B, case["heads"], seed, 1), float(torch.tensor(KV_G))
        enc = _e1m2 if case["kv"] == "e1m2" else _fp4
        out = [_attend(q[b], enc(_kv(n, HK, seed, 100 + 2 * b), g), enc(_kv(n, HK, seed, 101 + 2 * b), g), g, g)
               for b, n in enumerate(_lens(B, case["capacity"], case["ragged"]))]
        return dict(out=torch.stack(out))
    if kind == "block":
        return _exact_block(case, seed)
    return None


def _mlp(a, gate_up, down, fmt):
    g = _scale(torch.stack([w.float().abs().max() for w in gate_up])) if fmt == "nvfp4" else None
    gate, up = (_product(a, _values(w, fmt, g)) for w in gate_up)
    act = _values(gate * torch.sigmoid(gate) * up, fmt, ACT_G)
    return _product(act, _values(down, fmt))


def _exact_block(case, seed):
    B, h, H, HK = (case[k] for k in ("batch", "hidden", "heads", "kv_heads"))
    lens, d, bf = _block_lens(case), HEAD_DIM, torch.bfloat16
    w = lambda rows, cols, i: _values(_weight(rows, cols, seed, i), "nvfp4")  # noqa: E731
    qkv = _product(_values(_activation(B, h, seed, 0), "nvfp4"), w((H + 2 * HK) * d, h, 1))
    q, k, v = qkv.to(bf).view(B, H + 2 * HK, d).split([H, HK, HK], dim=1)
    cs = _rope_table(case["capacity"])[torch.tensor([n - 1 for n in lens], device=DEV)][:, None]
    q, k, g = _rope_f32(q, cs).to(bf), _rope_f32(k, cs), float(torch.tensor(KV_G))
    att = []
    for b, n in enumerate(lens):
        kk = _fp4(torch.cat([_kv(max(1, n - 1), HK, seed, 100 + 2 * b)[:n - 1].float(), k[b:b + 1]]), g)
        vv = _fp4(torch.cat([_kv(max(1, n - 1), HK, seed, 101 + 2 * b)[:n - 1], v[b:b + 1]]), g)
        att.append(_attend(q[b], kk, vv, g, g).reshape(-1))
    o = _product(_values(torch.stack(att).to(bf), "nvfp4", O_G), w(h, H * d, 2))
    return dict(y=o, qkv=qkv)
