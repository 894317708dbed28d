"""The calls that users of the quantized linear layer make, over the sizes that
they make them with, for timing and for comparing results.

Every case goes through the package's public entry points (``qlin``, the
translator MLP and the linear stack) with the buffers a program keeps across
calls: quantized weights, output buffers and the workspace are made once by
``prepare``; a pass quantizes its bf16 activations and runs its linears.

Sizes come from the package's own workloads (a 1024 x 1024 image's 4096 image
plus 512 text tokens, hidden width 3072, MLP width 12288, the translator's
1024 / 2560 / 3072 widths and 512 tokens) and from the ragged shapes of its
tests; drawn cases spread over the same ranges.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2609_21849_gb300 import qlin, stack, synthetic, translator

HIDDEN, MLP, TOKENS = synthetic.HIDDEN, synthetic.MLP, synthetic.M_TOKENS


# ---------------------------------------------------------------- the cases ---

def listed():
    return [
        # the smallest linear: a 128-token NVFP4 layer, where the launches and
        # the host path are all there is
        _case("tiny_nvfp4_linear", "linear", fmt="nvfp4", M=128, N=256, K=256),
        # the translator's second linear (long K, few tiles) as one call
        _case("translator_linear_nvfp4", "linear", fmt="nvfp4", M=512, N=1024, K=2560),
        # the translator MLP of a 512-token prompt: once per edit, latency
        # bound; captured as a CUDA graph, as an interactive program does
        _case("translator_mlp_nvfp4_graph", "translator", fmt="nvfp4", M=512, graph=True),
        # the same forward in FP8, called eagerly
        _case("translator_mlp_fp8", "translator", fmt="fp8", M=512, graph=False),
        # a ragged FP8 linear whose epilogue writes a column window of the
        # next layer's input (a prompt's odd token count)
        _case("ragged_fp8_fused_window", "fused", fmt="fp8", M=1333, N=2112, K=1088,
              rq_col0=704, rq_cols=1408),
        # the denoiser's hidden-size linear in FP8 (W8A8, dynamic scale)
        _case("denoise_fp8_linear", "linear", fmt="fp8", M=TOKENS, N=HIDDEN, K=HIDDEN),
        # the MLP up-projection in NVFP4 with its re-quantizing epilogue
        # (dynamic input scale): the benchmark's step
        _case("mlp_up_nvfp4_fused", "fused", fmt="nvfp4", M=TOKENS, N=MLP, K=HIDDEN,
              rq_col0=0, rq_cols=MLP),
        # a linear whose output takes its own dynamic scale: the QKV
        # projection in a chain without calibration
        _case("qkv_nvfp4_dynamic_chain", "chain", fmt="nvfp4", M=TOKENS, N=3 * HIDDEN, K=HIDDEN),
        # the unquantized bf16 linear on the value columns of a QKV output
        # (strided rows), the reference precision of the ladder
        _case("out_proj_bf16_strided", "float16", fmt="bf16", M=TOKENS, N=HIDDEN, K=HIDDEN, lda=3),
        # activation quantization alone at batch 4: the static (calibrated)
        # NVFP4 scale and the dynamic FP8 one
        _case("quantize_act_nvfp4_static_b4", "quantize", fmt="nvfp4", M=4 * TOKENS, K=HIDDEN,
              static=True),
        _case("quantize_act_fp8_dynamic_b4", "quantize", fmt="fp8", M=4 * TOKENS, K=HIDDEN,
              static=False),
        # one block's MLP (up, down) of the denoise-step stack at batch 4,
        # chained by the fused re-quantization: the largest call
        _case("mlp_stack_nvfp4_b4", "stack", fmt="nvfp4", B=4),
    ]


def _case(name, kind, **kw):
    return {"name": name, "kind": kind, **kw}


def _log_int(rng, lo, hi, multiple=1):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "fused", "fused", "chain", "float16",
                       "quantize", "quantize", "weight", "translator", "stack"])
    most = TOKENS * MLP * HIDDEN          # multiply-adds of one drawn linear
    if kind == "translator":
        return {"kind": kind, "fmt": rng.choice(["nvfp4", "fp8"]), "M": _log_int(rng, 16, 2048),
                "graph": rng.random() < 0.5}
    if kind == "stack":
        return {"kind": kind, "fmt": "nvfp4", "B": rng.choice([1, 2, 3])}
    M = _log_int(rng, 16, 4 * TOKENS)
    K = _log_int(rng, 64, MLP, 64)
    if kind in ("quantize", "weight"):
        if M * K > 4 * TOKENS * HIDDEN:
            M = max(1, 4 * TOKENS * HIDDEN // K)
        c = {"kind": kind, "fmt": rng.choice(["nvfp4", "fp8"]), "M": M, "K": K}
        return c if kind == "weight" else {**c, "static": rng.random() < 0.5}
    N = _log_int(rng, 64, MLP, 64)
    if M * N * K > most:
        M = max(1, most // (N * K))
    if kind == "float16":
        if M * N * K > most // 4:
            M = max(1, most // 4 // (N * K))
        return {"kind": kind, "fmt": rng.choice(["bf16", "fp16"]), "M": M, "N": N, "K": K,
                "lda": rng.choice([1, 3])}
    c = {"kind": kind, "fmt": "nvfp4" if kind == "chain" else rng.choice(["nvfp4", "fp8"]),
         "M": M, "N": N, "K": K}
    if kind == "fused":
        c["rq_col0"] = 64 * rng.randrange(0, N // 64)
        c["rq_cols"] = N - c["rq_col0"] if rng.random() < 0.5 else 64 * rng.randrange(
            1, (N - c["rq_col0"]) // 64 + 1)
    return c


# --------------------------------------------------------------- the inputs ---

def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + stream * 7919 + 17) % (1 << 62))


def _normal(seed, stream, rows, cols, sigma=1.0):
    x = torch.randn(rows, cols, generator=_gen(seed, stream), device="cuda", dtype=torch.float32)
    return x.mul_(sigma)


def _activations(case, seed, M, K):
    """N(0, 1) with the structure that the path meets: 1% of entries x20
    (NVFP4 linears), log-normal channel gains (FP8 linears), 1% of channels
    x20 (the stack), plain N(0, 1) (translator, 16-bit)."""
    x = _normal(seed, 1, M, K)
    if case["kind"] in ("translator", "float16"):
        return x
    g = _gen(seed, 2)
    if case["kind"] == "stack":
        ch = torch.randperm(K, generator=g, device="cuda")[:round(0.01 * K)]
        x[:, ch] *= 20.0
    elif case["fmt"] == "fp8":
        x *= torch.randn(K, generator=g, device="cuda").exp()
    else:
        x[torch.rand(M, K, generator=g, device="cuda") < 0.01] *= 20.0
    return x


def _shapes(case):
    """[(N, K)] of the case's weights, and their sigma."""
    if case["kind"] == "translator":
        h = synthetic.TRANSLATOR_HIDDEN
        return [(h, synthetic.TRANSLATOR_IN), (synthetic.TRANSLATOR_OUT, h)], 0.03
    if case["kind"] == "stack":
        return [(MLP, HIDDEN), (HIDDEN, MLP)], 0.02
    if case["kind"] == "weight":
        return [(case["M"], case["K"])], 0.02
    return [(case["N"], case["K"])], 0.02


def _inputs(case, seed):
    """The case's 16-bit activations (None for weight quantization) and
    weights."""
    dt = torch.float16 if case["fmt"] == "fp16" else torch.bfloat16
    x = None
    if case["kind"] != "weight":
        M = TOKENS * case["B"] if case["kind"] == "stack" else case["M"]
        K = {"stack": HIDDEN, "translator": synthetic.TRANSLATOR_IN}.get(case["kind"]) or case["K"]
        if case["kind"] == "float16":
            x = _activations(case, seed, M, case["lda"] * K).to(dt)[:, (case["lda"] - 1) * K:]
        else:
            x = _activations(case, seed, M, K).to(dt)
    if case["kind"] == "quantize":
        return x, []
    shapes, sigma = _shapes(case)
    return x, [_normal(seed, 10 + i, n, k, sigma).to(dt) for i, (n, k) in enumerate(shapes)]


def _sigma_x(case):
    """Standard deviation of the activations (1% of entries or channels x20)."""
    return 1.0 if case["kind"] == "translator" else math.sqrt(0.99 + 0.01 * 400.0)


def _next_scales(case):
    """Static decode scales of the re-quantized outputs, as a calibration
    pass would give them: six standard deviations over the format's range."""
    top = 448.0 * 6.0 if case["fmt"] == "nvfp4" else 448.0
    s, out = _sigma_x(case), []
    if case["fmt"] == "fp8" and case["kind"] == "fused":
        s = math.exp(1.0)                  # log-normal channel gains
    for (_, k) in _shapes(case)[0]:
        s = s * _shapes(case)[1] * math.sqrt(k)
        out.append(float(np.float32(6.0 * s / top)))
    return out


def _static_scale(case):
    top = 448.0 * 6.0 if case["fmt"] == "nvfp4" else 448.0
    return float(np.float32((80.0 if case["fmt"] == "nvfp4" else 40.0) / top))


def _scalar(v):
    return torch.tensor([v], dtype=torch.float32, device="cuda")


def _alloc(fmt, rows, K, per_channel=False):
    return qlin.alloc_nvfp4(rows, K) if fmt == "nvfp4" else qlin.alloc_fp8(rows, K, per_channel)


def _bits(w):
    return w.view(torch.int16).cpu().numpy().view(np.uint16)


# ---------------------------------------------------------------- the calls ---

def prepare(case, seed):
    kind, fmt = case["kind"], case["fmt"]
    x, ws = _inputs(case, seed)
    s = SimpleNamespace(case=case, x=x, workspace=qlin.alloc_workspace(), graph=None)
    code = qlin.QLIN_FMT_NVFP4 if fmt == "nvfp4" else qlin.QLIN_FMT_FP8
    if kind == "translator":
        s.mlp = translator.build_translator(fmt, _bits(ws[0]), _bits(ws[1]), case["M"])
        s.mlp.set_hidden_scale(_next_scales(case)[0])
        if case["graph"]:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                s.mlp.forward(x)
            torch.cuda.current_stream().wait_stream(side)
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s.graph):
                s.mlp.forward(x)
        return s
    if kind == "stack":
        s.stack = stack.build_stack(case["B"], weights=[(0, n, _bits(w)) for n, w in zip(("up", "down"), ws)])
        s.stack.set_next_scales(_next_scales(case))
        return s
    if kind == "weight":
        s.w = ws[0]
        s.out = _alloc(fmt, case["M"], case["K"], per_channel=True)
        return s
    M, K = x.shape
    if kind == "quantize":
        s.static = _scalar(_static_scale(case)) if case["static"] else None
        s.out = _alloc(fmt, M, K)
        return s
    N = case["N"]
    if kind == "float16":
        s.w = ws[0]
        s.y = torch.empty((M, N), dtype=x.dtype, device="cuda")
        return s
    s.W = qlin.qlin_quantize_weight(ws[0], code, workspace=s.workspace)
    s.x_q = _alloc(fmt, M, K)
    s.y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    if kind == "fused":
        s.next_scale = _scalar(_next_scales(case)[0])
        s.y_q = _alloc(fmt, M, case["rq_cols"])
    elif kind == "chain":
        s.y_q = _alloc(fmt, M, N)
    return s


def _quantize(s, fmt):
    if fmt == "nvfp4":
        return qlin.qlin_quantize_act_nvfp4(s.x, None, s.x_q, s.workspace)
    return qlin.qlin_quantize_act_fp8(s.x, None, s.x_q, s.workspace)


def _parts(q):
    if isinstance(q, qlin.NVFP4Tensor):
        return [q.codes, q.scales, q.tensor_scale]
    return [q.codes, q.scale]


def run(s):
    case = s.case
    kind, fmt = case["kind"], case["fmt"]
    if kind == "linear":
        a = _quantize(s, fmt)
        (qlin.qlin_gemm_nvfp4 if fmt == "nvfp4" else qlin.qlin_gemm_fp8)(a, s.W, s.y)
        return {"y": s.y, "x_q": _parts(a)}
    if kind == "fused":
        a = _quantize(s, fmt)
        (qlin.qlin_linear_fused if fmt == "nvfp4" else qlin.qlin_linear_fused_fp8)(
            a, s.W, s.y, s.next_scale, s.y_q, case["rq_col0"])
        return {"y": s.y, "x_q": _parts(a), "y_q": _parts(s.y_q)}
    if kind == "chain":
        a = _quantize(s, fmt)
        qlin.qlin_linear_dynamic(a, s.W, s.y, s.y_q, s.workspace)
        return {"y": s.y, "x_q": _parts(a), "y_q": _parts(s.y_q)}
    if kind == "float16":
        (qlin.qlin_gemm_bf16 if fmt == "bf16" else qlin.qlin_gemm_fp16)(s.x, s.w, s.y)
        return {"y": s.y}
    if kind == "quantize":
        if fmt == "nvfp4":
            qlin.qlin_quantize_act_nvfp4(s.x, s.static, s.out, s.workspace)
        else:
            qlin.qlin_quantize_act_fp8(s.x, s.static, s.out, s.workspace)
        return {"x_q": _parts(s.out)}
    if kind == "weight":
        code = qlin.QLIN_FMT_NVFP4 if fmt == "nvfp4" else qlin.QLIN_FMT_FP8
        qlin.qlin_quantize_weight(s.w, code, s.out, s.workspace)
        return {"x_q": _parts(s.out)}
    if kind == "translator":
        if s.graph is not None:
            s.graph.replay()
        else:
            s.mlp.forward(s.x)
        return {"y": s.mlp.y, "x_q": _parts(s.mlp.x_q), "y_q": _parts(s.mlp.h_q)}
    s.stack.forward(s.x)
    up, down = s.stack.layers
    return {"y": down.y, "h": up.y, "x_q": _parts(s.stack.a0), "y_q": _parts(up.out_q),
            "z_q": _parts(down.out_q)}


# ----------------------------------------------------------- what it stands for ---

def _q_bytes(fmt, rows, K):
    return rows * K * 9 / 16 if fmt == "nvfp4" else rows * K


def work(case):
    kind, fmt = case["kind"], case["fmt"]
    if kind in ("quantize", "weight"):
        n = case["M"] * case["K"]
        return {"bytes": 2 * n + _q_bytes(fmt, case["M"], case["K"]), "flops": 0}
    M = TOKENS * case["B"] if kind == "stack" else case["M"]
    shapes = _shapes(case)[0]
    flops = sum(2 * M * n * k for n, k in shapes)
    if kind == "float16":
        N, K = shapes[0]
        return {"bytes": 2 * (M * K + N * K + M * N), "flops": flops}
    K = shapes[0][1]
    b = 2 * M * K + _q_bytes(fmt, M, K) + sum(_q_bytes(fmt, n, k) for n, k in shapes)
    if kind == "translator":      # the hidden activations are written only quantized
        b += _q_bytes(fmt, M, shapes[0][0]) + 2 * M * shapes[1][0]
    elif kind == "stack":
        b += sum(2 * M * n + _q_bytes(fmt, M, n) for n, _ in shapes)
    else:
        b += 2 * M * shapes[0][0]
        if kind == "fused":
            b += _q_bytes(fmt, M, case["rq_cols"])
        elif kind == "chain":
            b += _q_bytes(fmt, M, case["N"])
    return {"bytes": b, "flops": flops}


def tolerance(case):
    """Codes and scales of the inputs are defined bit by bit.  A 16-bit output
    is the rounding of an fp32 sum: it is within half a unit of the last place
    of the exact product (relative 2-norm 1.7e-3 for bf16, 2.1e-4 for fp16),
    and two orders of summation differ in a few roundings (against the exact
    product rounded to bf16, 1e-5 of one layer's outputs and 3e-4 of two
    chained layers' measured different)."""
    kind = case["kind"]
    if kind in ("quantize", "weight"):
        return "exact"
    if kind == "float16":
        return {"rel": 8e-4 if case["fmt"] == "fp16" else 6e-3, "max": 3e-2}
    if kind in ("translator", "stack"):
        # the second layer's input codes may differ where a rounding of the
        # first layer's output does
        return {"rel": 7e-3, "max": 0.1, "differ": 2e-3}
    return {"rel": 6e-3, "max": 3e-2, "differ": 1e-3}


# ------------------------------------------------------------------ in 64 bits ---

_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _div(a, b):
    """fp32 quotient, rounded once (a Python divisor would become a product
    with its reciprocal)."""
    return torch.div(a, torch.full((1,), b, dtype=torch.float32, device="cuda"))


def _encode_scale(s_dec):
    s = torch.ones_like(s_dec) / s_dec
    return torch.where(torch.isinf(s), torch.full_like(s, torch.finfo(torch.float32).max), s)


def _tensor_scale(x, top, static):
    if static is not None:
        return _scalar(static)[0]
    amax = x.abs().amax().float()
    return torch.where(amax == 0, torch.ones_like(amax), _div(amax, top)[0])


def _nvfp4(x, static=None):
    """(decoded NVFP4 of x in 64 bits, S_dec): every fp32 operation of the
    format's definition rounded once."""
    rows, K = x.shape
    s_dec = _tensor_scale(x, 2688.0, static)
    s_enc = _encode_scale(s_dec)
    xb = x.float().view(rows, K // 16, 16)
    t = _div(xb.abs().amax(2) * s_enc, 6.0)
    sb = t.clamp(max=448.0).to(torch.float8_e4m3fn).float()
    r = torch.where(sb == 0, torch.zeros_like(sb), s_enc / sb)
    v = xb * r[:, :, None]
    a = v.abs()
    i = torch.zeros_like(a, dtype=torch.int32)
    # midpoints go to the even code
    for mid, even in ((0.25, 0), (0.75, 1), (1.25, 0), (1.75, 1), (2.5, 0), (3.5, 1), (5.0, 0)):
        i += (a >= mid) if even else (a > mid)
    e = torch.tensor(_E2M1, device="cuda", dtype=torch.float64)[i] * torch.sign(v).double()
    return (e * (sb.double() * s_dec.double())[:, :, None]).view(rows, K), s_dec


def _fp8(x, static=None):
    s_dec = _tensor_scale(x, 448.0, static)
    c = (x.float() * _encode_scale(s_dec)).clamp(-448.0, 448.0).to(torch.float8_e4m3fn)
    return c.double() * s_dec.double(), s_dec


def _fp8_rows(w):
    amax = w.float().abs().amax(1)
    s = torch.where(amax == 0, torch.ones_like(amax), _div(amax, 448.0))
    c = (w.float() * _encode_scale(s)[:, None]).clamp(-448.0, 448.0).to(torch.float8_e4m3fn)
    return c.double() * s.double()[:, None], s


def exact(case, seed):
    kind, fmt = case["kind"], case["fmt"]
    x, ws = _inputs(case, seed)
    quant = _nvfp4 if fmt == "nvfp4" else _fp8

    def scales(s):      # the place of an operand's scale among its parts
        s = s.double().view(-1)
        return [None, None, s] if fmt == "nvfp4" else [None, s]

    if kind == "float16":
        return {"y": x.double() @ ws[0].double().t()}
    if kind == "quantize":
        return {"x_q": scales(quant(x, _static_scale(case) if case["static"] else None)[1])}
    if kind == "weight":
        return {"x_q": scales(quant(ws[0])[1] if fmt == "nvfp4" else _fp8_rows(ws[0])[1])}
    wq = [(quant(w) if fmt == "nvfp4" else _fp8_rows(w))[0] for w in ws]
    a, s_x = quant(x)
    y = a @ wq[0].t()
    out = {"y": y, "x_q": scales(s_x)}
    if kind == "linear":
        return out
    if kind == "chain":
        return {**out, "y_q": scales(quant(y.bfloat16())[1])}
    nxt = _next_scales(case)
    out["y_q"] = scales(_scalar(nxt[0]))
    if kind == "fused":
        return out
    # two chained linears: the second takes the re-quantized bf16 output
    out["y"] = quant(y.bfloat16(), nxt[0])[0] @ wq[1].t()
    if kind == "stack":
        out["h"] = y
        out["z_q"] = scales(_scalar(nxt[1]))
    return out
