"""Performance cases of the NVFP4 linear-layer path, through the entry points of ``paper_2509_25149_b200.binding``.

A case is a dict of plain values; ``listed()`` names the fixed ones, ``draw()`` gives more of the same ranges.  Kinds:

``layer``     a linear layer, tokens x inp -> tokens x out: the forward call, the backward call or both, in NVFP4, MXFP4
              or BF16, with fresh or cached quantized weights and a written or an accumulated weight gradient;
``gemm``      one block-scaled product of two quantized operands (rows multiples of 128);
``quantize``  one quantizer call: an activation (1x16 blocks, nearest, transformed transposed copy), a gradient (the
              same with stochastic rounding), a weight (square blocks, from bf16 or from the binary32 master copy), or
              a row-wise copy with a scale per row; scale bytes in the GEMM's layout or row by row;
``error``     a quantization-error metric: tensor against its copy, or two dense tensors.
"""
import math

import torch

from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

SIGNS = synth.DEFAULT_RHT_SIGN_MASK
SIGNS32 = 0x1B5D73E5  # 32 sign bits for the MXFP4 transform
FORMATS = {"nvfp4": B.FORMAT_NVFP4, "mxfp4": B.FORMAT_MXFP4}


def listed():
    return [
        # the smallest training step of a layer: launches and latency
        _layer("layer_small", "nvfp4", "both", 512, 1024, 1024),
        # a mid-sized step whose sizes are odd multiples of the layer's granularity of 256
        _layer("layer_odd", "nvfp4", "both", 2816, 3328, 2304),
        # the first microbatch of an optimizer step on a wide layer: the weight changed and is quantized again
        _layer("layer_ffn_up", "nvfp4", "both", 8192, 20480, 5120),
        # a later microbatch: the quantized weight is reused and the FP32 weight gradient is accumulated; the input is
        # the output of a squared ReLU
        _layer("layer_ffn_down_microbatch", "nvfp4", "both", 8192, 5120, 20480, weight="cached", accumulate=True,
               act="relu2"),
        # the same layer in the comparison format
        _layer("layer_mxfp4", "mxfp4", "both", 8192, 7168, 5120),
        # a layer that is kept in BF16, with a ragged batch (multiples of 8)
        _layer("layer_bf16_ragged", "bf16", "both", 4088, 5128, 5112),
        # evaluation of a few tokens against a quantized weight
        _layer("forward_few_tokens", "nvfp4", "forward", 256, 7168, 5120, weight="cached"),
        # evaluation of a long batch, a scale per token
        _layer("forward_row_scales", "nvfp4", "forward", 16384, 5120, 5120, weight="cached", row_scales=True),
        # a product whose row counts are odd multiples of 128
        {"name": "gemm_odd_rows", "kind": "gemm", "fmt": "nvfp4", "m": 4224, "n": 5248, "k": 5120, "fp32": False,
         "accumulate": False},
        # a weight quantized from its binary32 master copy, both orientations
        {"name": "quantize_master_weight", "kind": "quantize", "role": "weight", "fmt": "nvfp4", "rows": 7168,
         "cols": 5120, "fp32": True, "linear": False},
        # a gradient of ragged size (multiples of 16), scale bytes row by row
        {"name": "quantize_gradient_ragged", "kind": "quantize", "role": "gradient", "fmt": "nvfp4", "rows": 5008,
         "cols": 4112, "fp32": False, "linear": True},
        # how well a tensor survives quantization (drives the choice of the layers that stay in BF16)
        {"name": "error_of_copy", "kind": "error", "against": "copy", "rows": 8192, "cols": 5120},
    ]


def _layer(name, fmt, direction, tokens, out, inp, weight="fresh", accumulate=False, row_scales=False, act="normal"):
    case = {"kind": "layer", "fmt": fmt, "pass": direction, "tokens": tokens, "out": out, "inp": inp, "weight": weight,
            "accumulate": accumulate, "row_scales": row_scales, "act": act}
    return dict(case, name=name) if name else case


def _log_size(rng, lo, hi, unit):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / unit)) * unit))


def draw(rng):
    """One more case of the ranges above; no dearer than the largest listed one."""
    most = max(_cost(c) for c in listed())
    while True:
        case = _draw_one(rng)
        if _cost(case) <= most:
            return case


def _draw_one(rng):
    kind = rng.choices(["layer", "gemm", "quantize", "error"], [6, 1.5, 3, 1])[0]
    if kind == "layer":
        fmt = rng.choices(["nvfp4", "mxfp4", "bf16"], [6, 1.5, 1.5])[0]
        unit, least = (8, 264) if fmt == "bf16" else (256, 256)
        tokens = _log_size(rng, least, 16384, unit)
        out, inp = (_log_size(rng, 512, 20480, unit) for _ in range(2))
        direction = rng.choices(["both", "forward", "backward"], [6, 2, 1])[0]
        cached = fmt != "bf16" and direction != "backward" and rng.random() < (0.8 if direction == "forward" else 0.4)
        return _layer(None, fmt, direction, tokens, out, inp, weight="cached" if cached else "fresh",
                      accumulate=direction != "forward" and rng.random() < 0.5,
                      row_scales=fmt == "nvfp4" and direction == "forward" and rng.random() < 0.3,
                      act=rng.choice(["normal", "normal", "relu2"]))
    if kind == "gemm":
        fp32 = rng.random() < 0.4
        return {"kind": "gemm", "fmt": rng.choice(["nvfp4", "nvfp4", "mxfp4"]), "m": _log_size(rng, 128, 16384, 128),
                "n": _log_size(rng, 256, 20480, 128), "k": _log_size(rng, 512, 20480, 256), "fp32": fp32,
                "accumulate": fp32 and rng.random() < 0.5}
    if kind == "quantize":
        role = rng.choice(["activation", "gradient", "weight", "row_scaled"])
        fmt = "mxfp4" if role != "row_scaled" and rng.random() < 0.2 else "nvfp4"
        linear = rng.random() < 0.35
        unit = 128 if not linear else 32 if fmt == "mxfp4" else 16
        return {"kind": "quantize", "role": role, "fmt": fmt, "rows": _log_size(rng, 256, 20480, unit),
                "cols": _log_size(rng, 512, 20480, unit), "fp32": role == "weight" and fmt == "nvfp4" and rng.random() < 0.5,
                "linear": linear}
    return {"kind": "error", "against": rng.choice(["copy", "dense"]), "rows": _log_size(rng, 256, 20480, 16),
            "cols": _log_size(rng, 512, 20480, 16)}


def _cost(case):
    """Rough time of a pass (seconds), to compare cases by."""
    w = work(case)
    return w["bytes"] / 5e12 + w["flops"] / (1.3e15 if case.get("fmt") == "bf16" else 4e15)


# ------------------------------------------------------------------------------------------------- inputs ----
def _activation(shape, seed, act):
    if act == "relu2":
        return synth.squared_relu_bf16_device(shape, seed)
    return synth.normal_with_outliers_bf16_device(shape, 0.001, 100.0, seed)


def prepare(case, seed):
    return {"layer": _prepare_layer, "gemm": _prepare_gemm, "quantize": _prepare_quantize,
            "error": _prepare_error}[case["kind"]](case, 10 * seed)


def _prepare_layer(case, seed):
    M, N, K, fmt = case["tokens"], case["out"], case["inp"], case["fmt"]
    s = {"case": case, "fwd": case["pass"] != "backward", "bwd": case["pass"] != "forward"}
    s["X"] = _activation((M, K), seed + 1, case["act"])
    s["W"] = synth.normal_bf16_device((N, K), 0.02, seed + 2)
    s["Y"] = torch.empty((M, N), dtype=torch.bfloat16, device="cuda") if s["fwd"] else None
    if s["bwd"]:
        s["dY"] = synth.normal_bf16_device((M, N), 1e-4, seed + 3)
        s["dX"] = torch.empty((M, K), dtype=torch.bfloat16, device="cuda")
        s["dW"] = torch.zeros((N, K), dtype=torch.float32, device="cuda")
    if fmt == "bf16":
        return s
    f = FORMATS[fmt]
    flags = B.LINEAR_ROW_SCALES if case["row_scales"] else 0
    s["opts"] = B.quant_opts(rht_sign_mask=SIGNS32 if fmt == "mxfp4" else SIGNS, seed=seed, sr_offset=1, flags=flags)
    s["W_row"] = B.alloc_tensor(N, K, format=f)
    s["W_col"] = B.alloc_tensor(K, N, format=f) if s["bwd"] else None
    s["X_col"] = B.alloc_tensor(K, M, format=f) if s["bwd"] else None
    s["ws_fwd"] = torch.empty(B.nvfp4_linear_fwd_workspace_bytes(M, K), dtype=torch.uint8, device="cuda")
    if s["bwd"]:
        s["ws_bwd"] = torch.empty(B.nvfp4_linear_bwd_workspace_bytes(M, N), dtype=torch.uint8, device="cuda")
    if case["weight"] == "cached" or not s["fwd"]:
        B.nvfp4_quantize(s["W"], B.quant_opts(block_rows=32 if fmt == "mxfp4" else 16), s["W_row"], s["W_col"])
    if not s["fwd"]:
        B.nvfp4_quantize(s["X"], B.quant_opts(rht_colwise=True, rht_sign_mask=s["opts"].rht_sign_mask), None, s["X_col"])
    return s


def _prepare_gemm(case, seed):
    M, N, K, f = case["m"], case["n"], case["k"], FORMATS[case["fmt"]]
    s = {"case": case, "A": B.alloc_tensor(M, K, format=f), "B": B.alloc_tensor(N, K, format=f)}
    B.nvfp4_quantize(_activation((M, K), seed + 1, "normal"), B.quant_opts(), s["A"], None)
    B.nvfp4_quantize(synth.normal_bf16_device((N, K), 0.02, seed + 2),
                     B.quant_opts(block_rows=32 if case["fmt"] == "mxfp4" else 16), s["B"], None)
    s["D"] = torch.zeros((M, N), dtype=torch.float32 if case["fp32"] else torch.bfloat16, device="cuda")
    return s


def _prepare_quantize(case, seed):
    R, C, fmt, role = case["rows"], case["cols"], case["fmt"], case["role"]
    layout = B.SF_LINEAR if case["linear"] else B.SF_SWIZZLED
    f = B.FORMAT_NVFP4_ROWSCALE if role == "row_scaled" else FORMATS[fmt]
    if role == "weight":
        x = (torch.randn((R, C), generator=torch.Generator("cuda").manual_seed(seed + 2), device="cuda").mul_(0.02)
             if case["fp32"] else synth.normal_bf16_device((R, C), 0.02, seed + 2))
        opts = B.quant_opts(block_rows=32 if fmt == "mxfp4" else 16, flags=B.INPUT_FP32 if case["fp32"] else 0)
    else:
        x = (synth.normal_bf16_device((R, C), 1e-4, seed + 3) if role == "gradient"
             else _activation((R, C), seed + 1, "normal"))
        opts = B.quant_opts(rounding=B.ROUND_STOCHASTIC if role == "gradient" else B.ROUND_NEAREST_EVEN,
                            rht_colwise=role != "row_scaled", rht_sign_mask=SIGNS32 if fmt == "mxfp4" else SIGNS,
                            seed=seed, sr_offset=1)
    return {"case": case, "x": x, "opts": opts, "row": B.alloc_tensor(R, C, layout, format=f),
            "col": None if role == "row_scaled" else B.alloc_tensor(C, R, layout, format=f)}


def _prepare_error(case, seed):
    R, C = case["rows"], case["cols"]
    s = {"case": case, "out": torch.empty(2, dtype=torch.float64, device="cuda")}
    if case["against"] == "copy":
        s["x"] = _activation((R, C), seed + 1, "normal")
        s["q"] = B.alloc_tensor(R, C, B.SF_SWIZZLED if R % 128 == 0 and C % 64 == 0 else B.SF_LINEAR)
        B.nvfp4_quantize(s["x"], B.quant_opts(), s["q"], None)
    else:  # two weight gradients of one layer, FP32
        g = torch.Generator("cuda").manual_seed(seed + 4)
        s["x"] = torch.randn((R, C), generator=g, device="cuda")
        s["q"] = s["x"] + 0.1 * torch.randn((R, C), generator=g, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------ one pass ----
def _buffers(t):
    return None if t is None else {"codes": t.codes, "scales": t.scales, "glob": t.glob}


def run(s):
    case = s["case"]
    if case["kind"] == "layer":
        return _run_layer(s, case)
    if case["kind"] == "gemm":
        B.nvfp4_gemm(s["A"], s["B"], s["D"], accumulate=case["accumulate"])
        return s["D"]
    if case["kind"] == "quantize":
        B.nvfp4_quantize(s["x"], s["opts"], s["row"], s["col"])
        return {"row": _buffers(s["row"]), "col": _buffers(s["col"])}
    if case["against"] == "copy":
        return B.nvfp4_quant_error(s["x"], s["q"], s["out"])
    return B.nvfp4_sq_error(s["x"], s["q"], s["out"])


def _run_layer(s, case):
    out = {}
    if case["fmt"] == "bf16":
        if s["fwd"]:
            B.nvfp4_linear_bf16_fwd(s["X"], s["W"], s["Y"])
            out["Y"] = s["Y"]
        if s["bwd"]:
            B.nvfp4_linear_bf16_bwd(s["dY"], s["X"], s["W"], case["inp"], s["dX"], s["dW"], case["accumulate"])
            out["dX"], out["dW"] = s["dX"], s["dW"]
        return out
    if s["fwd"]:
        cached = case["weight"] == "cached"
        B.nvfp4_linear_fwd(s["X"], None if cached else s["W"], s["opts"], s["Y"], s["X_col"], s["W_row"],
                           None if cached else s["W_col"], cached, s["ws_fwd"])
        out["Y"], out["X_col"] = s["Y"], _buffers(s["X_col"])
        if not cached:
            out["W_row"], out["W_col"] = _buffers(s["W_row"]), _buffers(s["W_col"])
    if s["bwd"]:
        B.nvfp4_linear_bwd(s["dY"], s["X_col"], s["W_col"], case["inp"], s["opts"], s["dX"], s["dW"], case["accumulate"],
                           s["ws_bwd"])
        out["dX"], out["dW"] = s["dX"], s["dW"]
    return out


# -------------------------------------------------------------------------------------- work and tolerance ----
def _copy_bytes(fmt, n):
    return n * (0.5 + (1 / 32 if fmt == "mxfp4" else 1 / 16))


def work(case):
    """Each input read once, each output written once; operand copies that live only inside a call are not counted."""
    if case["kind"] == "layer":
        M, N, K, fmt = case["tokens"], case["out"], case["inp"], case["fmt"]
        fwd, bwd = case["pass"] != "backward", case["pass"] != "forward"
        dW = 4 * N * K * (2 if case["accumulate"] else 1)
        flops = 2 * M * N * K * (fwd + 2 * bwd)
        if fmt == "bf16":
            b = 2 * (M * K + N * K + M * N) * fwd
            b += (2 * (M * N + M * K) + dW + (0 if fwd else 2 * (M * K + N * K))) * bwd
            return {"bytes": b, "flops": flops}
        b = 0
        if fwd:
            b += 2 * M * K + 2 * M * N + (_copy_bytes(fmt, M * K) if bwd else 0)
            b += _copy_bytes(fmt, N * K) if case["weight"] == "cached" else 2 * N * K + _copy_bytes(fmt, N * K) * (1 + bwd)
        if bwd:
            b += 2 * M * N + 2 * M * K + dW
            b += _copy_bytes(fmt, N * K) if not fwd or case["weight"] == "cached" else 0
            b += 0 if fwd else _copy_bytes(fmt, M * K)
        return {"bytes": b, "flops": flops}
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        d = m * n * (4 if case["fp32"] else 2) * (2 if case["accumulate"] else 1)
        return {"bytes": _copy_bytes(case["fmt"], (m + n) * k) + d, "flops": 2 * m * n * k}
    n = case["rows"] * case["cols"]
    if case["kind"] == "quantize":
        copies = 1 if case["role"] == "row_scaled" else 2
        return {"bytes": n * (4 if case["fp32"] else 2) + copies * _copy_bytes(case["fmt"], n), "flops": 0}
    return {"bytes": 2 * n + _copy_bytes("nvfp4", n) if case["against"] == "copy" else 8 * n, "flops": 0}


def tolerance(case):
    """Sums in another order, at the same precision; each figure is about four times what was measured.

    Block-scaled products against the binary64 product of the decoded operands: 5e-8 (FP32 result), and 1.2e-5 for a
    bf16 result against the rounded one: a sum that moves by one FP32 rounding can fall on the other side of a bf16
    boundary, one unit in the last place (2^-7 at the bottom of a binade).  BF16 layer: 1.7e-4, the same unit.
    Codes and scale bytes of a transformed copy: its 16 (32) terms are summed in FP32, and about one value in ten million
    lies so near a threshold that another order gives the neighbouring code; a weight gradient sees such a code as 2e-4
    at most.  Everything else that is quantized is exact.  Error metrics: FP32 over 16 elements, 5e-9 over a tensor of
    4e7 elements, more over a small one.
    """
    if case["kind"] == "error":
        return {"rel": 2e-7}
    if case["kind"] == "quantize":
        return "exact" if case["role"] in ("weight", "row_scaled") else {"rel": 5e-7, "differ": 2e-5}
    if case["kind"] == "gemm":
        return {"rel": 2e-7, "max": 1e-5} if case["fp32"] else {"rel": 5e-5, "max": 0.016}
    return {"rel": 7e-4 if case["fmt"] == "bf16" else 2e-4, "max": 0.016, "differ": 2e-5}
