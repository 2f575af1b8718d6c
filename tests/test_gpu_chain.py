"""Kernels of consecutive calls overlap their set-up with the kernel before them (programmatic dependent launch).  Whatever
precedes a call on the stream (another kernel, a copy, a fill, an event of another stream), directly or inside a captured
graph, the call sees its finished result: outputs are bit-identical to those of the same call on a quiet GPU."""
import pytest
import torch

from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu
M, N, K = 512, 768, 1024


def _call(kind, x, w_q, out):
    """One public call whose first kernel reads x; returns the tensors to compare."""
    if kind == "bf16":
        B.nvfp4_gemm_bf16(x, x, out["d32"])
        return [out["d32"]]
    if kind == "error":
        return [B.nvfp4_quant_error(x, out["row"], out["sums"]).float()]  # (FP64 atomics: the order varies)
    opts = {"nvfp4": B.quant_opts(rounding=1, rht_colwise=True, rht_sign_mask=synth.DEFAULT_RHT_SIGN_MASK, seed=1),
            "mxfp4": B.quant_opts(rht_colwise=True, rht_sign_mask=0x73E5), "rows": B.quant_opts(),
            "provided": B.quant_opts(flags=B.AMAX_PROVIDED)}[kind]
    t = {"mxfp4": "mx", "rows": "rs"}.get(kind, "")
    row, col = out[t + "row"], None if kind in ("rows", "provided") else out[t + "col"]
    B.nvfp4_quantize(x, opts, row, col)
    res = [row.codes, row.scales, row.glob] + ([col.codes, col.scales, col.glob] if col else [])
    if kind != "mxfp4":
        B.nvfp4_gemm(row, w_q, out["d"])
        res.append(out["d"])
    return res


@pytest.mark.parametrize("before", ["kernel", "copy", "fill", "other stream"])
@pytest.mark.parametrize("kind", ["nvfp4", "mxfp4", "rows", "provided", "bf16", "error"])
def test_a_call_sees_what_precedes_it(kind, before):
    src = torch.randn((M, K), generator=torch.Generator("cuda").manual_seed(1), device="cuda").to(torch.bfloat16)
    w_q = B.alloc_tensor(N, K)
    B.nvfp4_quantize(src[:256].repeat(3, 1).contiguous(), B.quant_opts(), w_q, None)
    out = {"row": B.alloc_tensor(M, K), "col": B.alloc_tensor(K, M),
           "mxrow": B.alloc_tensor(M, K, format=B.FORMAT_MXFP4), "mxcol": B.alloc_tensor(K, M, format=B.FORMAT_MXFP4),
           "rsrow": B.alloc_tensor(M, K, format=B.FORMAT_NVFP4_ROWSCALE),
           "d": torch.empty((M, N), dtype=torch.bfloat16, device="cuda"),
           "d32": torch.empty((M, M), dtype=torch.float32, device="cuda"),
           "sums": torch.empty(2, dtype=torch.float64, device="cuda")}
    B.nvfp4_quantize(src, B.quant_opts(), out["row"], None)
    if kind == "provided":
        out["row"].glob.fill_(8.0)
    big = torch.randn((4096, 4096), device="cuda")
    x, other = torch.empty_like(src), torch.cuda.Stream()

    def produce():  # x = src (or zeros for "fill"), the last operation before the call a slow or non-kernel one
        if before == "fill":
            x.copy_(src)
            x.view(torch.int16).zero_()
        elif before == "other stream":
            other.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(other):
                torch.mm(big, big)
                x.copy_(src)
            torch.cuda.current_stream().wait_stream(other)
        elif before == "copy":
            x.copy_(src)  # same type and shape: a device-to-device copy
        else:
            torch.mm(big, big)
            torch.mul(src, 1.0, out=x)

    produce()
    torch.cuda.synchronize()
    want = [t.clone() for t in _call(kind, x, w_q, out)]
    torch.cuda.synchronize()
    for _ in range(10):
        x.fill_(float("nan"))
        produce()
        for got, ref in zip(_call(kind, x, w_q, out), want):
            assert torch.equal(got, ref)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            produce()
            res = _call(kind, x, w_q, out)
    torch.cuda.synchronize()
    for _ in range(5):
        x.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        for got, ref in zip(res, want):
            assert torch.equal(got, ref)
    B.nvfp4_device_status()


# chunks of 16 a lane keeps: 2 | 2 of two warps | 5 | 5 of two | 5 of four | 10 of four | rows read twice
@pytest.mark.parametrize("cols", [1024, 2048, 2560, 5120, 10240, 20480, 20608])
@pytest.mark.parametrize("rounding", [B.ROUND_NEAREST_EVEN, B.ROUND_STOCHASTIC])
def test_row_scaled_copies_of_any_length_in_a_chain(cols, rounding):
    """The row-scaled quantizer is resident before the kernel that makes its source and the product that reads its last copy have
    finished: the source and the copy are those of a quiet GPU all the same."""
    rows = 128
    src = torch.randn((rows, cols), generator=torch.Generator("cuda").manual_seed(cols), device="cuda").to(torch.bfloat16)
    opts = B.quant_opts(rounding=rounding, seed=7, sr_offset=3)
    layout = B.SF_SWIZZLED if cols % 64 == 0 else B.SF_LINEAR
    want = B.alloc_tensor(rows, cols, layout, format=B.FORMAT_NVFP4_ROWSCALE)
    B.nvfp4_quantize(src, opts, want, None)
    torch.cuda.synchronize()
    x, got = torch.empty_like(src), B.alloc_tensor(rows, cols, layout, format=B.FORMAT_NVFP4_ROWSCALE)
    big = torch.randn((2048, 2048), device="cuda")
    total = torch.zeros(2, dtype=torch.float64, device="cuda")
    for _ in range(10):
        x.fill_(float("nan"))
        torch.mm(big, big)
        torch.mul(src, 1.0, out=x)
        B.nvfp4_quantize(x, opts, got, None)
        first = B.nvfp4_quant_error(x, got, total).clone()  # reads the copy while the next call is resident
        B.nvfp4_quantize(x, opts, got, None)
        for a, b in ((got.codes, want.codes), (got.scales, want.scales), (got.glob, want.glob)):
            assert torch.equal(a, b)
        assert float(first[0]) < 0.02 * float(first[1])


@pytest.mark.parametrize("dim", [2, 8, 128])
@pytest.mark.parametrize("copies", ["both", "row"])
def test_other_transform_sizes_in_a_chain(dim, copies):
    """The same for the kernel of the other transform sizes, which is launched either way (d = 128: by whether the transposed copy is
    asked for)."""
    rows, cols = 384, 640
    src = torch.randn((rows, cols), generator=torch.Generator("cuda").manual_seed(dim), device="cuda").to(torch.bfloat16)
    opts = B.quant_opts(rounding=1, rht_colwise=copies == "both", rht_rowwise=copies == "row", rht_sign_mask=0x73E5, rht_dim=dim, seed=1)

    def quantize(x):
        row, col = B.alloc_tensor(rows, cols), B.alloc_tensor(cols, rows) if copies == "both" else None
        B.nvfp4_quantize(x, opts, row, col)
        return [t for c in (row, col) if c for t in (c.codes, c.scales, c.glob)]

    want = quantize(src)
    torch.cuda.synchronize()
    x, big = torch.empty_like(src), torch.randn((2048, 2048), device="cuda")
    for _ in range(10):
        x.fill_(float("nan"))
        torch.mm(big, big)
        torch.mul(src, 1.0, out=x)
        first, second = quantize(x), quantize(x)
        assert all(torch.equal(a, b) and torch.equal(a, c) for a, b, c in zip(want, first, second))
