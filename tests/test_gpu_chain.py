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
    """Behind kernels of torch's, whose end the quantizer waits for, and before the metric, which reads the copy without a pause: source and
    copy are those of a quiet GPU.  (Copies that are overwritten while a kernel of this library may still read them:
    test_row_scaled_copies_between_products.)"""
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
    """The order of the launches inside a call (words, pass 1, pass 2), behind kernels of torch's and into fresh copies.  (Shared copies:
    test_other_transform_sizes_between_products.)"""
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


def _quantized(rows, cols, seed, scale):
    t = B.alloc_tensor(rows, cols)
    x = torch.randn((rows, cols), generator=torch.Generator("cuda").manual_seed(seed), device="cuda") * scale
    B.nvfp4_quantize(x.to(torch.bfloat16), B.quant_opts(block_rows=16), t, None)
    return t


class _Chain:
    """Two products write D in turn (one in FP4, one in BF16), `quantize` turns D into the shared copies, and a product on each copy
    reads them: every kernel is this library's own and resident before the one before it has finished, D and the copies are
    overwritten while the kernels that read them may still run."""

    def __init__(self, rows, cols, quantize, copies, fp32=False):
        g = torch.Generator("cuda").manual_seed(rows + cols)
        self.a, self.w = _quantized(rows, 256, 1, 1.0), _quantized(cols, 256, 2, 0.1)
        self.x, self.y = (torch.randn((n, 256), generator=g, device="cuda").to(torch.bfloat16) for n in (rows, cols))
        self.D = torch.empty((rows, cols), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
        self.quantize, self.copies = quantize, copies
        # products of 1024 columns, four tiles and more: they leave the GPU's SMs at different times
        self.other = [_quantized(1024, c.cols, 3, 1.0) for c in copies]
        self.out = [[torch.empty((c.rows, 1024), dtype=torch.bfloat16, device="cuda") for c in copies] for _ in range(2)]

    def round(self, i, sync=lambda: None):
        if i == 0:
            B.nvfp4_gemm(self.a, self.w, self.D)
        else:
            B.nvfp4_gemm_bf16(self.x, self.y, self.D)
        sync()
        self.quantize(self.D)
        sync()
        for c, o, e in zip(self.copies, self.other, self.out[i]):
            B.nvfp4_gemm(c, o, e)
            sync()

    def bytes(self):
        return [e.clone() for o in self.out for e in o] + [t.clone() for c in self.copies for t in (c.codes, c.scales, c.glob)]

    def check(self):
        for i in (0, 1):
            self.round(i, torch.cuda.synchronize)
        want = self.bytes()
        assert not torch.equal(self.out[0][0], self.out[1][0])
        for _ in range(5):
            for t in [e for o in self.out for e in o] + [c.codes for c in self.copies]:
                t.zero_()
            self.D.fill_(float("nan"))
            torch.cuda.synchronize()
            for _ in range(2):
                for i in (0, 1):
                    self.round(i)
            assert all(torch.equal(a, b) for a, b in zip(self.bytes(), want))
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.stream(side):
            with torch.cuda.graph(graph, stream=side):
                for i in (0, 1):
                    self.round(i)
        for _ in range(3):
            for o in self.out:
                for e in o:
                    e.zero_()
            graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(self.bytes(), want))
        B.nvfp4_device_status()


# the row lengths of the test above (multiples of 256, as the product on the copy contracts over them)
@pytest.mark.parametrize("cols", [1024, 2048, 2560, 5120, 10240, 20480, 20736])
@pytest.mark.parametrize("rounding", [B.ROUND_NEAREST_EVEN, B.ROUND_STOCHASTIC])
def test_row_scaled_copies_between_products(cols, rounding):
    rows = 256
    copy = B.alloc_tensor(rows, cols, format=B.FORMAT_NVFP4_ROWSCALE)
    opts = B.quant_opts(rounding=rounding, seed=7, sr_offset=3)
    _Chain(rows, cols, lambda x: B.nvfp4_quantize(x, opts, copy, None), [copy]).check()


# 8 tiles, 192 and 396 (one CTA per SM, two, as many as fit)
@pytest.mark.parametrize("rows,cols", [(256, 512), (1536, 2048), (2816, 2304)])
@pytest.mark.parametrize("dim", [4, 128])
@pytest.mark.parametrize("form", ["col", "row", "both rotated", "provided"])
def test_other_transform_sizes_between_products(rows, cols, dim, form):
    """The forms that differ in which of their launches are programmatic: the recipe's two copies, a row-wise one, two transformed ones,
    and two whose amax is provided, so that pass 2 is the call's first kernel."""
    row, col = B.alloc_tensor(rows, cols), B.alloc_tensor(cols, rows)
    kw = dict(rounding=B.ROUND_STOCHASTIC, rht_colwise=form != "row", rht_rowwise=form != "col", rht_sign_mask=0x73E5, rht_dim=dim, seed=1)
    opts = B.quant_opts(flags=B.AMAX_PROVIDED if form == "provided" else 0, **kw)
    for t in (row, col):
        t.glob[0] = 400.0  # (a bound on both products' outputs, and on their transforms')
    copies = [row] if form == "row" else [row, col]
    _Chain(rows, cols, lambda x: B.nvfp4_quantize(x, opts, row, col if form != "row" else None), copies).check()


@pytest.mark.parametrize("rows,cols", [(256, 512), (2816, 2304)])
@pytest.mark.parametrize("provided", [False, True])
def test_binary32_weights_between_products(rows, cols, provided):
    """Pass 1 of a binary32 source, which divides an SM for its loads, and pass 2 as the call's first kernel."""
    row, col = B.alloc_tensor(rows, cols), B.alloc_tensor(cols, rows)
    opts = B.quant_opts(block_rows=16, flags=B.INPUT_FP32 | (B.AMAX_PROVIDED if provided else 0))
    for t in (row, col):
        t.glob[0] = 400.0  # (a bound on both products' outputs)
    _Chain(rows, cols, lambda x: B.nvfp4_quantize(x, opts, row, col), [row, col], fp32=True).check()
