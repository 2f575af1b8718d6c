"""Quantizers and error metrics where a size meets the edge of a launch rule: every way a row is kept, every alignment of the
row-by-row scale bytes and of the transposed copy's rows, sums over a few elements."""
import numpy as np
import pytest
import torch

import oracle
import parity as P
from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rounding", [oracle.RNE, oracle.SR])
@pytest.mark.parametrize("cols", [16, 1024, 1040, 2048, 2064, 2560, 2576, 5120, 5136, 10240, 10256, 20480, 20496])
def test_every_way_a_row_is_kept(cols, rounding):
    """Row lengths on both sides of each limit of the row-scaled launch rule (1 / 2 / 4 warps, 2 / 5 / 10 chunks a lane)."""
    rows = 48
    x = synth.normal_with_outliers_bf16((rows, cols), 0.01, 50.0, cols, cols + 1)
    got = B.alloc_tensor(rows, cols, B.SF_LINEAR, format=B.FORMAT_NVFP4_ROWSCALE)
    B.nvfp4_quantize(x.cuda(), B.quant_opts(rounding=rounding, seed=9, sr_offset=2), got)
    want = oracle.quantize_rowscale(synth.bits(x), rounding=rounding, seed=9, sr_offset=2)
    assert np.array_equal(got.codes.cpu().numpy(), want.codes)
    assert np.array_equal(got.scales.cpu().numpy().reshape(rows, -1), want.scales)
    assert np.array_equal(got.glob.cpu().numpy().reshape(rows, 2), want.glob)


@pytest.mark.parametrize("shape", [(16, 16), (32, 272), (144, 256), (272, 144), (256, 192), (304, 2064), (2064, 304), (288, 1120)])
@pytest.mark.parametrize("block_rows", [1, 16])
@pytest.mark.parametrize("fp32", [False, True])
def test_scale_bytes_row_by_row(shape, block_rows, fp32):
    """Rows of 1, 2, 4 and odd numbers of scale bytes, tiles inside and across the edge, rows = 16 and 0 modulo 32."""
    x = synth.normal_with_outliers_bf16(shape, 0.01, 50.0, shape[0], shape[1])
    R, C = shape
    # a frame of canary bytes around the scales: nothing outside may be written
    row, col = B.alloc_tensor(R, C, B.SF_LINEAR), B.alloc_tensor(C, R, B.SF_LINEAR)
    frames = []
    for t in (row, col):
        n = t.scales.numel()
        frames.append(torch.full((n + 64,), 0xA5, dtype=torch.uint8, device="cuda"))
        t.scales = frames[-1][32:32 + n]
    B.nvfp4_quantize(x.float().cuda() if fp32 else x.cuda(), B.quant_opts(block_rows=block_rows), row, col)
    P.assert_exact(row, oracle.quantize(synth.bits(x), block_rows=block_rows), "row")
    P.assert_exact(col, oracle.quantize(synth.bits(x), block_rows=block_rows, colwise=True), "col")
    for f in frames:
        assert bool((f[:32] == 0xA5).all()) and bool((f[-32:] == 0xA5).all())


@pytest.mark.parametrize("shape", [(16, 16), (48, 208), (128, 64), (1040, 2064), (2064, 5136)])
@pytest.mark.parametrize("what", ["nvfp4", "mxfp4", "rows", "dense"])
def test_error_sums(shape, what):
    """FP32 over at most 16 elements, FP64 above: the bound is sixteen roundings of a sum of that size."""
    R, C = shape
    x = synth.normal_with_outliers_bf16((R, C), 0.01, 50.0, R, C).cuda()
    if what == "dense":
        y = x.float() * 1.03125 + 0.01
        got, d = B.nvfp4_sq_error(x, y), x.double() - y.double()
    else:
        if what == "mxfp4" and C % 32:
            pytest.skip("MXFP4 blocks are 32 long")
        f = {"nvfp4": B.FORMAT_NVFP4, "mxfp4": B.FORMAT_MXFP4, "rows": B.FORMAT_NVFP4_ROWSCALE}[what]
        if what == "mxfp4" and R % 32:
            x = x[: R // 32 * 32] if R >= 32 else x.repeat(2, 1)
            R = x.shape[0]
        q = B.alloc_tensor(R, C, B.SF_LINEAR, format=f)
        B.nvfp4_quantize(x.contiguous(), B.quant_opts(), q)
        got, d = B.nvfp4_quant_error(x.contiguous(), q), x.double() - B.nvfp4_dequantize(q).double()
    want = torch.stack([d.square().sum(), x.double().square().sum()])
    assert bool(((got - want).abs() <= 16 * 2.0 ** -24 * want).all())


@pytest.mark.parametrize("shape", [(128, 128), (640, 1152), (16, 5136), (2064, 4112), (5120, 7680)])
@pytest.mark.parametrize("kind", ["activation", "gradient", "weight"])
def test_both_tile_widths_of_the_quantizer(shape, kind):
    """The tile width follows the number of tiles: one tile to 2400, ragged and whole."""
    R, C = shape
    g = torch.Generator("cuda").manual_seed(R + C)
    x = torch.randn((R, C), generator=g, device="cuda").to(torch.bfloat16)
    x[R // 2, C // 3] = 40.0
    layout = B.SF_SWIZZLED if R % 128 == 0 and C % 128 == 0 else B.SF_LINEAR
    opts = dict(block_rows=16) if kind == "weight" else dict(rounding=oracle.SR if kind == "gradient" else oracle.RNE,
                                                            seed=4, sr_offset=1)
    row, col = B.alloc_tensor(R, C, layout), B.alloc_tensor(C, R, layout)
    B.nvfp4_quantize(x, B.quant_opts(**opts), row, col)
    B.nvfp4_device_status()
    P.assert_exact(row, oracle.quantize(synth.bits(x.cpu()), **opts), "row")
    P.assert_exact(col, oracle.quantize(synth.bits(x.cpu()), colwise=True, **opts), "col")
