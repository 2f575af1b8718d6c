"""Parity of the CUDA quantizer (through the C ABI) with the CPU oracle, element by element."""
import numpy as np
import pytest
import torch

import oracle
import parity as P
from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu
MASK = synth.DEFAULT_RHT_SIGN_MASK


def rand_bf16(shape, seed, std=1.0, outliers=0.0):
    if outliers:
        return synth.normal_with_outliers_bf16(shape, outliers, 50.0, seed, seed + 1)
    return synth.normal_bf16(shape, std, seed)


SHAPES = [(128, 128), (256, 384), (512, 1024)]          # full tiles (swizzled scale layout)
RAGGED = [(16, 16), (144, 208), (48, 400), (272, 16)]   # partial tiles (linear scale layout)


@pytest.mark.parametrize("shape", SHAPES + RAGGED)
@pytest.mark.parametrize("which", ["row", "col", "both"])
def test_rne_1x16_is_bit_exact(shape, which):
    x = rand_bf16(shape, 100 + shape[0], outliers=0.01)
    layout = B.SF_SWIZZLED if shape in SHAPES else B.SF_LINEAR
    row, col = P.gpu_quantize(x, rowwise=which != "col", colwise=which != "row", sf_layout=layout)
    if row is not None:
        P.assert_exact(row, oracle.quantize(synth.bits(x)), f"row {shape}")
    if col is not None:
        P.assert_exact(col, oracle.quantize(synth.bits(x), colwise=True), f"col {shape}")


@pytest.mark.parametrize("shape", [(128, 128), (1024, 1024), (48, 80), (144, 208)])
@pytest.mark.parametrize("which", ["row", "col", "both"])
def test_rne_16x16_weights_are_bit_exact_and_consistent(shape, which):
    w = rand_bf16(shape, 7, std=0.02)
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 and shape[1] % 128 == 0 else B.SF_LINEAR
    row, col = P.gpu_quantize(w, rowwise=which != "col", colwise=which != "row", sf_layout=layout, block_rows=16)
    if row is not None:
        P.assert_exact(row, oracle.quantize(synth.bits(w), block_rows=16), "W row")
    if col is not None:
        P.assert_exact(col, oracle.quantize(synth.bits(w), block_rows=16, colwise=True), "W col")
    if row is not None and col is not None:
        # Section 4.3: one quantized representation for both passes
        assert torch.equal(B.nvfp4_dequantize(row), B.nvfp4_dequantize(col).T.contiguous())


@pytest.mark.parametrize("shape", [(128, 128), (256, 384), (144, 208)])
@pytest.mark.parametrize("which", ["row", "col", "both"])
@pytest.mark.parametrize("independent", [False, True])
def test_stochastic_rounding_is_bit_exact_given_the_stream(shape, which, independent):
    x = rand_bf16(shape, 31, std=1e-3)
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 and shape[1] % 128 == 0 else B.SF_LINEAR
    seed, off = 0x1234_5678_9ABC_DEF0, (3 << 32) | 17
    row, col = P.gpu_quantize(x, rowwise=which != "col", colwise=which != "row", sf_layout=layout,
                              rounding=B.ROUND_STOCHASTIC, seed=seed, sr_offset=off,
                              flags=B.SR_INDEPENDENT_COPIES if independent else 0)
    if row is not None:
        P.assert_exact(row, oracle.quantize(synth.bits(x), rounding=oracle.SR, seed=seed, sr_offset=off), "SR row")
    if col is not None:
        off_c = off | (1 << 63) if independent else off
        P.assert_exact(col, oracle.quantize(synth.bits(x), colwise=True, rounding=oracle.SR, seed=seed,
                                            sr_offset=off_c), "SR col")


def test_sr_16x16_and_seed_zero():
    w = rand_bf16((128, 256), 5, std=0.02)
    row, col = P.gpu_quantize(w, colwise=True, block_rows=16, rounding=B.ROUND_STOCHASTIC)
    P.assert_exact(row, oracle.quantize(synth.bits(w), block_rows=16, rounding=oracle.SR), "2D SR row")
    P.assert_exact(col, oracle.quantize(synth.bits(w), block_rows=16, rounding=oracle.SR, colwise=True), "2D SR col")


@pytest.mark.parametrize("shape", [(32, 32), (256, 384), (160, 224)])
@pytest.mark.parametrize("fmt", ["mxfp4", "binary32", "binary32, amax provided"])
def test_square_blocks_with_draws_of_their_own(shape, fmt):
    """Both copies of a weight in one call, the transposed one rounded with the second stream."""
    w = rand_bf16(shape, 5, std=0.02)
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 and shape[1] % 128 == 0 else B.SF_LINEAR
    opt = dict(rounding=B.ROUND_STOCHASTIC, seed=11, sr_offset=6, flags=B.SR_INDEPENDENT_COPIES)
    sr = dict(rounding=oracle.SR, seed=11)
    if fmt == "mxfp4":
        row, col = P.gpu_quantize_mx(w, colwise=True, sf_layout=layout, block_rows=32, **opt)
        P.assert_exact_mx(row, oracle.quantize_mx(synth.bits(w), block_rows=32, sr_offset=6, **sr), "row")
        P.assert_exact_mx(col, oracle.quantize_mx(synth.bits(w), block_rows=32, colwise=True, sr_offset=6 | (1 << 63), **sr),
                          "col")
        return
    w = w.float()
    row, col = (B.alloc_tensor(*s, layout) for s in (shape, shape[::-1]))
    if "provided" in fmt:
        opt["flags"] |= B.AMAX_PROVIDED
        row.glob[0] = col.glob[0] = float(w.abs().max())
    B.nvfp4_quantize(w.cuda(), B.quant_opts(block_rows=16, **opt), row, col)
    P.assert_exact(row, oracle.quantize(w.numpy(), block_rows=16, sr_offset=6, **sr), "row")
    P.assert_exact(col, oracle.quantize(w.numpy(), block_rows=16, colwise=True, sr_offset=6 | (1 << 63), **sr), "col")


@pytest.mark.parametrize("shape", [(128, 128), (256, 384), (144, 208)])
@pytest.mark.parametrize("rounding", [B.ROUND_NEAREST_EVEN, B.ROUND_STOCHASTIC])
def test_rht_copies_follow_the_tolerance_protocol(shape, rounding):
    x = rand_bf16(shape, 55, outliers=0.01)
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 and shape[1] % 128 == 0 else B.SF_LINEAR
    row, col = P.gpu_quantize(x, colwise=True, sf_layout=layout, rht_rowwise=True, rht_colwise=True,
                              rht_sign_mask=MASK, rounding=rounding, seed=9, sr_offset=1)
    xd = x.cuda()
    y_row = B.nvfp4_rht16(xd, False, MASK).cpu().numpy()
    y_col = B.nvfp4_rht16(xd, True, MASK).cpu().numpy()
    s1 = P.assert_rht_close(synth.bits(x), row, y_row, colwise=False, sign_mask=MASK, rounding=rounding, seed=9,
                            sr_offset=1, what="RHT row")
    s2 = P.assert_rht_close(synth.bits(x), col, y_col, colwise=True, sign_mask=MASK, rounding=rounding, seed=9,
                            sr_offset=1, what="RHT col")
    assert s1["excused_codes"] + s2["excused_codes"] <= 1e-3 * 2 * x.numel()


def test_recipe_combination_row_plain_col_rht():
    # the activation recipe: row-wise copy untouched (bit-exact), column-wise copy rotated (tolerance)
    x = rand_bf16((256, 256), 77, outliers=0.01)
    row, col = P.gpu_quantize(x, colwise=True, rht_colwise=True, rht_sign_mask=MASK)
    P.assert_exact(row, oracle.quantize(synth.bits(x)), "row of mixed call")
    y_col = B.nvfp4_rht16(x.cuda(), True, MASK).cpu().numpy()
    P.assert_rht_close(synth.bits(x), col, y_col, colwise=True, sign_mask=MASK, rounding=oracle.RNE, what="col of mixed")


def test_degenerate_inputs():
    z = torch.zeros((128, 128), dtype=torch.bfloat16)
    row, col = P.gpu_quantize(z, colwise=True)
    P.assert_exact(row, oracle.quantize(synth.bits(z)), "zeros row")
    P.assert_exact(col, oracle.quantize(synth.bits(z), colwise=True), "zeros col")
    # tiny and huge magnitudes, blocks that underflow the E4M3 range, negative zero
    x = rand_bf16((128, 128), 3)
    x[0, :16] = 3.0e38
    x[5, 32:48] = 1e-30
    x[7, 0] = -0.0
    row, col = P.gpu_quantize(x, colwise=True)
    P.assert_exact(row, oracle.quantize(synth.bits(x)), "extremes row")
    P.assert_exact(col, oracle.quantize(synth.bits(x), colwise=True), "extremes col")
    # leading dimension larger than the row length
    wide = rand_bf16((128, 256), 4).cuda()
    sub = wide[:, :128]
    r = B.alloc_tensor(128, 128)
    B.nvfp4_quantize(sub, B.quant_opts(), r, None)
    P.assert_exact(r, oracle.quantize(synth.bits(wide.cpu())[:, :128]), "strided input")
    # provided amax
    r2 = B.alloc_tensor(128, 128)
    r2.glob[0] = r.glob[0]
    B.nvfp4_quantize(sub, B.quant_opts(flags=B.AMAX_PROVIDED), r2, None)
    P.assert_exact(r2, oracle.quantize(synth.bits(wide.cpu())[:, :128]), "amax provided")


@pytest.mark.parametrize("scale", [1e-30, 1e-36, 3e-39, 1e30])
@pytest.mark.parametrize("rounding", [B.ROUND_NEAREST_EVEN, B.ROUND_STOCHASTIC])
def test_extreme_magnitudes_stay_bit_exact(scale, rounding):
    """Whole tensors near the ends of the bf16 range: the global encode scale clamps at FLT_MAX (amax below
    2688 / FLT_MAX), block amaxes are denormal (the exact-division path of amax_b / 6), products land in the
    denormal range (no flush to zero anywhere), and at the top 2688 / amax is itself tiny."""
    x = (synth.normal_bf16((128, 256), 1.0, 21).float() * scale).to(torch.bfloat16)
    x[3, 16:32] = 0.0
    for block_rows in (1, 16):
        row, col = P.gpu_quantize(x, colwise=True, block_rows=block_rows, rounding=rounding, seed=5, sr_offset=9)
        kw = dict(block_rows=block_rows, rounding=rounding, seed=5, sr_offset=9)
        P.assert_exact(row, oracle.quantize(synth.bits(x), **kw), f"row scale {scale} blocks {block_rows}")
        P.assert_exact(col, oracle.quantize(synth.bits(x), colwise=True, **kw), f"col scale {scale} blocks {block_rows}")


@pytest.mark.parametrize("amax", [5.0e-25, 5.8e-25])
@pytest.mark.parametrize("shape", [(128, 128), (144, 208)])
@pytest.mark.parametrize("rounding", [B.ROUND_NEAREST_EVEN, B.ROUND_STOCHASTIC])
def test_blocks_beside_the_limit_of_the_plain_division(amax, shape, rounding):
    """amax_b / 6 is divided without a branch while s_enc = 2688 / amax is at most 5e27 (amax 5.4e-25): tensors on either side,
    with blocks whose amax is 1, 1e-3 ... 1e-12 of the tensor's, i.e. above and below 1e-30 and below the smallest normal."""
    x = rand_bf16(shape, 77).float()
    decades = torch.arange(shape[0] // 16).repeat_interleave(16)[:, None] + torch.arange(shape[1] // 16).repeat_interleave(16)
    x = x / x.abs().max() * amax * 10.0 ** (-3.0 * (decades % 5))
    x[0, 0] = amax
    x = x.bfloat16()
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 else B.SF_LINEAR
    row, col = P.gpu_quantize(x, rowwise=True, colwise=True, sf_layout=layout, rounding=rounding, seed=3, sr_offset=2)
    kw = dict(rounding=oracle.RNE if rounding == B.ROUND_NEAREST_EVEN else oracle.SR, seed=3, sr_offset=2)
    P.assert_exact(row, oracle.quantize(synth.bits(x), **kw), "row")
    P.assert_exact(col, oracle.quantize(synth.bits(x), colwise=True, **kw), "col")


@pytest.mark.parametrize("case", ["both_tiny", "transformed_tiny", "plain_tiny"])
@pytest.mark.parametrize("shape", [(128, 128), (144, 208)])
@pytest.mark.parametrize("rounding,flags", [(B.ROUND_NEAREST_EVEN, 0), (B.ROUND_STOCHASTIC, 0),
                                            (B.ROUND_STOCHASTIC, B.SR_INDEPENDENT_COPIES)])
def test_transformed_copies_beside_the_limit_of_the_plain_division(case, shape, rounding, flags):
    """The limit is an amax of 5.4e-25, and either copy's decides for both: a transformed copy below it beside a plain one above
    (one large element: its transform has a quarter of it), the reverse (a chunk whose signs are the transform's: four times)."""
    x = rand_bf16(shape, 78).float()
    decades = torch.arange(shape[0] // 16).repeat_interleave(16)[:, None] + torch.arange(shape[1] // 16).repeat_interleave(16)
    x = x / x.abs().max() * (2.0e-25 if case == "both_tiny" else 2.0e-26) * 10.0 ** (-3.0 * (decades % 5))
    if case == "transformed_tiny":
        x[5, 7] = 9.0e-25
    if case == "plain_tiny":
        x[16:32, 9] = 3.0e-25 * torch.tensor([1.0 - 2.0 * (MASK >> j & 1) for j in range(16)])
    x = x.bfloat16()
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 else B.SF_LINEAR
    row, col = P.gpu_quantize(x, rowwise=True, colwise=True, sf_layout=layout, rounding=rounding, seed=3, sr_offset=2, flags=flags,
                              rht_colwise=True, rht_sign_mask=MASK)
    amaxes = float(row.glob[0]), float(col.glob[0])
    assert [a < 5.37e-25 for a in amaxes] == [case != "transformed_tiny", case != "plain_tiny"], amaxes
    kw = dict(rounding=oracle.RNE if rounding == B.ROUND_NEAREST_EVEN else oracle.SR, seed=3)
    P.assert_exact(row, oracle.quantize(synth.bits(x), sr_offset=2, **kw), "row")
    y = B.nvfp4_rht16(x.cuda(), True, MASK).cpu().numpy()
    P.assert_rht_close(synth.bits(x), col, y, colwise=True, sign_mask=MASK, sr_offset=2 | (1 << 63 if flags else 0), what="col", **kw)


@pytest.mark.parametrize("kind", ["activation", "weight", "rows", "mxfp4"])
def test_a_nan_changes_no_other_element(kind):
    """What an element that is no number becomes is unspecified, but the maxima pass over it, in either half of a word and with
    either sign: scales and other codes are those of the tensor with zeros there."""
    x = rand_bf16((128, 256), 79)
    where = torch.zeros(x.shape, dtype=torch.bool)
    for r, c in ((0, 0), (3, 17), (3, 18), (40, 255), (127, 128)):
        where[r, c] = True
    where[64, 32:64] = True  # whole blocks
    nan = torch.where(torch.arange(256) % 3 == 0, -torch.tensor(float("nan")), torch.tensor(float("nan")))
    fmt = {"rows": B.FORMAT_NVFP4_ROWSCALE, "mxfp4": B.FORMAT_MXFP4}.get(kind, B.FORMAT_NVFP4)
    got = []
    for src in (torch.where(where, nan, x.float()).bfloat16(), torch.where(where, 0.0, x.float()).bfloat16()):
        row, col = B.alloc_tensor(128, 256, format=fmt), None if kind == "rows" else B.alloc_tensor(256, 128, format=fmt)
        B.nvfp4_quantize(src.cuda(), B.quant_opts(block_rows=16 if kind == "weight" else 1), row, col)
        got.append((row, col))
    for (a, b), elsewhere in zip(zip(*got), (~where, ~where.T)):
        if a is None:
            continue
        assert torch.equal(a.glob, b.glob) and torch.equal(a.scales, b.scales)
        nibbles = [P.unpack(t.codes.cpu().numpy()) for t in (a, b)]
        assert np.array_equal(nibbles[0][elsewhere.numpy()], nibbles[1][elsewhere.numpy()])


def test_an_infinite_row_leaves_the_others_their_scales():
    x = rand_bf16((32, 10304), 80)
    row = []
    for v in (float("inf"), 0.0):
        x[9, 4000] = v
        row.append(B.alloc_tensor(32, 10304, B.SF_LINEAR, format=B.FORMAT_NVFP4_ROWSCALE))
        B.nvfp4_quantize(x.cuda(), B.quant_opts(), row[-1], None)
    keep = torch.arange(32) != 9
    for name, width in (("codes", 5152), ("scales", 644), ("glob", 2)):
        a, b = (getattr(t, name).reshape(32, width)[keep.cuda()] for t in row)
        assert torch.equal(a, b), name
    assert float(row[0].glob.reshape(32, 2)[9, 0]) == float("inf")


def test_gpu_sr_is_unbiased_over_seeds():
    x = rand_bf16((128, 128), 8, std=1e-3)
    xd = x.cuda()
    S = 512
    acc = torch.zeros((128, 128), dtype=torch.float64, device="cuda")
    acc_c = torch.zeros((128, 128), dtype=torch.float64, device="cuda")
    row, col = B.alloc_tensor(128, 128), B.alloc_tensor(128, 128)
    for seed in range(S):
        B.nvfp4_quantize(xd, B.quant_opts(rounding=B.ROUND_STOCHASTIC, seed=seed), row, col)
        acc += B.nvfp4_dequantize(row).double()
        acc_c += B.nvfp4_dequantize(col).double().T
    ref = oracle.quantize(synth.bits(x))
    sb = np.vectorize(oracle.e4m3_decode)(ref.scales).repeat(16, axis=1) * float(ref.s_dec)
    xf = x.double().numpy()
    sat = np.maximum(np.abs(xf) - 6.0 * sb, 0.0)
    assert np.all(np.abs(acc.cpu().numpy() / S - xf) <= sat + 2.0 * sb * (1 / 512 + 2.5 / np.sqrt(S)) + 1e-12)
    refc = oracle.quantize(synth.bits(x), colwise=True)
    sbc = (np.vectorize(oracle.e4m3_decode)(refc.scales).repeat(16, axis=1) * float(refc.s_dec)).T
    satc = np.maximum(np.abs(xf) - 6.0 * sbc, 0.0)
    assert np.all(np.abs(acc_c.cpu().numpy() / S - xf) <= satc + 2.0 * sbc * (1 / 512 + 2.5 / np.sqrt(S)) + 1e-12)


def test_config1_tensors_all_roles():
    p = synth.config1()
    # X: row-wise plain + column-wise rotated, RNE
    row, col = P.gpu_quantize(p.X, colwise=True, rht_colwise=True, rht_sign_mask=p.rht_sign_mask)
    P.assert_exact(row, oracle.quantize(synth.bits(p.X)), "cfg1 X row")
    P.assert_rht_close(synth.bits(p.X), col, B.nvfp4_rht16(p.X.cuda(), True, p.rht_sign_mask).cpu().numpy(),
                       colwise=True, sign_mask=p.rht_sign_mask, rounding=oracle.RNE, what="cfg1 X col")
    # W: 16x16 both copies
    row, col = P.gpu_quantize(p.W, colwise=True, block_rows=16)
    P.assert_exact(row, oracle.quantize(synth.bits(p.W), block_rows=16), "cfg1 W row")
    P.assert_exact(col, oracle.quantize(synth.bits(p.W), block_rows=16, colwise=True), "cfg1 W col")
    # dY: SR, row-wise plain + column-wise rotated
    row, col = P.gpu_quantize(p.dY, colwise=True, rht_colwise=True, rht_sign_mask=p.rht_sign_mask,
                              rounding=B.ROUND_STOCHASTIC, seed=p.sr_seed, sr_offset=p.sr_offset)
    P.assert_exact(row, oracle.quantize(synth.bits(p.dY), rounding=oracle.SR, seed=p.sr_seed, sr_offset=p.sr_offset),
                   "cfg1 dY row")
    P.assert_rht_close(synth.bits(p.dY), col, B.nvfp4_rht16(p.dY.cuda(), True, p.rht_sign_mask).cpu().numpy(),
                       colwise=True, sign_mask=p.rht_sign_mask, rounding=oracle.SR, seed=p.sr_seed,
                       sr_offset=p.sr_offset, what="cfg1 dY col")


@pytest.mark.parametrize("shape", [(128, 128), (256, 384), (144, 208)])
@pytest.mark.parametrize("block_rows", [1, 16])
@pytest.mark.parametrize("rounding", [B.ROUND_NEAREST_EVEN, B.ROUND_STOCHASTIC])
def test_binary32_source_is_bit_exact(shape, block_rows, rounding):
    """Appendix B: the source may be FP32 (e.g. master weights).  Values with full 24-bit mantissas."""
    g = torch.Generator().manual_seed(77)
    x = torch.randn(shape, generator=g, dtype=torch.float32) * 0.02
    x[3, 5] = 1.2345678  # the amax, not representable in bf16
    layout = B.SF_SWIZZLED if shape[0] % 128 == 0 and shape[1] % 128 == 0 else B.SF_LINEAR
    R, C = shape
    row, col = B.alloc_tensor(R, C, layout), B.alloc_tensor(C, R, layout)
    B.nvfp4_quantize(x.cuda(), B.quant_opts(block_rows=block_rows, rounding=rounding, seed=11, sr_offset=2), row, col)
    kw = dict(block_rows=block_rows, rounding=rounding, seed=11, sr_offset=2)
    P.assert_exact(row, oracle.quantize(x.numpy(), **kw), "f32 row")
    P.assert_exact(col, oracle.quantize(x.numpy(), colwise=True, **kw), "f32 col")
    only = B.alloc_tensor(C, R, layout)
    B.nvfp4_quantize(x.cuda(), B.quant_opts(block_rows=block_rows, rounding=rounding, seed=11, sr_offset=2), None, only)
    P.assert_exact(only, oracle.quantize(x.numpy(), colwise=True, **kw), "f32 col only")
    with pytest.raises(B.NVFP4Error) as e:  # no transform on a binary32 source
        B.nvfp4_quantize(x.cuda(), B.quant_opts(rht_colwise=True, rht_sign_mask=MASK), row, col)
    assert e.value.status == 8
