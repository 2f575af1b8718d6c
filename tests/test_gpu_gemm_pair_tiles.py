"""CTA-pair tiles at the edges: M and N odd multiples of 128 (half of the last tile lies outside), one tile and many, one
k-block and many, both output types, both formats, accumulation, two problems in one launch."""
import numpy as np
import pytest
import torch

import oracle
import parity as P
from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(128, 128, 256), (128, 640, 768), (384, 256, 512), (640, 384, 2304), (1152, 2688, 512)])
@pytest.mark.parametrize("tile", [512, 640, 768, 0])
@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("fmt", ["nvfp4", "mxfp4"])
def test_odd_multiples_of_128(shape, tile, fp32, fmt):
    M, N, K = shape
    X = synth.normal_with_outliers_bf16((M, K), 0.01, 50.0, M + N, M + N + 1)
    W = synth.normal_bf16((N, K), 0.02, M + N + 2)
    f = B.FORMAT_MXFP4 if fmt == "mxfp4" else B.FORMAT_NVFP4
    # the operands sit inside larger buffers filled with NaN scale bytes: nothing beyond the last group may be used
    A, Bt = B.alloc_tensor(M, K, format=f), B.alloc_tensor(N, K, format=f)
    for t in (A, Bt):
        big = torch.full((t.scales.numel() * 2 + 65536,), 0xFF, dtype=torch.uint8, device="cuda")
        t.scales = big[: t.scales.numel()]
    B.nvfp4_quantize(X.cuda(), B.quant_opts(), A, None)
    B.nvfp4_quantize(W.cuda(), B.quant_opts(block_rows=32 if fmt == "mxfp4" else 16), Bt, None)
    # exact reference: the decoded operands in binary64 (their codes are checked by the quantizer tests)
    a, b = (B.nvfp4_dequantize(t).double() for t in (A, Bt))
    Dref, T = (a @ b.T).cpu().numpy(), (a.abs() @ b.abs().T).cpu().numpy()
    wide = torch.full((M + 8, N + 64), 7.0, dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    D = wide[:M, :N]
    B.nvfp4_set_gemm_tile_n(tile)
    try:
        B.nvfp4_gemm(A, Bt, D)
        B.nvfp4_device_status()
        P.assert_gemm_close(D.float().cpu().numpy(), Dref, T, not fp32, f"{fmt} {shape} tile {tile}")
        assert torch.all(wide[M:] == 7.0) and torch.all(wide[:, N:] == 7.0)
        if fp32:  # what is added is the very product
            once = D.clone()
            B.nvfp4_gemm(A, Bt, D, accumulate=True)
            B.nvfp4_device_status()
            assert torch.equal(D, once + once)
    finally:
        B.nvfp4_set_gemm_tile_n(0)


@pytest.mark.parametrize("shape", [(256, 512, 256), (768, 1280, 1024)])
@pytest.mark.parametrize("tile", [512, 640, 768])
def test_layer_is_the_same_on_every_tile(shape, tile):
    """Dgrad and Wgrad share a launch: on every tile, forced or chosen by size, Y, dX and dW are the same up to the order of
    FP32 sums (and a bf16 boundary crossed here and there): 5e-5 of their norm."""
    M, N, K = shape
    X, W = synth.normal_bf16((M, K), 1.0, 1).cuda(), synth.normal_bf16((N, K), 0.02, 2).cuda()
    dY = synth.normal_bf16((M, N), 1e-3, 3).cuda()
    opts = B.quant_opts(rht_sign_mask=synth.DEFAULT_RHT_SIGN_MASK, seed=1)
    ws_f = torch.empty(B.nvfp4_linear_fwd_workspace_bytes(M, K), dtype=torch.uint8, device="cuda")
    ws_b = torch.empty(B.nvfp4_linear_bwd_workspace_bytes(M, N), dtype=torch.uint8, device="cuda")

    def run(t):
        X_col, W_row, W_col = B.alloc_tensor(K, M), B.alloc_tensor(N, K), B.alloc_tensor(K, N)
        Y, dX = (torch.empty(s, dtype=torch.bfloat16, device="cuda") for s in ((M, N), (M, K)))
        dW = torch.empty((N, K), dtype=torch.float32, device="cuda")
        B.nvfp4_set_gemm_tile_n(t)
        try:
            B.nvfp4_linear_fwd(X, W, opts, Y, X_col, W_row, W_col, False, ws_f)
            B.nvfp4_linear_bwd(dY, X_col, W_col, K, opts, dX, dW, False, ws_b)
            B.nvfp4_device_status()
        finally:
            B.nvfp4_set_gemm_tile_n(0)
        return Y, dX, dW

    for got, ref in zip(run(tile), run(0)):
        d = (got.double() - ref.double()).norm() / ref.double().norm()
        assert float(d) < 5e-5  # FP32 sums in another order, at most a bf16 boundary crossed here and there


@pytest.mark.parametrize("shape", [(8, 8, 8), (264, 520, 72), (776, 1096, 200), (2056, 2568, 136), (1032, 5128, 72)])
@pytest.mark.parametrize("layouts", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("fp32", [False, True])
def test_bf16_ragged_on_both_tiles(shape, layouts, fp32):
    """One round of 256 x 128 tiles (the first three shapes) and several of 256 x 256, edges of every kind, in a larger
    buffer."""
    M, N, K = shape
    g = torch.Generator("cuda").manual_seed(M + N)
    A, Bt = (torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for s in ((M, K), (N, K)))
    ref, T = A.double() @ Bt.double().T, A.double().abs() @ Bt.double().abs().T
    a = A.T.contiguous() if layouts[0] else A
    b = Bt.T.contiguous() if layouts[1] else Bt
    wide = torch.full((M + 8, N + 8), 7.0, dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    D = wide[:M, :N]
    B.nvfp4_gemm_bf16(a, b, D, *layouts)
    B.nvfp4_device_status()
    bound = 1e-4 * T + (0 if fp32 else 2.0 ** -8) * ref.abs()  # FP32 sums of exact products; one bf16 rounding
    assert bool(((D.double() - ref).abs() <= bound + 1e-12).all())
    assert torch.all(wide[M:] == 7.0) and torch.all(wide[:, N:] == 7.0)
    if fp32:
        once = D.clone()
        B.nvfp4_gemm_bf16(a, b, D, *layouts, accumulate=True)
        B.nvfp4_device_status()
        assert torch.equal(D, once + once)


@pytest.mark.parametrize("shape", [(256, 256, 256), (256, 768, 512), (512, 1280, 1024)])
@pytest.mark.parametrize("tile", [512, 640, 768])
@pytest.mark.parametrize("rows_on", ["A", "B", "AB"])
@pytest.mark.parametrize("fp32", [False, True])
def test_scale_vectors_on_every_pair_tile(shape, tile, rows_on, fp32):
    M, N, K = shape

    def operand(R, per_row, seed):
        x = synth.normal_bf16((R, K), 1.0, seed)
        x *= torch.exp2(torch.arange(R) % 13 - 6).to(torch.bfloat16)[:, None]  # rows far apart: a mixed-up factor shows
        t = B.alloc_tensor(R, K, format=B.FORMAT_NVFP4_ROWSCALE if per_row else B.FORMAT_NVFP4)
        B.nvfp4_quantize(x.cuda(), B.quant_opts(), t, None)
        return t

    A, Bt = operand(M, "A" in rows_on, 3), operand(N, "B" in rows_on, 4)
    a, b = (B.nvfp4_dequantize(t).double() for t in (A, Bt))
    D = torch.full((M, N), float("nan"), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    B.nvfp4_set_gemm_tile_n(tile)
    try:
        B.nvfp4_gemm(A, Bt, D)
        B.nvfp4_device_status()
    finally:
        B.nvfp4_set_gemm_tile_n(0)
    P.assert_gemm_close(D.float().cpu().numpy(), (a @ b.T).cpu().numpy(), (a.abs() @ b.abs().T).cpu().numpy(), not fp32,
                        f"rows {rows_on} tile {tile}")


@pytest.mark.parametrize("tile", [640, 642, 644, 768, 128])
def test_measurement_aids_leave_the_other_tiles_alone(tile):
    """No MMAs, no output, a capped grid and a probe are asked for: only the kernel with 256 x 256 tiles heeds them."""
    A, Bt = B.alloc_tensor(256, 1024), B.alloc_tensor(512, 1024)
    for t, seed in ((A, 1), (Bt, 2)):
        B.nvfp4_quantize(synth.normal_bf16((t.rows, t.cols), 1.0, seed).cuda(), B.quant_opts(), t, None)
    D, want = (torch.zeros((256, 512), device="cuda") for _ in range(2))
    probe = torch.zeros(8 * 74, dtype=torch.int64, device="cuda")
    B.nvfp4_set_gemm_tile_n(tile)
    try:
        B.nvfp4_gemm(A, Bt, want)
        B.nvfp4_set_gemm_experiment(1 | 8, 1, probe)
        B.nvfp4_gemm(A, Bt, D)
        B.nvfp4_device_status()
    finally:
        B.nvfp4_set_gemm_experiment()
        B.nvfp4_set_gemm_tile_n(0)
    assert torch.equal(D, want) and not probe.any()


# 143, 144 and 148 tiles of 128 x 128 (one round of 148 CTAs) where 256 x 128 would take two rounds of 74 pairs; then 150, and 72 pairs
@pytest.mark.parametrize("shape,single", [((1664, 1408, 512), True), ((1152, 2048, 2048), True), ((128, 18944, 768), True),
                                          ((1280, 1920, 512), False), ((1536, 1536, 512), False), ((1664, 1408, 8192), False)])
@pytest.mark.parametrize("fmt", [B.FORMAT_NVFP4, B.FORMAT_MXFP4])
@pytest.mark.parametrize("fp32", [False, True])
def test_single_tiles_where_pairs_would_go_round_twice(shape, single, fmt, fp32):
    """Chosen by size; the bits are those of the pair tiles, accumulated outputs included.  Blocks far apart in magnitude, so that
    the order of the additions shows."""
    M, N, K = shape
    if torch.cuda.get_device_properties(0).multi_processor_count == 148 and not fp32 and fmt == B.FORMAT_NVFP4:
        assert (B.nvfp4_gemm_tile(False, M, N, K, False) == 128) == single
    gen = torch.Generator("cuda").manual_seed(M + K)
    ops = []
    for rows in (M, N):
        x = torch.randn((rows, K), generator=gen, device="cuda")
        e = torch.randint(-9, 10, (rows // 32, K // 32), generator=gen, device="cuda").float()
        x = (x * torch.exp2(e).repeat_interleave(32, 0).repeat_interleave(32, 1)).to(torch.bfloat16)
        ops.append(B.alloc_tensor(rows, K, format=fmt))
        B.nvfp4_quantize(x, B.quant_opts(), ops[-1])
    dtype = torch.float32 if fp32 else torch.bfloat16
    wide = torch.full((M + 8, N + 64), 7.0, dtype=dtype, device="cuda")
    D, want = wide[:M, :N], torch.empty((M, N), dtype=dtype, device="cuda")
    for accumulate in (False, True)[:1 + fp32]:
        B.nvfp4_gemm(*ops, D, accumulate=accumulate)
        B.nvfp4_set_gemm_tile_n(512)
        try:
            B.nvfp4_gemm(*ops, want, accumulate=accumulate)
        finally:
            B.nvfp4_set_gemm_tile_n(0)
        B.nvfp4_device_status()
        assert torch.equal(D, want) and torch.all(wide[M:] == 7.0) and torch.all(wide[:, N:] == 7.0)
    if fp32:  # the forced kernel adds a rounded product, as the others do
        B.nvfp4_set_gemm_tile_n(128)
        try:
            B.nvfp4_gemm(*ops, D, accumulate=True)
        finally:
            B.nvfp4_set_gemm_tile_n(0)
        B.nvfp4_gemm(*ops, want, accumulate=True)
        assert torch.equal(D, want)
