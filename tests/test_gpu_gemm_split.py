"""Products whose contraction several CTA pairs share (block-scaled and BF16): shares of equal and unequal length down to one k-block, tiles half
outside, both output types, every scale format, accumulation, and sizes on both sides of the rule that chooses it."""
import pytest
import torch

import parity as P
from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu


def _operands(M, N, K, fmt):
    f = B.FORMAT_MXFP4 if fmt == "mxfp4" else B.FORMAT_NVFP4
    A = B.alloc_tensor(M, K, format=B.FORMAT_NVFP4_ROWSCALE if fmt == "rows" else f)
    Bt = B.alloc_tensor(N, K, format=f)
    B.nvfp4_quantize(synth.normal_with_outliers_bf16((M, K), 0.01, 50.0, M + N, M + N + 1).cuda(), B.quant_opts(), A, None)
    B.nvfp4_quantize(synth.normal_bf16((N, K), 0.02, M + N + 2).cuda(),
                     B.quant_opts(block_rows=32 if fmt == "mxfp4" else 16), Bt, None)
    a, b = B.nvfp4_dequantize(A).double(), B.nvfp4_dequantize(Bt).double()
    return A, Bt, (a @ b.T).cpu().numpy(), (a.abs() @ b.abs().T).cpu().numpy()


@pytest.mark.parametrize("shape", [(256, 256, 512), (256, 256, 1024), (128, 384, 1280), (512, 512, 1792), (384, 128, 5120),
                                   (256, 8192, 1024)])
@pytest.mark.parametrize("tile", [642, 644])
@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("fmt", ["nvfp4", "mxfp4", "rows"])
def test_shared_contraction(shape, tile, fp32, fmt):
    M, N, K = shape
    if fmt == "rows":
        M, N = (M + 255) // 256 * 256, (N + 255) // 256 * 256
    A, Bt, want, T = _operands(M, N, K, fmt)
    wide = torch.full((M + 8, N + 64), 7.0, dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    D = wide[:M, :N]
    B.nvfp4_set_gemm_tile_n(tile)
    try:
        B.nvfp4_gemm(A, Bt, D)
        B.nvfp4_device_status()
        P.assert_gemm_close(D.float().cpu().numpy(), want, T, not fp32, f"{fmt} {shape} split {tile}")
        assert torch.all(wide[M:] == 7.0) and torch.all(wide[:, N:] == 7.0)
        once = D.clone()
        B.nvfp4_gemm(A, Bt, D)
        assert torch.equal(D, once)  # the shares are added in a fixed order
        if fp32:  # what is added is the very product
            B.nvfp4_gemm(A, Bt, D, accumulate=True)
            B.nvfp4_device_status()
            assert torch.equal(D, once + once)
    finally:
        B.nvfp4_set_gemm_tile_n(0)


@pytest.mark.parametrize("shape", [(256, 256, 1280), (256, 256, 2560), (256, 1024, 4096), (1024, 1024, 8192), (1024, 1152, 8192),
                                   (128, 128, 20480)])
def test_sizes_around_the_rule(shape):
    """Chosen by size: 8 products behind each other (their clusters start while the one before drains) give the same bits."""
    M, N, K = shape
    A, Bt, want, T = _operands(M, N, K, "nvfp4")
    outs = [torch.empty((M, N), device="cuda") for _ in range(8)]
    for D in outs:
        B.nvfp4_gemm(A, Bt, D)
    B.nvfp4_device_status()
    P.assert_gemm_close(outs[0].cpu().numpy(), want, T, False, f"{shape}")
    assert all(torch.equal(D, outs[0]) for D in outs)


# shares of one k-block (K = 256) and of unequal length, ragged sizes; the last two lie beyond the rule (33 tiles and more)
@pytest.mark.parametrize("shape", [(256, 128, 256), (264, 520, 1000), (520, 264, 2056), (512, 1024, 4096), (1000, 1000, 1032),
                                   (128, 4096, 1024), (1000, 2000, 1000), (1288, 1024, 776)])
def test_bf16_products(shape):
    """Against binary64.  A sum of K products in FP32: K roundings of 2^-23 of what the terms' magnitudes add up to at most."""
    M, N, K = shape
    gen = torch.Generator("cuda").manual_seed(M + N + K)
    X, W, dY = (torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16) for s in ((M, K), (N, K), (M, N)))
    Y, dX = (torch.full((M, n), 7.0, dtype=torch.bfloat16, device="cuda") for n in (N, K))
    dW = torch.full((N, K), 2.0, device="cuda")
    B.nvfp4_linear_bf16_fwd(X, W, Y)
    B.nvfp4_linear_bf16_bwd(dY, X, W, K, dX, dW, True)
    B.nvfp4_device_status()
    x, w, dy = X.double(), W.double(), dY.double()
    for got, a, b, depth, bf16 in ((Y, x, w, K, True), (dX, dy, w.T, N, True), (dW - 2.0, dy.T, x.T, M, False)):
        want, T = a @ b.T, a.abs() @ b.abs().T
        bound = depth * 2.0 ** -23 * T + (2.0 ** -8 * want.abs() if bf16 else 2.0 ** -22 * (want.abs() + 2.0))
        assert torch.all((got.double() - want).abs() <= bound)
    again = torch.empty_like(Y)
    B.nvfp4_linear_bf16_fwd(X, W, again)
    assert torch.equal(again, Y)


# the first two are split by the rule (dX, dW); 1280 and 1792: shares of unequal length
@pytest.mark.parametrize("size", [(512, 3584, 768), (2048, 512, 512), (256, 1280, 1792), (1792, 256, 1280), (256, 256, 512)])
@pytest.mark.parametrize("tile", [0, 642, 644])
@pytest.mark.parametrize("fmt", [B.FORMAT_NVFP4, B.FORMAT_MXFP4])
def test_backward_call_sums_as_its_products_do(size, tile, fmt):
    """Blocks far apart in magnitude, so that the FP32 sums are not exact: the bits tell the order of the additions."""
    M, N, K = size
    gen = torch.Generator("cuda").manual_seed(M + N + K)

    def source(rows, cols):
        x = torch.randn((rows, cols), generator=gen, device="cuda")
        return (x * torch.exp2(torch.randint(-9, 10, (rows // 32, cols // 32), generator=gen, device="cuda").float())
                .repeat_interleave(32, 0).repeat_interleave(32, 1)).to(torch.bfloat16)

    dy = source(M, N)
    xc, wc, gr, gc = (B.alloc_tensor(r, c, format=fmt) for r, c in ((K, M), (K, N), (M, N), (N, M)))
    B.nvfp4_quantize(source(K, M), B.quant_opts(), xc)
    B.nvfp4_quantize(source(K, N), B.quant_opts(), wc)
    opts = B.quant_opts(rounding=B.ROUND_STOCHASTIC, rht_colwise=True, rht_sign_mask=0x73E5, seed=3)
    B.nvfp4_quantize(dy, opts, gr, gc)
    ws = torch.empty(B.nvfp4_linear_bwd_workspace_bytes(M, N), dtype=torch.uint8, device="cuda")

    def buffers():
        return torch.zeros((M, K), dtype=torch.bfloat16, device="cuda"), torch.full((N, K), 0.5, device="cuda")

    B.nvfp4_set_gemm_tile_n(tile)
    try:
        (dx0, dw0), (dx1, dw1), (dx2, dw2) = buffers(), buffers(), buffers()
        B.nvfp4_gemm(gr, wc, dx0)
        B.nvfp4_gemm(gc, xc, dw0, accumulate=True)
        B.nvfp4_linear_bwd(dy, xc, wc, K, opts, dx1, dw1, True, ws)
        B.nvfp4_linear_bwd(dy, xc, wc, K, opts, dx2, None, True, ws)
        B.nvfp4_linear_bwd(dy, xc, wc, K, opts, None, dw2, True, ws)
        B.nvfp4_device_status()
    finally:
        B.nvfp4_set_gemm_tile_n(0)
    assert torch.equal(dx1, dx0) and torch.equal(dw1, dw0) and torch.equal(dx2, dx0) and torch.equal(dw2, dw0)


# one k-block or an unequal number of them to a share, ragged in every direction, more clusters than are resident
@pytest.mark.parametrize("shape", [(8, 8, 256), (264, 520, 328), (776, 264, 1000), (1032, 2056, 264)])
@pytest.mark.parametrize("tile", [642, 644])
def test_bf16_products_on_split_tiles(shape, tile):
    """Both forms are forced: all four operand layouts, both outputs, accumulation, and two problems in one launch."""
    M, N, K = shape
    gen = torch.Generator("cuda").manual_seed(M + N + K)
    a, b = (torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16) for s in ((M, K), (N, K)))
    want, T = a.double() @ b.double().T, a.double().abs() @ b.double().abs().T
    B.nvfp4_set_gemm_tile_n(tile)
    try:
        assert B.nvfp4_gemm_tile(True, M, N, K, False) == tile
        for layouts in ((0, 0), (0, 1), (1, 0), (1, 1)):
            ops = [t.T.contiguous() if mn else t for t, mn in zip((a, b), layouts)]
            for dtype in (torch.float32, torch.bfloat16):
                wide = torch.full((M + 8, N + 8), 7.0, dtype=dtype, device="cuda")
                D = wide[:M, :N]
                B.nvfp4_gemm_bf16(*ops, D, *layouts)
                B.nvfp4_device_status()
                # K roundings of what the magnitudes add up to at most, and the rounding of the output
                bound = K * 2.0 ** -23 * T + (2.0 ** -8 * want.abs() if dtype == torch.bfloat16 else 0)
                assert torch.all((D.double() - want).abs() <= bound + 1e-30)
                assert torch.all(wide[M:] == 7.0) and torch.all(wide[:, N:] == 7.0)
                if dtype == torch.float32:
                    once = D.clone()
                    B.nvfp4_gemm_bf16(*ops, D, *layouts, accumulate=True)
                    assert torch.equal(D, once + once)
        # as a layer's backward call: dX = dY W and dW = dY^T X with dY [M x N], W [N x K], X [M x K], each as by itself
        dy = want.to(torch.bfloat16)
        dx, dw = torch.empty_like(a), torch.empty((N, K), device="cuda")
        B.nvfp4_linear_bf16_bwd(dy, a, b, K, dx, dw, False)
        if N > 192 and M > 192:  # (otherwise a share would be empty, and the call is not split)
            one, two = torch.empty_like(dx), torch.empty_like(dw)
            B.nvfp4_linear_bf16_bwd(dy, None, b, K, one, None, False)
            B.nvfp4_linear_bf16_bwd(dy, a, None, K, None, two, False)
            assert torch.equal(dx, one) and torch.equal(dw, two)
        B.nvfp4_device_status()
        T = dy.double().abs() @ b.double().abs()
        assert torch.all((dx.double() - dy.double() @ b.double()).abs() <= N * 2.0 ** -23 * T + 2.0 ** -7 * T)
        T = dy.double().abs().T @ a.double().abs()
        assert torch.all((dw.double() - dy.double().T @ a.double()).abs() <= M * 2.0 ** -23 * T + 1e-30)
    finally:
        B.nvfp4_set_gemm_tile_n(0)


def test_the_rule_splits_where_it_says():
    """Few tiles and a long contraction, by size alone (any GPU keeps two clusters resident); short ones and many tiles stay whole."""
    split = {642, 644}
    for bf16, size, want in [(False, (256, 256, 5120), split), (False, (128, 128, 20480), split), (True, (256, 128, 4096), split),
                             (True, (264, 128, 1032), split), (False, (256, 256, 1280), {640}), (True, (256, 128, 256), {640}),
                             (False, (4096, 4096, 4096), {512, 640, 768}), (True, (4096, 4096, 4096), {512})]:
        for fp32 in (False, True):
            assert B.nvfp4_gemm_tile(bf16, *size, fp32) in want, (bf16, size)
    for bf16, size in [(False, (64, 128, 256)), (False, (128, 128, 128)), (True, (4, 8, 8)), (True, (8, 8, 0))]:
        assert B.nvfp4_gemm_tile(bf16, *size, False) == -1


# one column tile of 512 and nine of 256; two and twelve; thirteen and three; 16 and 17 k-blocks, the last of 8 and 40 elements;
# row lengths that are odd multiples of 16 bytes
@pytest.mark.parametrize("shape", [(1608, 2600, 968), (1056, 3960, 1032), (2056, 7176, 1064)])
def test_bf16_products_on_512_wide_tiles(shape):
    M, N, K = shape
    gen = torch.Generator("cuda").manual_seed(M + N + K)
    a, b = (torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16) for s in ((M, K), (N, K)))
    want, T = a.double() @ b.double().T, a.double().abs() @ b.double().abs().T
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert B.nvfp4_gemm_tile(True, M, N, K, False) == 1024
    for layouts in ((0, 0), (0, 1), (1, 0), (1, 1)):
        ops = [t.T.contiguous() if mn else t for t, mn in zip((a, b), layouts)]
        for dtype in (torch.float32, torch.bfloat16):
            wide = torch.full((M + 8, N + 8), 7.0, dtype=dtype, device="cuda")
            D = wide[:M, :N]
            B.nvfp4_gemm_bf16(*ops, D, *layouts)
            B.nvfp4_device_status()
            # K roundings of what the magnitudes add up to at most, and the rounding of the output
            bound = K * 2.0 ** -23 * T + (2.0 ** -8 * want.abs() if dtype == torch.bfloat16 else 0)
            assert torch.all((D.double() - want).abs() <= bound + 1e-30)
            assert torch.all(wide[M:] == 7.0) and torch.all(wide[:, N:] == 7.0)
            if dtype == torch.float32:
                once = D.clone()
                B.nvfp4_gemm_bf16(*ops, D, *layouts, accumulate=True)
                assert torch.equal(D, once + once)


@pytest.mark.parametrize("shape", [(1040, 3664, 904), (1544, 1680, 1912), (1592, 1552, 2128), (1112, 1144, 2344), (1224, 1192, 2328)])
def test_bf16_backward_call_on_512_wide_tiles(shape):
    """Tiles of both widths and of both products in one launch; each product has the bits that it has alone."""
    M, N, K = shape
    gen = torch.Generator("cuda").manual_seed(M + N + K)
    dy, x, w = (torch.randn(s, generator=gen, device="cuda").to(torch.bfloat16) for s in ((M, N), (M, K), (N, K)))
    dx, dw = torch.empty_like(x), torch.empty((N, K), device="cuda")
    one, two = torch.empty_like(dx), torch.empty_like(dw)
    B.nvfp4_linear_bf16_bwd(dy, x, w, K, dx, dw, False)
    B.nvfp4_linear_bf16_bwd(dy, None, w, K, one, None, False)
    B.nvfp4_linear_bf16_bwd(dy, x, None, K, None, two, False)
    B.nvfp4_device_status()
    T = dy.double().abs() @ w.double().abs()
    assert torch.all((dx.double() - dy.double() @ w.double()).abs() <= N * 2.0 ** -23 * T + 2.0 ** -8 * T)
    T = dy.double().abs().T @ x.double().abs()
    assert torch.all((dw.double() - dy.double().T @ x.double()).abs() <= M * 2.0 ** -23 * T + 1e-30)
    assert torch.equal(dx, one) and torch.equal(dw, two)


def test_bf16_products_of_slices_that_begin_beside_64_bytes():
    """Rows a multiple of 64 bytes apart, the first one 16 bytes behind such a boundary (tiles 512 wide on 148 SMs), in every layout."""
    M, N, K = 1536, 4608, 1024
    gen = torch.Generator("cuda").manual_seed(9)

    def slice_(rows, cols):
        buf = torch.randn((rows, cols + 32), generator=gen, device="cuda").to(torch.bfloat16)
        return buf[:, 8:8 + cols]

    for layouts in ((0, 0), (0, 1), (1, 0), (1, 1)):
        a, b = (slice_(K, n) if mn else slice_(n, K) for n, mn in zip((M, N), layouts))
        D = torch.empty((M, N), device="cuda")
        B.nvfp4_gemm_bf16(a, b, D, *layouts)
        B.nvfp4_device_status()
        A64, B64 = (t.double().T if mn else t.double() for t, mn in zip((a, b), layouts))
        # K roundings of what the magnitudes add up to at most
        assert torch.all((D.double() - A64 @ B64.T).abs() <= K * 2.0 ** -23 * (A64.abs() @ B64.abs().T))
