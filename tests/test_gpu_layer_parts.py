"""Pass 1 of a layer's call leaves the maximum of each of its tiles (128 x 256) in an output that the call writes last, while
four times as many tiles fit the resident CTAs (74 tiles on 148 SMs); the quantizer by itself takes them into one word.  Both
ways, on either side of that limit and where an output lies over an input, every byte is the same."""
import pytest
import torch

from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu
OPTS = dict(rht_sign_mask=synth.DEFAULT_RHT_SIGN_MASK, seed=3, sr_offset=5)


def _bytes(t):
    return [t.codes, t.scales, t.glob]


def _separate(x, w, dy):
    """The same step by separate calls."""
    (M, K), N = x.shape, w.shape[0]
    xr, xc, wr, wc = B.alloc_tensor(M, K), B.alloc_tensor(K, M), B.alloc_tensor(N, K), B.alloc_tensor(K, N)
    gr, gc = B.alloc_tensor(M, N), B.alloc_tensor(N, M)
    B.nvfp4_quantize(x, B.quant_opts(rht_colwise=True, **OPTS), xr, xc)
    B.nvfp4_quantize(w, B.quant_opts(block_rows=16), wr, wc)
    B.nvfp4_quantize(dy, B.quant_opts(rounding=B.ROUND_STOCHASTIC, rht_colwise=True, **OPTS), gr, gc)
    y, dx = (torch.empty((M, n), dtype=torch.bfloat16, device="cuda") for n in (N, K))
    dw = torch.empty((N, K), dtype=torch.float32, device="cuda")
    B.nvfp4_gemm(xr, wr, y)
    B.nvfp4_gemm(gr, wc, dx)
    B.nvfp4_gemm(gc, xc, dw)
    return y, dx, dw, _bytes(xc) + _bytes(wr) + _bytes(wc)


# tiles of X and W together | of dY: 2, 64, 72 | 80 (forward limit 74), 72 | 80 (backward)
@pytest.mark.parametrize("size", [(256, 256, 256), (1024, 1024, 1024), (1024, 1280, 1024), (1024, 1536, 1024), (1024, 2304, 512),
                                  (1280, 2048, 256), (256, 2304, 1792)])
@pytest.mark.parametrize("cached", [False, True])
@pytest.mark.parametrize("in_place", [False, True])
def test_layer_equals_its_steps(size, cached, in_place):
    M, N, K = size
    if in_place:
        N = K = max(N, K)
    src = synth.normal_with_outliers_bf16((M, K), 0.01, 50.0, M, K).cuda()
    w = synth.normal_bf16((N, K), 0.02, N).cuda()
    dsrc = synth.normal_bf16((M, N), 1e-4, M + N).cuda()
    y_want, dx_want, dw_want, copies_want = _separate(src, w, dsrc)
    xc, wr, wc = B.alloc_tensor(K, M), B.alloc_tensor(N, K), B.alloc_tensor(K, N)
    for t in (xc, wr, wc):
        t.glob.fill_(3e38)  # whatever the words held before
    if cached:
        B.nvfp4_quantize(w, B.quant_opts(block_rows=16), wr, wc)
    x, dy = torch.zeros_like(src), torch.zeros_like(dsrc)
    y = x if in_place else torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    dx = dy if in_place else torch.empty((M, K), dtype=torch.bfloat16, device="cuda")
    dw = torch.empty((N, K), dtype=torch.float32, device="cuda")
    opts = B.quant_opts(**OPTS)
    ws = torch.empty(max(B.nvfp4_linear_fwd_workspace_bytes(M, K), B.nvfp4_linear_bwd_workspace_bytes(M, N)),
                     dtype=torch.uint8, device="cuda")
    x.copy_(src)  # the calls' first kernels begin while these copies run
    B.nvfp4_linear_fwd(x, None if cached else w, opts, y, xc, wr, None if cached else wc, cached, ws)
    y_got = y.clone()
    dy.copy_(dsrc)
    B.nvfp4_linear_bwd(dy, xc, wc, K, opts, dx, dw, False, ws)
    assert torch.equal(y_got, y_want) and torch.equal(dx, dx_want) and torch.equal(dw, dw_want)
    for got, want in zip(_bytes(xc) + _bytes(wr) + _bytes(wc), copies_want):
        assert torch.equal(got, want)
    if not in_place:  # one product of the backward call alone
        dw.zero_()
        B.nvfp4_linear_bwd(dy, xc, wc, K, opts, None, dw, False, ws)
        assert torch.equal(dw, dw_want)
        dx.zero_()
        B.nvfp4_linear_bwd(dy, xc, wc, K, opts, dx, None, False, ws)
        assert torch.equal(dx, dx_want)
