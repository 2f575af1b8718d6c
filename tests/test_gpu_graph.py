"""The composed calls are stream-ordered and allocation-free, so a step can be captured in a CUDA graph and replayed;
the replay must reproduce the direct calls bit for bit (the kernels are deterministic)."""
import ctypes

import pytest
import torch

from paper_2509_25149_b200 import binding as B
from paper_2509_25149_b200 import synth

pytestmark = pytest.mark.gpu


def test_captured_step_replays_bit_for_bit():
    M, N, K = 1024, 1536, 768
    g = torch.Generator(device="cuda").manual_seed(7)
    X = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16)
    dY = (torch.randn((M, N), generator=g, device="cuda") * 1e-3).to(torch.bfloat16)
    opts = B.quant_opts(rht_sign_mask=synth.DEFAULT_RHT_SIGN_MASK, seed=3, sr_offset=5)
    X_col, W_row, W_col = B.alloc_tensor(K, M), B.alloc_tensor(N, K), B.alloc_tensor(K, N)
    Y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    dX = torch.empty((M, K), dtype=torch.bfloat16, device="cuda")
    dW = torch.empty((N, K), dtype=torch.float32, device="cuda")
    ws_f = torch.empty(B.nvfp4_linear_fwd_workspace_bytes(M, K), dtype=torch.uint8, device="cuda")
    ws_b = torch.empty(B.nvfp4_linear_bwd_workspace_bytes(M, N), dtype=torch.uint8, device="cuda")

    def step():
        B.nvfp4_linear_fwd(X, W, opts, Y, X_col, W_row, W_col, False, ws_f)
        B.nvfp4_linear_bwd(dY, X_col, W_col, K, opts, dX, dW, False, ws_b)

    step()  # first call outside the capture: it sets kernel attributes and fills the tensor-map cache
    torch.cuda.synchronize()
    B.nvfp4_device_status()
    want = [t.clone() for t in (Y, dX, dW, W_row.codes, W_col.codes, X_col.codes, W_row.glob, X_col.glob)]

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            step()
    torch.cuda.current_stream().wait_stream(side)
    for t in (Y, dX, dW, W_row.codes, W_col.codes, X_col.codes):
        t.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    B.nvfp4_device_status()
    for got, ref in zip((Y, dX, dW, W_row.codes, W_col.codes, X_col.codes, W_row.glob, X_col.glob), want):
        assert torch.equal(got, ref)


@pytest.mark.parametrize("call", ["rows", "transform", "weight", "gemm"])
def test_a_refused_launch_is_reported_once(call):
    """On a stream whose capture has been invalidated (by a synchronisation) launches are refused: the call reports that, and the next
    call, whose kernel is launched the ordinary way, does not find the error again."""
    xf = torch.randn((256, 512), device="cuda")
    x = xf.to(torch.bfloat16)
    row, col = B.alloc_tensor(256, 512), B.alloc_tensor(512, 256)
    rows = B.alloc_tensor(256, 512, format=B.FORMAT_NVFP4_ROWSCALE)
    B.nvfp4_quantize(x, B.quant_opts(), row, col)
    D = torch.empty((256, 256), dtype=torch.bfloat16, device="cuda")
    calls = {"rows": lambda: B.nvfp4_quantize(x, B.quant_opts(), rows, None),
             "transform": lambda: B.nvfp4_quantize(x, B.quant_opts(rht_colwise=True, rht_dim=4, flags=B.AMAX_PROVIDED), row, col),
             "weight": lambda: B.nvfp4_quantize(xf, B.quant_opts(block_rows=16), row, col),
             "gemm": lambda: B.nvfp4_gemm(row, row, D)}
    calls[call]()
    B.nvfp4_dequantize(row)
    out = torch.empty((256, 512), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.12")  # (the one that torch has loaded)
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreateWithFlags(ctypes.byref(stream), 1) == 0
    try:
        assert rt.cudaStreamBeginCapture(stream, 1) == 0  # thread-local
        assert rt.cudaStreamSynchronize(stream) != 0
        with torch.cuda.stream(torch.cuda.ExternalStream(stream.value)):
            with pytest.raises(B.NVFP4Error):
                calls[call]()
        assert rt.cudaStreamEndCapture(stream, ctypes.byref(graph)) != 0 and not graph.value
    finally:
        rt.cudaStreamDestroy(stream)
        rt.cudaGetLastError()
    B.nvfp4_dequantize(row, out)  # before anything else: it asks for the last error of the library's own runtime
    torch.cuda.synchronize()
    calls[call]()
    B.nvfp4_device_status()
