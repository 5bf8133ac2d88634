"""mxattn_last_launch_count against the kernel nodes that the same call leaves in a captured CUDA graph, on every path that
launches a different number of kernels; and the captured graph gives what the call gives."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def nodes_of(call):
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        call()
    n = ctypes.c_size_t(0)
    rt = ctypes.CDLL("libcudart.so.12")
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    g.instantiate()
    return n.value, g


@pytest.mark.parametrize("op,H,nq,nkv,flags,launches", [
    ("mxfp4", 2, 300, 300, 3, 2),        # operands, attention
    ("mxfp4", 2, 300, 300, 11, 3),       # ... and the rotation of Q and K
    ("mxfp4", 38, 1000, 700, 3, 2),      # a wave and a bit, all in one attention launch
    ("mxfp4", 38, 897, 6200, 3, 4),      # Q, K and V apart
    ("mxfp4", 38, 897, 12800, 3, 5),     # ... and a wave of pairs of attention tiles, the rest in small CTAs
    ("mxfp4", 37, 8192, 130, 3, 4),      # Q, K and V quantized apart; whole waves
    ("mxfp4", 38, 8192, 1000, 11, 3),    # rotated; the last wave with the others
    ("mxfp4", 38, 897, 12800, 11, 4),    # ... and in small CTAs
    ("nvfp4", 2, 300, 300, 0, 4),        # zeroing, maxima, operands, attention
    ("nvfp4", 37, 8192, 130, 2, 6),      # Q, K and V apart
    ("bf16", 2, 300, 300, 0, 2),         # zeroing, attention
    ("rowsum", 2, 300, 300, 1, 2),       # operands, diagnostic
    ("rowsum", 2, 300, 300, 9, 3),
])
def test_count_equals_the_captured_kernels(op, H, nq, nkv, flags, launches):
    import paper_2607_24377_b200 as mx
    fn, size = {"mxfp4": (mx.forward_ws, mx.forward_workspace_bytes), "rowsum": (mx.rowsum_diagnostic, mx.forward_workspace_bytes),
                "nvfp4": (mx.forward_nvfp4, mx.forward_nvfp4_workspace_bytes), "bf16": (mx.forward_bf16, mx.forward_bf16_workspace_bytes)}[op]
    q, k, v = (torch.randn(1, H, n, 128, device="cuda").to(torch.bfloat16) for n in (nq, nkv, nkv))
    ws = torch.empty(size(1, H, nq, nkv, 128), dtype=torch.uint8, device="cuda")
    o = torch.empty((1, H, nq, 6) if op == "rowsum" else (1, H, nq, 128), dtype=torch.float32 if op == "rowsum" else torch.bfloat16, device="cuda")
    call = lambda: fn(*((q, k) if op == "rowsum" else (q, k, v)), o, 1, H, nq, nkv, 128, 128 ** -0.5, flags, ws)
    call()
    want = o.clone()
    assert mx.last_launch_count() == launches
    captured, graph = nodes_of(call)
    assert mx.last_launch_count() == captured == launches
    mx.quantize_mxfp4_batched(q, ws, ws[H * nq * 64:], H, nq, 128, 1, mx.MODE_UOS, mx.LAYOUT_CANONICAL)       # not a forward call
    assert mx.last_launch_count() == launches
    o.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(o, want)


@pytest.mark.parametrize("rows,kernels", [(16384, 1), (16385, 2)])       # a cluster per matrix; zeroing and a grid
def test_kernels_of_the_tensor_maximum(rows, kernels):
    import paper_2607_24377_b200 as mx
    x, amax = torch.randn(rows, 128, device="cuda").to(torch.bfloat16), torch.empty(1, device="cuda")
    mx.tensor_amax(x, amax, 1, rows, 128)
    assert nodes_of(lambda: mx.tensor_amax(x, amax, 1, rows, 128))[0] == kernels
