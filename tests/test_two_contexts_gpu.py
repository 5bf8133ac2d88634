"""Kernels that need an attribute (dynamic shared memory, clusters of 16) run in every context of a device, not only in the one
that called them first."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_second_context_of_a_device():
    import paper_2607_24377_b200 as mx
    L, cu = mx.lib(), ctypes.CDLL("libcuda.so.1")
    H, n, flags = 2, 300, mx.FLAG_UOS | mx.FLAG_PNQ | mx.FLAG_HADAMARD
    g = torch.Generator()
    g.manual_seed(3)
    host = torch.randn(H * n * 128, generator=g).to(torch.bfloat16)
    # in torch's context first: rotating quantizer, attention, tensor maximum by clusters
    x, o = host.cuda(), torch.empty(H * n * 128, dtype=torch.bfloat16, device="cuda")
    size = mx.forward_workspace_bytes(1, H, n, n, 128)
    ws, amax = torch.empty(size, dtype=torch.uint8, device="cuda"), torch.empty(H, device="cuda")
    mx.forward_ws(x, x, x, o, 1, H, n, n, 128, 128 ** -0.5, flags, ws)
    mx.tensor_amax(x, amax, H, n, 128)
    want, want_amax = o.cpu(), amax.cpu()

    def ok(rc):
        assert rc == 0, rc

    ctx, old = ctypes.c_void_p(), ctypes.c_void_p()
    ok(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, 0))                   # becomes current
    try:
        bufs = []
        for nbytes in (host.numel() * 2, host.numel() * 2, size, 256):
            p = ctypes.c_uint64()
            ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(nbytes)))
            bufs.append(p.value)
        dx, do, dws, damax = bufs
        ok(cu.cuMemcpyHtoD_v2(ctypes.c_uint64(dx), ctypes.c_void_p(host.data_ptr()), ctypes.c_size_t(host.numel() * 2)))
        for _ in range(2):
            ok(L.mxattn_forward_ws(dx, dx, dx, do, 1, H, n, n, 128, 128 ** -0.5, flags, dws, size, None))
            ok(L.mxattn_tensor_amax(dx, damax, H, n, 128, None))
        got, got_amax = torch.empty_like(want), torch.empty_like(want_amax)
        ok(cu.cuMemcpyDtoH_v2(ctypes.c_void_p(got.data_ptr()), ctypes.c_uint64(do), ctypes.c_size_t(got.numel() * 2)))
        ok(cu.cuMemcpyDtoH_v2(ctypes.c_void_p(got_amax.data_ptr()), ctypes.c_uint64(damax), ctypes.c_size_t(4 * H)))
    finally:
        ok(cu.cuCtxPopCurrent_v2(ctypes.byref(old)))
        ok(cu.cuCtxDestroy_v2(ctx))
    assert torch.equal(got, want) and torch.equal(got_amax, want_amax)
    mx.forward_ws(x, x, x, o.fill_(0), 1, H, n, n, 128, 128 ** -0.5, flags, ws)       # and the first one still works
    assert torch.equal(o.cpu(), want)
