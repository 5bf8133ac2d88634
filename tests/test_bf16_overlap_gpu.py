"""The bf16 forward with an output that overlaps its inputs in memory gives the bits that it gives without."""
import pytest
import torch

from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,nq,nkv", [(40, 700, 700), (5, 300, 1000), (170, 129, 77)])
@pytest.mark.parametrize("f32", [False, True])
def test_output_over_an_input(H, nq, nkv, f32):
    import paper_2607_24377_b200 as mx
    dt, flags = (torch.float32, mx.FLAG_OUT_FP32) if f32 else (torch.bfloat16, 0)
    n = [H * m * 128 for m in (nq, nkv, nkv)]
    pad = 2 * max(n) + 4096                                  # room for an output that starts anywhere in the inputs
    src = torch.randn(sum(n) + pad, device="cuda").to(torch.bfloat16)
    ws = util.guarded(mx.forward_bf16_workspace_bytes(1, H, nq, nkv, 128), torch.uint8)

    def run(at, into):                                       # q, k, v one behind the other in `into`, the output at element `at`
        q, k, v = (into[sum(n[:i]):sum(n[:i + 1])] for i in range(3))
        raw = into if at is not None else torch.empty_like(into)
        o = raw[at or 0:][:n[0] * (2 if f32 else 1)].view(dt)
        mx.forward_bf16(q, k, v, o, 1, H, nq, nkv, 128, 128 ** -0.5, flags, ws.t)
        assert mx.device_status(ws.t) == 0
        ws.check()
        return o.clone()

    want = run(None, src.clone())
    assert bool(torch.isfinite(want).all())
    # exactly over q, k, v; a row, half a tile and 16 bytes into them; over two of them
    for at in (0, n[0], n[0] + n[1], 128, 64 * 128, 8, n[0] - 64 * 128, n[0] + 8, n[0] + n[1] - 128, n[0] + n[1] + 64 * 128):
        assert torch.equal(run(at, src.clone()), want), at


def test_one_buffer_for_all():
    import paper_2607_24377_b200 as mx
    H, n = 40, 700
    x = torch.randn(1, H, n, 128, device="cuda").to(torch.bfloat16)
    ws = torch.empty(mx.forward_bf16_workspace_bytes(1, H, n, n, 128), dtype=torch.uint8, device="cuda")
    want = torch.empty_like(x)
    mx.forward_bf16(x, x, x, want, 1, H, n, n, 128, 128 ** -0.5, 0, ws)
    mx.forward_bf16(x, x, x, x, 1, H, n, n, 128, 128 ** -0.5, 0, ws)
    assert mx.device_status(ws) == 0 and torch.equal(x, want)
