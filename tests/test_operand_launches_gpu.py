"""The forward call quantizes Q, K and V in shared launches (one for short problems, separate ones for long ones, the
rotating quantizer for Q and K together); its output must equal, bit for bit, the attention launch on operands quantized
one by one through the public quantizer."""
import pytest
import torch

import synth_inputs as si
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,nq,nkv", [(1, 1, 1, 1), (1, 3, 129, 127), (2, 2, 63, 300), (1, 2, 257, 128), (3, 5, 65, 1), (2, 40, 2900, 130)])
@pytest.mark.parametrize("uos,rotate", [(True, False), (False, False), (True, True)])
def test_forward_equals_separately_quantized_operands(B, H, nq, nkv, uos, rotate):
    import paper_2607_24377_b200 as mx
    cfg = si.custom_config("ol", B, H, nq, nkv, 31 + nq)
    dq, dk, dv = (util.to_dev_bf16(x) for x in si.make_all(cfg))
    flags = (mx.FLAG_UOS if uos else 0) | mx.FLAG_PNQ | (mx.FLAG_HADAMARD if rotate else 0)
    want = torch.full((B, H, nq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    ws = torch.full((mx.forward_workspace_bytes(B, H, nq, nkv, 128),), 0xA5, dtype=torch.uint8, device="cuda")
    mx.forward_ws(dq, dk, dv, want, B, H, nq, nkv, 128, cfg.softmax_scale, flags, ws)
    assert mx.device_status(ws) == 0
    mode = (mx.MODE_UOS if uos else mx.MODE_OCP)
    bufs = []
    for x, n, axis in ((dq, nq, 1), (dk, nkv, 1), (dv, nkv, 0)):
        codes, scales = (torch.empty((B * H, -(-n // 128), b), dtype=torch.uint8, device="cuda") for b in (8192, 512))
        mx.quantize_mxfp4_batched(x, codes, scales, B * H, n, 128, axis, mode | (mx.MODE_HADAMARD if rotate and axis == 1 else 0), mx.LAYOUT_TILE)
        bufs += [codes, scales]
    got = torch.full_like(want, float("nan"))
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    mx.forward_prequantized(*bufs, got, B, H, nq, nkv, 128, cfg.softmax_scale, flags, status)
    assert int(status[0].item()) == 0 and torch.equal(got, want) and bool(torch.isfinite(want.float()).all())
