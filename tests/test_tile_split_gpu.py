"""The bf16 and NVFP4 attention kernels give a CTA two query tiles, or one where the last wave would be half empty (and for an
odd head's last tile): the same head alone (one tile per CTA), 148 times (whole waves: two per CTA throughout) and 160 times
(whole waves of two, then one per CTA) must come out the same, bit for bit."""
import pytest
import torch

import synth_inputs as si
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["bf16", "nvfp4_direct", "nvfp4_pnq"])
@pytest.mark.parametrize("nq,nkv", [(129, 128), (256, 300), (300, 1000), (200, 77)])
def test_same_result_however_the_tiles_are_divided(fmt, nq, nkv):
    import paper_2607_24377_b200 as mx
    one = si.custom_config("ts", 1, 1, nq, nkv, 9)
    q, k, v = (util.to_dev_bf16(x) for x in si.make_all(one))
    outs = []
    for heads in (1, 148, 160):
        size, call = ((mx.forward_bf16_workspace_bytes, mx.forward_bf16) if fmt == "bf16" else (mx.forward_nvfp4_workspace_bytes, mx.forward_nvfp4))
        out = util.guarded((1, heads, nq, 128), torch.bfloat16, float("nan"))
        ws = util.guarded(size(1, heads, nq, nkv, 128), torch.uint8)
        call(*(x.expand(1, heads, -1, -1).contiguous() for x in (q, k, v)), out.t, 1, heads, nq, nkv, 128, one.softmax_scale,
             mx.FLAG_PNQ if fmt == "nvfp4_pnq" else 0, ws.t)
        assert mx.device_status(ws.t) == 0
        out.check(); ws.check()
        outs.append(out.t.clone())
    assert bool(torch.isfinite(outs[0].float()).all())
    assert torch.equal(outs[1], outs[0].expand_as(outs[1])) and torch.equal(outs[2], outs[0].expand_as(outs[2]))
