"""Host-buffer forward: every way its heads are cut into pipeline stages gives the device path's result, bit for bit."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Nq,Nkv", [
    (1, 300, 300),        # one stage
    (2, 5000, 5000),      # two stages of one head
    (3, 900, 900),        # less than two stages of the least size
    (23, 2200, 2200),     # copies in are the bound: growing, then shrinking stages
    (13, 6000, 100),      # copies out weigh as much: equal stages
    (9, 130, 9000),       # Q and the output are small
    (4, 19500, 19500),    # two heads are more than a wave: the larger stages first
])
def test_host_stages_equal_the_device_path(H, Nq, Nkv):
    import paper_2607_24377_b200 as mx
    cfg = si.custom_config("stages", 1, H, Nq, Nkv, 1000 * H + Nkv)
    q, k, v = si.make_all(cfg)
    flags = mx.FLAG_UOS | mx.FLAG_PNQ
    out = torch.empty((1, H, Nq, 128), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(mx.forward_workspace_bytes(1, H, Nq, Nkv, 128), dtype=torch.uint8, device="cuda")
    mx.forward_ws(util.to_dev_bf16(q), util.to_dev_bf16(k), util.to_dev_bf16(v), out, 1, H, Nq, Nkv, 128, cfg.softmax_scale, flags, ws)
    assert mx.device_status(ws) == 0
    hq, hk, hv = (torch.from_numpy(x.view(np.int16)).pin_memory() for x in (q, k, v))
    ho = torch.zeros((1, H, Nq, 128), dtype=torch.bfloat16).pin_memory()
    arena = torch.empty(mx.forward_host_arena_bytes(1, H, Nq, Nkv, 128, flags), dtype=torch.uint8, device="cuda")
    mx.forward_host(hq, hk, hv, ho, 1, H, Nq, Nkv, 128, cfg.softmax_scale, flags, arena)
    assert torch.equal(ho.view(torch.int16), out.cpu().view(torch.int16))
