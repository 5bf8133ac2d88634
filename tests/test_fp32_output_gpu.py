"""fp32 output of the attention kernels: the bf16 output is its rounding, element for element, and rows behind the last one
are not touched -- at query counts around the 32-row boxes that the result leaves in, with one CTA per work item, with CTAs
that walk several, and with few query rows per CTA."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["mxfp4", "nvfp4", "bf16"])
@pytest.mark.parametrize("BH,Nq,Nkv", [(1, 1, 40), (2, 33, 300), (3, 1000, 100), (60, 1281, 200), (60, 1311, 130), (30, 2100, 640)])
def test_bf16_output_is_the_rounded_fp32_output(op, BH, Nq, Nkv):
    import paper_2607_24377_b200 as mx
    g = torch.Generator(device="cuda")
    g.manual_seed(100 * Nq + Nkv)
    q, k, v = (torch.randn(1, BH, n, 128, generator=g, device="cuda").to(torch.bfloat16) for n in (Nq, Nkv, Nkv))
    fn, size = {"mxfp4": (mx.forward_ws, mx.forward_workspace_bytes), "nvfp4": (mx.forward_nvfp4, mx.forward_nvfp4_workspace_bytes),
                "bf16": (mx.forward_bf16, mx.forward_bf16_workspace_bytes)}[op]
    ws = torch.empty(size(1, BH, Nq, Nkv, 128), dtype=torch.uint8, device="cuda")
    out = []
    for dt, extra in ((torch.bfloat16, 0), (torch.float32, mx.FLAG_OUT_FP32)):
        o = torch.full((BH * Nq + 64, 128), float("nan"), dtype=dt, device="cuda")
        fn(q, k, v, o, 1, BH, Nq, Nkv, 128, 128 ** -0.5, (mx.FLAG_UOS | mx.FLAG_PNQ if op == "mxfp4" else 0) | extra, ws)
        assert bool(torch.isnan(o[BH * Nq:]).all())
        out.append(o[:BH * Nq])
    assert torch.equal(out[1].to(torch.bfloat16), out[0])
