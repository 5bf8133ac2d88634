"""The attention kernel whose CTAs walk items of one query tile (two teams of softmax warps take the KV tiles in turn): the same
heads alone, which small CTAs of another kernel compute, and copied often enough that every CTA walks several items.  The KV
tiles of an item are one, two, three (teams change from item to item), as many as buffers come round (4 to 9) and more; query
and key counts end inside a tile, a half and a block."""
import pytest
import torch

import synth_inputs as si
from tests import util


@pytest.mark.parametrize("pnq", [True, False])
def test_what_the_walking_kernel_takes(pnq):
    for heads, nq, nkv in ((40, 4096, 4096), (40, 75600, 512), (24, 8192, 8192), (40, 75600, 75600), (3, 50000, 300), (14, 1300, 777), (13, 1300, 777),
                           (37, 1000, 12800), (74, 512, 40000), (37, 4096, 33000), (2, 5000, 40000), (3, 6200, 400 * 128), (50, 128, 40000)):
        assert util.plan(148, heads, nq, nkv, pnq) == (heads * ((-(-nq // 128) + 1) // 2), 0) and util.walked(148, heads, nq, nkv, pnq)


@pytest.mark.parametrize("pnq", [True, False])
def test_small_problems_go_to_small_ctas(pnq):
    # one wave of 32 rows, whatever the length; one of 64 rows up to 6 KV tiles (direct row sum 14); none of 128
    for heads, nq, nkv, pairs, r in ((1, 1, 1, 0, 4), (2, 1024, 1024, 0, 4), (1, 4096, 40000, 0, 4), (37, 128, 4096, 0, 4), (37, 129, 768, 0, 2), (1, 4737, 768, 0, 2), (1, 4737, 769, *((19, 0) if pnq else (0, 2))),
                                     (1, 9472, 128, 0, 2), (1, 4737, 14 * 128, *((19, 0) if pnq else (0, 2))), (1, 4737, 1793, 19, 0), (1, 9473, 128, 38, 0), (38, 256, 128, 38, 0), (12, 1300, 128, 72, 0)):
        assert util.plan(148, heads, nq, nkv, pnq) == (pairs, r), (heads, nq, nkv)


@pytest.mark.parametrize("pnq", [True, False])
def test_last_wave_goes_where_it_is_estimated_to_end_first(pnq):
    # a few pairs more than a wave: their rounds of single tiles, or a second launch of CTAs of 32 rows, from 72 (direct row sum 29) KV tiles on
    last = 71 if pnq else 28
    for heads, nq in ((38, 1000), (1, 152 * 256), (39, 897), (2, 379 * 256)):
        total = heads * ((-(-nq // 128) + 1) // 2)
        for t in (1, 6, last, last + 1, 100, 300):
            assert util.plan(148, heads, nq, t * 128, pnq) == ((total, 0) if t <= last else (total // 148 * 148, 4)), (heads, nq, t)
    assert util.plan(148, 1, 186 * 256, 12800, pnq) == (186, 0)              # 38 pairs are more than a wave of 32 rows
    assert util.plan(148, 25, 1500, 12800, pnq)[1] == 4 and util.plan(148, 30, 1150, 12800, pnq) == (150, 0)      # odd heads: 270 tiles are two rounds either way


@pytest.mark.parametrize("pnq", [True, False])
def test_beside_other_launches(pnq):
    for heads, nq, nkv, by_walk in ((24, 4096, 6144, True), (24, 4096, 6145, False), (14, 1300, 777, False), (13, 1300, 777, True), (3, 40000, 128 * 128, False),
                                    (3, 40000, 128 * 128 + 1, True), (3, 7000, 30000, False), (1, 1, 1, True)):
        assert util.plan(148, heads, nq, nkv, pnq, True) == (heads * ((-(-nq // 128) + 1) // 2), 0)      # no small CTAs
        assert util.walked(148, heads, nq, nkv, pnq, True) == by_walk, (heads, nq, nkv)


def test_tiles_of_a_cta_are_counted_in_32_bits():
    # above 48 tiles, where a CTA takes items that others have not begun, they may all be its own; with fixed shares it has its own only
    for n, nkv, by_walk in ((72 << 20, 72 << 20, False), (6_000_000, 6_000_000, False), (5_900_000, 5_900_000, True), (1 << 30, 49 * 128, True), (1 << 36, 20 * 128, True)):
        tiles, t = -(-n // 128), -(-nkv // 128)
        assert ((tiles if t > 48 else -(-tiles // 148)) * t <= 0x7FFFFF00) == by_walk
        for pnq in (True, False):
            assert util.walked(148, 1, n, nkv, pnq) == by_walk and util.plan(148, 1, n, nkv, pnq)[0] == (tiles + 1) // 2


@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(1, 1), (129, 128), (300, 200), (128, 257), (257, 384), (100, 511), (640, 700), (385, 1000), (200, 1152), (300, 5000)])
@pytest.mark.parametrize("uos,pnq,f32", [(True, True, False), (True, False, True), (False, True, True), (False, False, False)])
def test_walked_items_equal_a_single_head(nq, nkv, uos, pnq, f32):
    import paper_2607_24377_b200 as mx
    flags = (mx.FLAG_UOS if uos else 0) | (mx.FLAG_PNQ if pnq else 0) | (mx.FLAG_OUT_FP32 if f32 else 0)
    one = si.custom_config("wk", 1, 3, nq, nkv, 3 + nq)
    q, k, v = si.make_all(one)
    outs = []
    for copies in (1, 149):                                                  # 447 heads: three to fifteen items per CTA, not a whole number
        heads = 3 * copies
        dev = [util.to_dev_bf16(x).repeat(1, copies, 1, 1).contiguous() for x in (q, k, v)]
        out = util.guarded((1, heads, nq, 128), torch.float32 if f32 else torch.bfloat16, float("nan"))
        ws = util.guarded(mx.forward_workspace_bytes(1, heads, nq, nkv, 128), torch.uint8)
        for _ in range(2):                                                   # the second launch follows the first closely
            mx.forward_ws(*dev, out.t, 1, heads, nq, nkv, 128, one.softmax_scale, flags, ws.t)
        assert mx.device_status(ws.t) == 0
        out.check(); ws.check()
        outs.append(out.t.clone())
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert util.plan(n_sm, 3, nq, nkv, pnq)[0] == 0 and util.plan(n_sm, 447, nq, nkv, pnq)[0] > 0
    assert n_sm % (3 * -(-nq // 128)) != 0                                   # a CTA's items differ from one another
    assert bool(torch.isfinite(outs[0].float()).all())
    assert torch.equal(outs[1], outs[0].repeat(1, 149, 1, 1))


@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(1, 700), (300, 700), (300, 128)])
@pytest.mark.parametrize("pnq", [True, False])
def test_scores_that_are_not_numbers(nq, nkv, pnq):
    """Given operands may carry the E8M0 code of NaN: here the scales of one head's first KV tile, and of one query of another.
    A tile that has no maximum leaves the running one at -inf, in whichever kernel the row is computed, and the next tile's maximum
    then drops what came before (with the row sum from the quantized probabilities, which are finite)."""
    import paper_2607_24377_b200 as mx
    one = si.custom_config("nn", 1, 3, nq, nkv, 9)
    ops = []
    for x, n, axis in zip(si.make_all(one), (nq, nkv, nkv), (1, 1, 0)):
        codes = torch.empty((3, -(-n // 128), 8192), dtype=torch.uint8, device="cuda")
        scales = torch.empty((3, -(-n // 128), 512), dtype=torch.uint8, device="cuda")
        mx.quantize_mxfp4_batched(util.to_dev_bf16(x), codes, scales, 3, n, 128, axis, mx.MODE_UOS, mx.LAYOUT_TILE)
        ops += [codes, scales]
    ops[3][0, 0] = 255
    ops[1][1, 0, util.tile_scale_offset(0, 0)] = 255
    flags, outs = mx.FLAG_UOS | (mx.FLAG_PNQ if pnq else 0) | mx.FLAG_OUT_FP32, []
    for copies in (1, 149):
        out = torch.empty((1, 3 * copies, nq, 128), device="cuda")
        status = torch.zeros(4, dtype=torch.int32, device="cuda")
        mx.forward_prequantized(*(x.repeat(copies, 1, 1) for x in ops), out, 1, 3 * copies, nq, nkv, 128, one.softmax_scale, flags, status)
        assert int(status[0]) == 0
        outs.append(out)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert util.plan(n_sm, 3, nq, nkv, pnq)[0] == 0 and util.plan(n_sm, 447, nq, nkv, pnq)[0] > 0
    want = outs[0].repeat(1, 149, 1, 1)
    assert not pnq or bool(torch.isfinite(want[0, 0]).all())
    assert torch.equal(torch.isnan(outs[1]), torch.isnan(want))
    assert torch.equal(torch.nan_to_num(outs[1]), torch.nan_to_num(want))


# Above 48 KV tiles the CTAs take one item after another from the grid: several different items each (three heads, so that a CTA
# never sees one head again and again), tile counts that swap the teams' roles from item to item and ones that do not, query and
# key counts that end inside a tile; two launches back to back, and one beside a launch that holds some of the SMs.
@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(129, 49 * 128), (300, 49 * 128 + 1), (257, 51 * 128 - 31), (385, 64 * 128 + 77), (130, 127 * 128 + 5)])
@pytest.mark.parametrize("uos,pnq,f32", [(True, True, False), (True, False, True), (False, True, True), (False, False, False)])
def test_taken_items_equal_a_single_head(nq, nkv, uos, pnq, f32):
    import paper_2607_24377_b200 as mx
    flags = (mx.FLAG_UOS if uos else 0) | (mx.FLAG_PNQ if pnq else 0) | (mx.FLAG_OUT_FP32 if f32 else 0)
    one = si.custom_config("tk", 1, 3, nq, nkv, 5 + nq)
    q, k, v = (util.to_dev_bf16(x) for x in si.make_all(one))
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert util.plan(n_sm, 3, nq, nkv, pnq)[0] == 0 and util.plan(n_sm, 237, nq, nkv, pnq)[0] > 0
    assert n_sm % (3 * -(-nq // 128)) != 0

    def run(copies, beside=None):
        heads = 3 * copies
        dev = [x.repeat(1, copies, 1, 1).contiguous() for x in (q, k, v)]
        out = util.guarded((1, heads, nq, 128), torch.float32 if f32 else torch.bfloat16, float("nan"))
        ws = util.guarded(mx.forward_workspace_bytes(1, heads, nq, nkv, 128), torch.uint8)
        torch.cuda.synchronize()
        if beside is not None:
            beside()
        for _ in range(2):
            mx.forward_ws(*dev, out.t, 1, heads, nq, nkv, 128, one.softmax_scale, flags, ws.t)
        assert mx.device_status(ws.t) == 0
        out.check(); ws.check()
        return out.t.clone()

    want = run(1).repeat(1, 79, 1, 1)
    assert bool(torch.isfinite(want.float()).all())
    assert torch.equal(run(79), want)
    side, long_kv = torch.cuda.Stream(), 400_000                             # 4 groups of rows: 4 CTAs that take 2 ms
    lq, lk, lv = (torch.randn(1, 1, n, 128, device="cuda").to(torch.bfloat16) for n in (128, long_kv, long_kv))
    lo, lws = torch.empty_like(lq), torch.empty(mx.forward_workspace_bytes(1, 1, 128, long_kv, 128), dtype=torch.uint8, device="cuda")

    def hold():
        with torch.cuda.stream(side):
            mx.forward_ws(lq, lk, lv, lo, 1, 1, 128, long_kv, 128, one.softmax_scale, mx.FLAG_UOS | mx.FLAG_PNQ, lws)

    got = run(79, hold)
    side.synchronize()                                                       # before its buffers go
    assert torch.equal(got, want) and mx.device_status(lws) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("fmt,heads,n,nkv", [("mxfp4", 24, 8192, 8192), ("nvfp4", 40, 4096, 4096), ("nvfp4", 40, 18900, 512)])
def test_a_launch_that_holds_few_sms_does_not_hold_up_whole_shares(fmt, heads, n, nkv):
    """24 heads of 8192: ten and a half items per SM.  Beside 4 CTAs that run for 8 ms, the items of those 4 SMs are
    spread over the others (about 1.1 times the time alone); with shares that are fixed at the launch they come last (1.5 to 1.6 times)."""
    import paper_2607_24377_b200 as mx
    mk = lambda h, n: torch.randn(1, h, n, 128, device="cuda").to(torch.bfloat16)
    q, k, v = mk(heads, n), mk(heads, nkv), mk(heads, nkv)
    lq, lk, lv = mk(1, 128), mk(1, 1 << 21), mk(1, 1 << 21)
    o, lo = torch.empty_like(q), torch.empty_like(lq)
    call, size = (mx.forward_ws, mx.forward_workspace_bytes) if fmt == "mxfp4" else (mx.forward_nvfp4, mx.forward_nvfp4_workspace_bytes)
    ws, lws = (torch.empty(f(1, *a, 128), dtype=torch.uint8, device="cuda") for f, a in ((size, (heads, n, nkv)), (mx.forward_workspace_bytes, (1, 128, 1 << 21))))
    side, flags = torch.cuda.Stream(), mx.FLAG_UOS | mx.FLAG_PNQ

    def timed():
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call(q, k, v, o, 1, heads, n, nkv, 128, 128 ** -0.5, flags if fmt == "mxfp4" else mx.FLAG_PNQ, ws)
        b.record(); b.synchronize()
        return a.elapsed_time(b)

    def hold():
        with torch.cuda.stream(side):
            mx.forward_ws(lq, lk, lv, lo, 1, 1, 128, 1 << 21, 128, 128 ** -0.5, flags, lws)

    hold(); timed(); torch.cuda._sleep(1)                                    # kernels are loaded
    alone, beside = [], []
    for _ in range(5):
        torch.cuda.synchronize()
        alone.append(timed())
        torch.cuda.synchronize()
        hold()
        torch.cuda._sleep(1_000_000)                                         # its attention has started
        beside.append(timed())
        still = not side.query()
        side.synchronize()                                                   # before its buffers go
        assert still                                                         # it ran all the while
    assert sorted(beside)[2] < 1.35 * sorted(alone)[2]


@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(130, 256 * 128 + 1), (257, 300 * 128)])
@pytest.mark.parametrize("pnq", [True, False])
def test_long_sequences_equal_small_ctas(nq, nkv, pnq):
    """Above 256 KV tiles: one head alone (CTAs of 32 rows), and copied until the walking kernel's CTAs take items from one another."""
    import paper_2607_24377_b200 as mx
    g = torch.Generator(device="cuda"); g.manual_seed(nq)
    q, k, v = (torch.randn(1, 1, n, 128, generator=g, device="cuda", dtype=torch.bfloat16) for n in (nq, nkv, nkv))
    outs = []
    for heads in (1, 76):
        dev = [x.repeat(1, heads, 1, 1).contiguous() for x in (q, k, v)]
        o = util.guarded((1, heads, nq, 128), torch.float32, float("nan"))
        ws = util.guarded(mx.forward_workspace_bytes(1, heads, nq, nkv, 128), torch.uint8)
        mx.forward_ws(*dev, o.t, 1, heads, nq, nkv, 128, 128 ** -0.5, mx.FLAG_UOS | (mx.FLAG_PNQ if pnq else 0) | mx.FLAG_OUT_FP32, ws.t)
        assert mx.device_status(ws.t) == 0
        o.check(); ws.check()
        outs.append(o.t.clone())
    assert util.plan(torch.cuda.get_device_properties(0).multi_processor_count, 1, nq, nkv, pnq) == (0, 4)
    assert bool(torch.isfinite(outs[0]).all()) and torch.equal(outs[1], outs[0].expand_as(outs[1]))


@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(1, 1), (129, 128), (300, 200), (128, 257), (257, 384), (100, 511), (640, 700), (200, 1152), (130, 48 * 128 + 3)])
@pytest.mark.parametrize("pnq,f32", [(True, False), (False, True), (True, True), (False, False)])
def test_walked_nvfp4_items_equal_single_heads(nq, nkv, pnq, f32):
    """NVFP4: heads of different tensor scales alone (one item per CTA), and copied until every CTA walks items of several heads."""
    import paper_2607_24377_b200 as mx
    one = si.custom_config("wn", 1, 3, nq, nkv, 5 + nq)
    q, k, v = (util.to_dev_bf16(x) * torch.tensor([1.0, 0.125, 6.0], device="cuda").view(1, 3, 1, 1).bfloat16() for x in si.make_all(one))
    flags = (mx.FLAG_PNQ if pnq else 0) | (mx.FLAG_OUT_FP32 if f32 else 0)
    outs = []
    for copies in (1, 149):
        heads = 3 * copies
        dev = [x.repeat(1, copies, 1, 1).contiguous() for x in (q, k, v)]
        o = util.guarded((1, heads, nq, 128), torch.float32 if f32 else torch.bfloat16, float("nan"))
        ws = util.guarded(mx.forward_nvfp4_workspace_bytes(1, heads, nq, nkv, 128), torch.uint8)
        for _ in range(2):
            mx.forward_nvfp4(*dev, o.t, 1, heads, nq, nkv, 128, one.softmax_scale, flags, ws.t)
        assert mx.device_status(ws.t) == 0
        o.check(); ws.check()
        outs.append(o.t.clone())
    assert bool(torch.isfinite(outs[0].float()).all())
    assert torch.equal(outs[1], outs[0].repeat(1, 149, 1, 1))
