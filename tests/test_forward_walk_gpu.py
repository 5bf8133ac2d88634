"""The attention kernel whose CTAs walk items of one query tile (two teams of softmax warps take the KV tiles in turn): the same
heads alone, which small CTAs of another kernel compute, and copied often enough that every CTA walks several items.  The KV
tiles of an item are one, two, three (teams change from item to item), as many as buffers come round (4 to 9) and more; query
and key counts end inside a tile, a half and a block."""
import ctypes

import pytest
import torch

import synth_inputs as si
from tests import util


def walk_split(n_sm, heads, nq, nkv, pnq, followed=False):
    """(whether the kernel is used, pairs of query tiles it takes), asked of the library"""
    import paper_2607_24377_b200 as mx

    class Row(ctypes.Structure):
        _fields_ = [("pairs_256", ctypes.c_int64), ("R", ctypes.c_int)]

    class Walk(ctypes.Structure):
        _fields_ = [("walk", ctypes.c_bool), ("pairs", ctypes.c_int64)]

    f = getattr(mx.lib(), "_ZN6mxattn18forward_walk_splitEllllbbRKNS_8RowSplitE")
    f.argtypes, f.restype = [ctypes.c_int64] * 4 + [ctypes.c_bool] * 2 + [ctypes.POINTER(Row)], Walk
    w = f(n_sm, heads, nq, nkv, pnq, followed, ctypes.byref(Row(*util.row_split(n_sm, heads, nq, nkv, pnq))))
    return w.walk, w.pairs


@pytest.mark.parametrize("pnq", [True, False])
def test_what_the_walking_kernel_takes(pnq):
    for heads, nq, nkv in ((1, 1, 1), (2, 1024, 1024), (40, 4096, 4096), (40, 75600, 512), (24, 8192, 8192), (3, 50000, 300)):
        walk, pairs = walk_split(148, heads, nq, nkv, pnq)
        total, (whole, r) = heads * ((-(-nq // 128) + 1) // 2), util.row_split(148, heads, nq, nkv, pnq)
        assert walk and pairs in (whole, total) and (r != 0 or pairs == total)
    assert walk_split(148, 2, 1024, 1024, pnq)[1] == 0                       # small CTAs alone
    assert walk_split(148, 40, 4096, 4096, pnq)[1] == 640                    # nine waves of single tiles, no second launch
    assert walk_split(148, 14, 1300, 777, pnq)[0] == (not pnq) and walk_split(148, 13, 1300, 777, pnq)[0]      # one wave of pairs, two rounds of tiles; one round
    assert walk_split(148, 24, 4096, 6144, pnq, True)[0] and not walk_split(148, 24, 4096, 6145, pnq, True)[0]      # beside other launches
    assert walk_split(148, 40, 256 * 128, 256 * 128, pnq)[0] and walk_split(148, 40, 256, 256 * 128 + 1, pnq)[0] == (not pnq)


def test_few_whole_waves_of_pairs_with_the_direct_row_sum():
    # 74 x 512 and 37 x 4096: exactly one and four waves of pairs, two and eight rounds of single tiles
    for heads, nq in ((74, 512), (37, 4096)):
        assert walk_split(148, heads, nq, 256 * 128, False) == (True, heads * nq // 256)
        assert not walk_split(148, heads, nq, 256 * 128 + 1, False)[0]
    assert walk_split(148, 37, 8192, 600 * 128, False)[0]                    # eight waves
    assert walk_split(148, 14, 1300, 100 * 128, False)[0] and not walk_split(148, 14, 1300, 777, False, True)[0]     # beside other launches
    assert walk_split(148, 3, 6200, 400 * 128, False) == (True, 75)          # 147 single tiles: one round where pairs take one of twice the time


@pytest.mark.parametrize("pnq", [True, False])
def test_last_wave_goes_where_it_is_estimated_to_end_first(pnq):
    # cycles of n single tiles in one walk, and of a launch of small CTAs behind them (the figures stand at the rule)
    rounds = lambda n, t: -(-n // 148) * (t * (1390 if pnq else 1500) + 1000) + 4400
    split = 0
    for heads, nq, nkv in ((38, 1000, 700), (38, 8192, 1000), (51, 700, 300), (38, 897, 6200), (38, 1000, 130), (40, 2000, 1024), (24, 8192, 8192), (39, 897, 6300)):
        whole, r = util.row_split(148, heads, nq, nkv, pnq)
        t, tiles = -(-nkv // 128), -(-nq // 128)
        pairs, groups = (tiles + 1) // 2, -(-nq // (128 // r))
        ahead = whole // pairs * tiles + whole % pairs * 2
        small = -(-(heads * groups - whole // pairs * groups - whole % pairs * 2 * r) // 148) * (t * {4: 1200, 2: 1530, 1: 2125}[r] + 4500)
        one = rounds(heads * tiles, t) <= rounds(ahead, t) + 4000 + small
        assert walk_split(148, heads, nq, nkv, pnq) == (True, heads * pairs if one else whole)
        split += not one
    assert split == 2


def test_what_is_left_for_the_walking_kernel():
    import paper_2607_24377_b200 as mx
    rule = getattr(mx.lib(), "_ZN6mxattn17forward_walk_restEllllbbRKNS_8RowSplitE")
    rule.argtypes, rule.restype = [ctypes.c_int64] * 4 + [ctypes.c_bool] * 2 + [ctypes.c_void_p], ctypes.c_bool
    for heads, nq, nkv, walked in ((14, 1300, 777, True), (37, 1000, 12800, True), (40, 75600, 75600, True), (2, 5000, 40000, True),
                                   (1, 4096, 40000, False), (2, 1024, 1024, False), (1, 6_000_000, 6_000_000, False)):
        split = (ctypes.c_int64 * 2)(*util.row_split(148, heads, nq, nkv, True))
        assert not walk_split(148, heads, nq, nkv, True)[0] or nkv <= 256 * 128
        assert rule(148, heads, nq, nkv, True, False, split) == walked, (heads, nq, nkv)
        direct = (ctypes.c_int64 * 2)(*util.row_split(148, heads, nq, nkv, False))
        assert rule(148, heads, nq, nkv, False, False, direct) == walked, (heads, nq, nkv)
    none = (ctypes.c_int64 * 2)(600, 0)                                      # beside other launches there are no small CTAs
    for pnq in (True, False):
        assert rule(148, 3, 40000, 128 * 128 + 1, pnq, True, none) and not rule(148, 3, 40000, 128 * 128, pnq, True, none)
        assert not rule(148, 3, 7000, 30000, pnq, True, none)


def test_tiles_of_a_cta_are_counted_in_32_bits():
    # one head of n queries and keys with the direct row sum: up to 2^31 - 256 tiles per CTA
    for n, taken in ((72 << 20, False), (73_000_000, False), (64 << 20, True)):
        tiles = -(-n // 128)
        assert (-(-tiles // 148) * tiles <= 0x7FFFFF00) == taken
        assert taken or not walk_split(148, 1, n, n, False)[0]
    # above 48 tiles, where a CTA takes items that others have not begun, they may all be its own
    assert not walk_split(148, 1, 6_000_000, 6_000_000, False)[0] and walk_split(148, 1, 100 << 20, 48 * 128, False)[0]


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
    assert walk_split(n_sm, 3, nq, nkv, pnq)[1] == 0 and walk_split(n_sm, 447, nq, nkv, pnq)[1] > 0
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
    assert walk_split(n_sm, 3, nq, nkv, pnq)[1] == 0 and walk_split(n_sm, 447, nq, nkv, pnq)[1] > 0
    want = outs[0].repeat(1, 149, 1, 1)
    assert not pnq or bool(torch.isfinite(want[0, 0]).all())
    assert torch.equal(torch.isnan(outs[1]), torch.isnan(want))
    assert torch.equal(torch.nan_to_num(outs[1]), torch.nan_to_num(want))


# Above 23 KV tiles the CTAs take one item after another from the grid: several different items each (three heads, so that a CTA
# never sees one head again and again), tile counts that swap the teams' roles from item to item and ones that do not, query and
# key counts that end inside a tile; two launches back to back, and one beside a launch that holds some of the SMs.
@pytest.mark.gpu
@pytest.mark.parametrize("nq,nkv", [(129, 24 * 128), (257, 25 * 128 - 31), (129, 49 * 128), (300, 49 * 128 + 1), (257, 51 * 128 - 31), (385, 64 * 128 + 77), (130, 127 * 128 + 5)])
@pytest.mark.parametrize("uos,pnq,f32", [(True, True, False), (True, False, True), (False, True, True), (False, False, False)])
def test_taken_items_equal_a_single_head(nq, nkv, uos, pnq, f32):
    import paper_2607_24377_b200 as mx
    flags = (mx.FLAG_UOS if uos else 0) | (mx.FLAG_PNQ if pnq else 0) | (mx.FLAG_OUT_FP32 if f32 else 0)
    one = si.custom_config("tk", 1, 3, nq, nkv, 5 + nq)
    q, k, v = (util.to_dev_bf16(x) for x in si.make_all(one))
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert walk_split(n_sm, 3, nq, nkv, pnq)[1] == 0 and walk_split(n_sm, 237, nq, nkv, pnq)[1] > 0
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
@pytest.mark.parametrize("fmt,heads,n,nkv", [("mxfp4", 24, 8192, 8192), ("mxfp4", 40, 4096, 24 * 128), ("nvfp4", 40, 4096, 4096), ("nvfp4", 40, 18900, 512)])
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
def test_long_sequences_equal_small_ctas(nq, nkv):
    """Above 256 KV tiles: one head alone (CTAs of 32 rows), and copied until the walking kernel's CTAs take items from one another."""
    import paper_2607_24377_b200 as mx
    g = torch.Generator(device="cuda"); g.manual_seed(nq)
    q, k, v = (torch.randn(1, 1, n, 128, generator=g, device="cuda", dtype=torch.bfloat16) for n in (nq, nkv, nkv))
    outs = []
    for heads in (1, 76):
        dev = [x.repeat(1, heads, 1, 1).contiguous() for x in (q, k, v)]
        o = util.guarded((1, heads, nq, 128), torch.float32, float("nan"))
        ws = util.guarded(mx.forward_workspace_bytes(1, heads, nq, nkv, 128), torch.uint8)
        mx.forward_ws(*dev, o.t, 1, heads, nq, nkv, 128, 128 ** -0.5, mx.FLAG_UOS | mx.FLAG_PNQ | mx.FLAG_OUT_FP32, ws.t)
        assert mx.device_status(ws.t) == 0
        o.check(); ws.check()
        outs.append(o.t.clone())
    assert util.row_split(torch.cuda.get_device_properties(0).multi_processor_count, 1, nq, nkv, True) == (0, 4)
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
