"""The attention kernel for few query rows (128/R rows per CTA, R = 4 or 2, replicated R times down the operand tile):
against the oracle at its edges, and bit for bit against the walking kernel, which the same heads reach when many copies of
them fill the GPU."""
import numpy as np
import pytest
import torch

import synth_inputs as si
from oracle import attention
from tests import util

pytestmark = pytest.mark.gpu


def run(cfg, q, k, v, flags):
    import paper_2607_24377_b200 as mx
    f32 = bool(flags & mx.FLAG_OUT_FP32)
    out = util.guarded((cfg.B, cfg.H, cfg.Nq, 128), torch.float32 if f32 else torch.bfloat16, float("nan"))
    ws = util.guarded(mx.forward_workspace_bytes(cfg.B, cfg.H, cfg.Nq, cfg.Nkv, 128), torch.uint8)
    mx.forward_ws(*(util.to_dev_bf16(x) for x in (q, k, v)), out.t, cfg.B, cfg.H, cfg.Nq, cfg.Nkv, 128, cfg.softmax_scale, flags, ws.t)
    assert mx.device_status(ws.t) == 0
    out.check(); ws.check()
    return out.t.clone()


def rows_per_cta(heads, nq, nkv, pnq):
    """(pairs of query tiles that are walked, R of the rest) on this device"""
    return util.plan(torch.cuda.get_device_properties(0).multi_processor_count, heads, nq, nkv, pnq)


# R = 4 (few heads) or 2 (50 and 70 heads), and single tiles walked (20 heads); query counts around the row groups, key counts around blocks and tiles
@pytest.mark.parametrize("H,nq,nkv", [(1, 1, 1), (2, 31, 33), (2, 33, 128), (1, 97, 129), (3, 64, 640), (1, 160, 1100),
                                      (50, 127, 300), (70, 65, 31), (20, 449, 257)])
@pytest.mark.parametrize("uos,pnq", [(True, True), (False, False)])
def test_against_the_oracle(H, nq, nkv, uos, pnq):
    import paper_2607_24377_b200 as mx
    cfg = si.custom_config("rw", 1, H, nq, nkv, 17 + nq + nkv)
    q, k, v = si.make_all(cfg)
    got = run(cfg, q, k, v, (mx.FLAG_UOS if uos else 0) | (mx.FLAG_PNQ if pnq else 0) | mx.FLAG_OUT_FP32).double().cpu().numpy()
    want = attention.forward(*(util.bits_to_f64(x) for x in (q, k, v)), cfg.softmax_scale, uos, pnq)
    assert np.isfinite(got).all()
    assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want) and np.abs(got - want).max() <= 4e-3


@pytest.mark.parametrize("heads", [2, 40])
@pytest.mark.parametrize("f32", [False, True])
def test_bit_identical_to_many_copies(heads, f32):
    import paper_2607_24377_b200 as mx
    flags = mx.FLAG_UOS | mx.FLAG_PNQ | (mx.FLAG_OUT_FP32 if f32 else 0)
    one = si.custom_config("rb", 1, heads, 300, 700, 5)
    q, k, v = si.make_all(one)
    assert rows_per_cta(heads, 300, 700, True) == ((0, 4) if heads == 2 else (80, 0))
    want = run(one, q, k, v, flags)
    many = si.custom_config("rm", 640 // heads, heads, 300, 700, 5)    # 1280 pairs of query tiles
    rep = lambda x: np.ascontiguousarray(np.broadcast_to(x, (many.B,) + x.shape[1:]))
    got = run(many, rep(q), rep(k), rep(v), flags)
    assert torch.equal(got, want.expand_as(got))


# 152 to 156 pairs of query tiles: the second wave would be nearly empty.  At 100 KV tiles (50 with the direct row sum) whole waves are
# walked and the pairs behind them are cut into small CTAs; at fewer the walking kernel takes them all (the last head's tiles ragged)
@pytest.mark.parametrize("heads,nq,nkv", [(38, 1000, 700), (39, 897, 6300), (39, 897, 12711), (51, 700, 300)])
@pytest.mark.parametrize("pnq", [True, False])
def test_last_wave_cut_into_small_ctas(heads, nq, nkv, pnq):
    import paper_2607_24377_b200 as mx
    flags = mx.FLAG_UOS | (mx.FLAG_PNQ if pnq else 0)
    one = si.custom_config("lw", 1, 1, nq, nkv, 6)
    q, k, v = si.make_all(one)
    want = run(one, q, k, v, flags)
    divided = nkv > (9000 if pnq else 6000)
    assert rows_per_cta(1, nq, nkv, pnq) == (0, 4) and rows_per_cta(heads, nq, nkv, pnq) == ((148, 4) if divided else (heads * -(-nq // 256), 0))
    many = si.custom_config("lm", 1, heads, nq, nkv, 6)
    rep = lambda x: np.ascontiguousarray(np.broadcast_to(x, (1, heads) + x.shape[2:]))
    assert torch.equal(run(many, rep(q), rep(k), rep(v), flags), want.expand(1, heads, nq, 128))


# 64 rows per CTA (70 x 1100 with PNQ and from 44 heads on: walked): every head must come out as it does among 148, which are walked
@pytest.mark.parametrize("heads,nq,nkv,split", [(49, 127, 300, (0, 2)), (70, 65, 1100, (70, 0)), (49, 128, 640, (0, 2)), (60, 127, 6 * 128, (0, 2)),
                                                (44, 1000, 700, (176, 0)), (45, 897, 1300, (180, 0)), (50, 1000, 700, (200, 0))])
@pytest.mark.parametrize("pnq", [True, False])
def test_64_rows_per_cta_equal_the_walking_kernel(heads, nq, nkv, split, pnq):
    import paper_2607_24377_b200 as mx
    flags = mx.FLAG_UOS | (mx.FLAG_PNQ if pnq else 0)
    assert rows_per_cta(heads, nq, nkv, pnq) == ((0, 2) if nkv == 1100 and not pnq else split) and rows_per_cta(148, nq, nkv, pnq)[1] == 0
    few = si.custom_config("h64", 1, heads, nq, nkv, 8)
    q, k, v = si.make_all(few)
    got = run(few, q, k, v, flags)
    many = si.custom_config("h64m", 1, 148, nq, nkv, 8)
    rep = lambda x: np.ascontiguousarray(x[:, np.arange(148) % heads])
    assert torch.equal(run(many, rep(q), rep(k), rep(v), flags)[:, :heads], got)


# Every way a problem is divided, by the rule of the launch itself: how many pairs of query tiles are walked, and R of the small CTAs
# behind them (0: none).  Each of three heads comes out as it does alone.
@pytest.mark.parametrize("heads,nq,nkv,pnq,way", [
    (50, 129, 31, True, (50, 0)), (50, 129, 31, False, (50, 0)), (120, 127, 127, True, (120, 0)), (50, 129, 33000, True, (50, 0)),
    (50, 65, 31, True, (0, 2)), (50, 65, 31, False, (0, 2)), (50, 65, 33000, True, (50, 0)),
    (38, 897, 6200, True, (152, 0)), (38, 897, 6200, False, (148, 4)), (38, 897, 12800, True, (148, 4)), (38, 897, 33000, True, (148, 4)), (38, 897, 33000, False, (148, 4)),
    (50, 513, 33000, True, (150, 0)), (64, 513, 33000, True, (192, 0)), (70, 513, 33000, True, (210, 0)),
    (50, 257, 33000, True, (100, 0)), (50, 257, 33000, False, (100, 0)), (14, 1300, 777, True, (84, 0)),
    (14, 1300, 777, False, (84, 0)), (50, 513, 31, True, (150, 0)), (50, 513, 33000, False, (150, 0))])
def test_every_division_equals_single_heads(heads, nq, nkv, pnq, way):
    import paper_2607_24377_b200 as mx
    flags = mx.FLAG_UOS | (mx.FLAG_PNQ if pnq else 0)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert util.walked(n_sm, heads, nq, nkv, pnq) and (n_sm != 148 or rows_per_cta(heads, nq, nkv, pnq) == way)
    want = []
    for h in range(3):
        one = si.custom_config("dv", 1, 1, nq, nkv, 21 + h)
        qkv = si.make_all(one)
        want.append((qkv, run(one, *qkv, flags)))
    many = si.custom_config("dvm", 1, heads, nq, nkv, 21)
    of = np.arange(heads) % 3
    got = run(many, *(np.concatenate([w[0][i] for w in want], axis=1)[:, of] for i in range(3)), flags)
    assert torch.equal(got, torch.cat([w[1] for w in want], dim=1)[:, torch.from_numpy(of).cuda()])
