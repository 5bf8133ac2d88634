"""The rules that choose between kernels, asked directly (they are functions of sizes; no GPU needed)."""
import ctypes

import pytest


def rule(name, *argtypes, restype=ctypes.c_bool):
    import paper_2607_24377_b200 as mx
    f = getattr(mx.lib(), name)
    f.argtypes, f.restype = argtypes, restype
    return f


@pytest.mark.parametrize("batch,chunks,form", [(1, 1, True), (1, 1 << 18, True), (1, (1 << 18) + 1, False), (40, 18022, True), (40, 18023, False)])
def test_tensor_maximum_by_clusters_only_where_they_fit(batch, chunks, form):
    # chunks of 16 bytes: up to 4 MiB per matrix and 11 MiB in all; never where a cluster of 16 cannot run
    by_cluster = rule("_ZN6mxattn15amax_by_clusterEllb", ctypes.c_int64, ctypes.c_int64, ctypes.c_bool)
    assert by_cluster(batch, chunks, True) == form
    assert not by_cluster(batch, chunks, False)


@pytest.mark.parametrize("n_sm", [148, 132, 40])
@pytest.mark.parametrize("pnq", [True, False])
def test_last_wave_is_divided_for_the_sms_that_there_are(n_sm, pnq):
    from tests import util
    divided = 0
    for heads, nq, nkv in ((1, 1, 1), (2, 1024, 1024), (38, 1000, 700), (40, 4096, 4096), (3, 50000, 300), (1, 256 * n_sm + 300, 12800), (n_sm, 200, 12800)):
        total = heads * ((-(-nq // 128) + 1) // 2)
        pairs, r = util.plan(n_sm, heads, nq, nkv, pnq)
        assert r in (0, 2, 4)
        assert pairs == (total if r == 0 else total // n_sm * n_sm)          # whole waves, or everything
        divided += r > 0 and pairs > 0
    assert divided == 1
    assert util.plan(n_sm, n_sm, 256, 1024, pnq) == (n_sm, 0)                 # exactly a wave
    assert util.plan(n_sm, 1, 32, 1024, pnq) == (0, 4)                        # a single group of rows


def stages(heads, nq, nkv, n_sm=148):
    f = rule("_ZN6mxattn11host_stagesEmllmmiPmPb", ctypes.c_size_t, ctypes.c_int64, ctypes.c_int64, ctypes.c_size_t, ctypes.c_size_t, ctypes.c_int,
             ctypes.POINTER(ctypes.c_size_t), ctypes.POINTER(ctypes.c_bool), restype=ctypes.c_size_t)
    first, alone = (ctypes.c_size_t * (heads + 1))(), ctypes.c_bool()
    n = f(heads, nq, nkv, 256 * (nq + 2 * nkv), 256 * nq, n_sm, first, ctypes.byref(alone))
    assert first[0] == 0 and first[n] == heads
    return [first[i + 1] - first[i] for i in range(n)]


def test_stages_of_the_host_form():
    for heads in (*range(1, 20), 40, 160):                    # every head once, no empty stage, whatever the sizes
        for nq, nkv in ((1, 1), (300, 300), (8192, 8192), (18000, 18000), (21070, 21070), (28000, 28000), (75600, 512), (130, 9000), (75600, 75600)):
            s = stages(heads, nq, nkv)
            assert min(s) >= 1 and sum(s) == heads
    # two heads fit the SMs: sizes double or halve towards the end; they do not, and heads are few: two single ones at the end
    assert stages(4, 18000, 18000) == [1, 2, 1] and stages(24, 8192, 8192) == [3, 6, 8, 4, 2, 1]
    assert stages(4, 21070, 21070) == [2, 1, 1] and stages(5, 28000, 28000) == [1, 2, 1, 1] and stages(6, 24000, 24000) == [1, 1, 2, 1, 1]
    assert stages(4, 21070, 21070, n_sm=300) == [1, 2, 1] and stages(12, 21070, 21070)[-2:] == [2, 1]
