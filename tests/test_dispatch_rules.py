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
    for heads, nq, nkv in ((1, 1, 1), (2, 1024, 1024), (38, 1000, 700), (40, 4096, 4096), (3, 50000, 300)):
        total = heads * ((-(-nq // 128) + 1) // 2)
        pairs, r = util.row_split(n_sm, heads, nq, nkv, pnq)
        assert r in (0, 1, 2, 4)
        assert pairs == (total if r == 0 else total // n_sm * n_sm)          # whole waves, or everything
    assert util.row_split(n_sm, n_sm, 256, 1024, pnq) == (n_sm, 0)            # exactly a wave
    assert util.row_split(n_sm, 1, 32, 1024, pnq) == (0, 4)                   # a single group of rows
