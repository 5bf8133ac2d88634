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
