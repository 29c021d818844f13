"""Kernel launches of a TSMTTSM call by variant: the row variants always end in
the final kernel, also where the partials of the grid are few; the others as
the shape and the grid say."""

import os

import pytest


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


@pytest.mark.parametrize("dt,name", [(0, "r64"), (1, "c64")])
def test_launches_by_variant(tsm, dt, name):
    lib = tsm.load()
    index = {v["name"]: v["index"] for v in tsm.variants(tsm.KIND_TSMTTSM)}
    row, direct = index["tsmttsm_%s_row" % name], index["tsmttsm_%s_direct_t1x1_u4" % name]
    count = lib.tsm_tsmttsm_variant_kernels
    for M, N, grid in ((1, 1, 1), (4, 4, 152), (16, 16, 128), (16, 16, 129)):
        assert count(row, dt, M, N, grid) == 2
        assert count(direct, dt, M, N, grid) == lib.tsm_tsmttsm_kernels_per_call(dt, M, N, grid)
    assert count(row, dt, 0, 4, 152) == count(row, dt, 4, 4, 0) == count(-1, dt, 4, 4, 152) == -1
    assert count(row, 1 - dt, 4, 4, 152) == count(len(index), dt, 4, 4, 152) == -1
