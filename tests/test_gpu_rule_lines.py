"""The dispatch at calls that the row kernels had slowed down: they keep, or
get back, the kernel or the grid that was measured to be the faster one, and
their neighbours on the other side of each line stay with the row kernel."""

import os

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


def _choice(tsm, kind, cplx, M, N, K):
    names = {v["index"]: v["name"] for v in tsm.variants(kind)}
    v, grid = tsm.choose(kind, cplx, M, N, K)
    return names[v].endswith("_row"), grid


@pytest.mark.parametrize("cplx,M,N,K", [(1, 50, 13, 5163793), (1, 22, 15, 4920029), (1, 9, 7, 5163793), (0, 11, 23, 6419820)])
def test_long_tsmttsm_stays(tsm, cplx, M, N, K):
    assert not _choice(tsm, tsm.KIND_TSMTTSM, cplx, M, N, K)[0]


@pytest.mark.parametrize("cplx,M,N,K,per_sm", [
    (1, 2, 12, 78231, 1), (1, 5, 2, 1294916, 2),   # two CTAs fill the register file, or leave room
    (0, 35, 35, 19610, 1), (0, 5, 59, 68213, 2),   # wide CTAs with long strips, few rows or more
    (0, 64, 2, 334665, 3), (0, 32, 5, 398825, 2),  # from DRAM with few FMAs per set of rows, or more
    (0, 8, 8, 902858, 3), (0, 8, 8, 501754, 2)])
def test_ctas_per_sm_of_the_row_kernel(tsm, cplx, M, N, K, per_sm):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert _choice(tsm, tsm.KIND_TSMTTSM, cplx, M, N, K) == (True, per_sm * sms)


@pytest.mark.parametrize("beta,M,N,K,row", [
    (1, 2, 39, 8874093, False), (0, 2, 39, 8874093, True), (1, 2, 45, 184608, True),  # B read as well, from DRAM
    (0, 2, 23, 200000, False), (0, 2, 23, 2000000, True),                            # one result a thread, from L2
    (0, 32, 1, 4955571, False), (0, 33, 1, 4955571, True),                           # one column
    (0, 2, 4, 10800, False), (0, 2, 19, 7000, True)])                               # as short as a launch
def test_tsmm(tsm, beta, M, N, K, row):
    kind = tsm.KIND_TSMM_BETA if beta else tsm.KIND_TSMM
    names = {v["index"]: v["name"] for v in tsm.variants(tsm.KIND_TSMM)}
    assert names[tsm.choose(kind, 0, M, N, K)[0]].endswith("_row") is row
