"""The row kernels (strip length, orientation and CTA size chosen per shape)
against the oracle: both orientations, the shortest and longest strips, one
to many row lanes, fewer rows than CTAs, padded rows, and the rule that picks
them for short products.  Small integers must match bit for bit; the
tolerance for random data is the library's normwise 1e-12."""

import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
TOL = 1e-12

SHAPES = [(1, 1), (3, 2), (5, 64), (64, 5), (37, 53), (53, 37), (64, 63), (13, 13), (2, 60), (9, 41), (17, 33)]


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


def _row(tsm, cplx):
    name = "tsmttsm_%s_row" % ("c64" if cplx else "r64")
    return [v["index"] for v in tsm.variants(tsm.KIND_TSMTTSM) if v["name"] == name][0]


@pytest.mark.parametrize("cplx", [False, True], ids=["r64", "c64"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d" % s)
def test_row_kernel(tsm, shape, cplx):
    import torch
    M, N = shape
    v = _row(tsm, cplx)
    if not tsm.load().tsm_variant_supports(tsm.KIND_TSMTTSM, v, int(cplx), M, N):
        assert cplx and M * N > 7 * 512  # more strips than a CTA has threads
        return
    for K in (1, 31, 4099, 40009):
        for dist in ("smallint", "uniform"):
            A = synth.block_vector(1, K, M, ld=M + 3, complex_=cplx, dist=dist)
            B = synth.block_vector(2, K, N, ld=N + 1, complex_=cplx, dist=dist)
            C0 = synth.small_matrix(3, M, N, complex_=cplx, dist=dist)
            dA, dB = torch.from_numpy(A).cuda()[:, :M], torch.from_numpy(B).cuda()[:, :N]
            a, b = np.ascontiguousarray(A[:, :M]), np.ascontiguousarray(B[:, :N])
            for op in (("T", "C") if cplx else ("T",)):
                for grid in (0, 1, 152, 304, 999):
                    got = tsm.tsmttsm(dA, dB, op=op, variant=v, grid=grid).cpu().numpy()
                    if dist == "smallint":
                        assert np.array_equal(got, oracle.gram(a, b, op)), (K, op, grid)
                    else:
                        assert oracle.rel_fro(got, oracle.gram(a, b, op)) <= TOL, (K, op, grid)
                C = torch.from_numpy(C0).cuda()
                tsm.tsmttsm(dA, dB, C, -2.0, 3.0, op=op, variant=v)
                assert oracle.rel_fro(C.cpu().numpy(), oracle.gram(a, b, op, -2.0, 3.0, C0)) <= TOL, (K, op)


def test_rule_for_short_products(tsm):
    """Short products take the row kernels (the very shortest of the narrow
    widths do not), products from 2^21 rows on only without an entry for their
    shape in a table that has others, and an entry tuned for the very bucket
    of K stands."""
    from paper_1905_03136_gb300 import costmodel as cm
    rows = (_row(tsm, False), _row(tsm, True))
    for cplx, M, N, K in [(0, 4, 4, 60000), (1, 8, 8, 100000), (0, 25, 25, 60000), (0, 37, 53, 300007),
                          (0, 58, 13, 1 << 23), (1, 45, 32, 1 << 22)]:
        assert tsm.choose(tsm.KIND_TSMTTSM, cplx, M, N, K)[0] == rows[cplx], (cplx, M, N, K)
    for cplx, M, N, K in [(0, 4, 4, 1 << 21), (0, 4, 4, 10000), (1, 64, 64, 5000), (0, 9, 1, 1 << 23), (0, 4, 4, 900000)]:
        assert tsm.choose(tsm.KIND_TSMTTSM, cplx, M, N, K)[0] != rows[cplx], (cplx, M, N, K)
    for cplx, M, N in [(0, 58, 13), (1, 45, 32)]:
        assert not cm.heuristic_pick(tsm.KIND_TSMTTSM, cplx, M, N, 1 << 22)[0].endswith("_row")
    lib = tsm.load()
    other = [v["index"] for v in tsm.variants(tsm.KIND_TSMTTSM) if v["name"] == "tsmttsm_r64_direct_t1x1_u4"][0]
    assert lib.tsm_set_tuning(tsm.KIND_TSMTTSM, 0, 11, 6, 5000, other, 152) == 0
    assert tsm.choose(tsm.KIND_TSMTTSM, 0, 11, 6, 5000) == (other, 152)
    assert tsm.choose(tsm.KIND_TSMTTSM, 0, 11, 6, 20000)[0] == rows[0]
