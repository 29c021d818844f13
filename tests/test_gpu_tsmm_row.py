"""TSMM's row kernel (results per thread, row lanes and grid chosen per launch)
against the oracle: every count of results per thread, rows fewer than, equal
to and just past the CTAs, odd last rows of a range, beta of each kind, padded
rows, more CTAs than rows, and the rule that picks it.  Small integers must
match bit for bit; the tolerance for random data is the library's normwise
1e-12.  Rows of B past K and columns past N must stay as they were."""

import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
TOL = 1e-12

SHAPES = [(1, 1), (3, 2), (8, 3), (5, 64), (64, 5), (37, 53), (23, 11), (64, 64), (7, 10), (2, 19)]


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


def _row(tsm, cplx):
    name = "tsmm_%s_row" % ("c64" if cplx else "r64")
    return [v["index"] for v in tsm.variants(tsm.KIND_TSMM) if v["name"] == name][0]


@pytest.mark.parametrize("cplx", [False, True], ids=["r64", "c64"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d" % s)
def test_row_kernel(tsm, shape, cplx):
    import torch
    M, N = shape
    v = _row(tsm, cplx)
    for K in (1, 33, 152, 153, 1000, 4099, 40009):
        for dist in ("smallint", "uniform"):
            A = synth.block_vector(1, K, M, ld=M + 3, complex_=cplx, dist=dist)
            B0 = synth.block_vector(2, K + 5, N, ld=N + 1, complex_=cplx, dist=dist)
            C = synth.small_matrix(3, M, N, complex_=cplx, dist=dist)
            a, b = np.ascontiguousarray(A[:, :M]), np.ascontiguousarray(B0[:K, :N])
            dA, dC = torch.from_numpy(A).cuda()[:, :M], torch.from_numpy(C).cuda()
            scalars = [(1.0, 0.0), (-1.0, 1.0), (2.0, -3.0)] + ([(1.0 + 2.0j, 3.0 - 1.0j)] if cplx else [])
            for alpha, beta in scalars:
                want = alpha * (a @ C) + beta * b
                for grid in (0, 1, 304, 999):
                    B = torch.from_numpy(B0).cuda()
                    tsm.tsmm(dA, dC, B[:K, :N], alpha, beta, variant=v, grid=grid)
                    got = B.cpu().numpy()
                    if dist == "smallint":
                        assert np.array_equal(got[:K, :N], want), (K, alpha, beta, grid)
                    else:
                        assert oracle.rel_fro(got[:K, :N], want) <= TOL, (K, alpha, beta, grid)
                    assert np.array_equal(got[K:], B0[K:]) and np.array_equal(got[:, N:], B0[:, N:])


def test_rule(tsm):
    """Short products, and longer ones whose other kernel pads or leaves the
    chip idle, take the row kernel; from 2^22 rows on none does without a
    tuning table; products bound by memory do not; an entry tuned for the very
    bucket of K stands."""
    from paper_1905_03136_gb300 import costmodel as cm
    rows = (_row(tsm, False), _row(tsm, True))
    for cplx, M, N, K in [(1, 64, 64, 1000), (0, 8, 8, 6000), (1, 23, 11, 200003), (0, 18, 21, 1500000), (0, 36, 3, 10000000)]:
        for kind in (tsm.KIND_TSMM, tsm.KIND_TSMM_BETA):
            assert tsm.choose(kind, cplx, M, N, K)[0] == rows[cplx], (cplx, M, N, K)
    for cplx, M, N, K in [(0, 2, 2, 1 << 20), (0, 1, 8, 160000), (0, 31, 11, 567000)]:
        assert tsm.choose(tsm.KIND_TSMM, cplx, M, N, K)[0] != rows[cplx], (cplx, M, N, K)
    assert not cm.heuristic_pick(tsm.KIND_TSMM, 0, 36, 3, 1 << 23)[0].endswith("_row")
    lib = tsm.load()
    other = [v["index"] for v in tsm.variants(tsm.KIND_TSMM) if v["name"] == "tsmm_r64_rt_npt4_u2"][0]
    assert lib.tsm_set_tuning(tsm.KIND_TSMM, 0, 11, 6, 5000, other, 152) == 0
    assert tsm.choose(tsm.KIND_TSMM, 0, 11, 6, 5000) == (other, 152)
    assert tsm.choose(tsm.KIND_TSMM, 0, 11, 6, 20000)[0] == rows[0]


def test_threads_with_different_shared_memory(tsm):
    """Threads whose launches of one kernel pin different numbers of CTAs per
    SM, and so ask for different amounts of shared memory, at the same time."""
    import threading

    import torch
    shapes = [(16, 16, 500), (16, 16, 60000), (60, 60, 700), (60, 60, 30000)]
    errors = []

    def work(M, N, K):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                A = torch.randint(-3, 4, (K, M), device="cuda").to(torch.float64)
                C = torch.randint(-3, 4, (M, N), device="cuda").to(torch.float64)
                B, G = torch.empty((K, N), dtype=torch.float64, device="cuda"), torch.empty_like(C)
                for _ in range(150):
                    tsm.tsmm(A, C, B, 1.0, 0.0)
                    tsm.tsmttsm(A, B, G)
                st.synchronize()
                if not (torch.equal(B, A @ C) and torch.equal(G, A.T @ B)):
                    errors.append((M, N, K, "values"))
        except Exception as e:
            errors.append((M, N, K, repr(e)))

    threads = [threading.Thread(target=work, args=s) for s in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
