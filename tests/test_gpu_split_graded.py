"""The split path's column exponents where rows of very different size follow
one another: small rows that come first keep the bits that the columns'
running maxima leave them, whatever the next rows of their range hold; values
that exceed 2^e by less than a bit, as often as a tile may hold them, stay
exact; and with 5 slices, the growing data of the 4 and 6 slice test.

Tolerance: 32 * 2^-(8S-1) of the products of the column norms, over the rows
that count; integers exactly.
"""

import os

import numpy as np
import pytest

import oracle
from test_gpu_split_exponents import SHAPES, _data

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib, split
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return split


def _err(got, A, B, op):
    scale = np.linalg.norm(np.linalg.norm(A, axis=0)[:, None] * np.linalg.norm(B, axis=0)[None, :])
    return np.linalg.norm(got - oracle.gram(A, B, op)) / scale


@pytest.mark.parametrize("slices", [4, 5, 6])
@pytest.mark.parametrize("big", ["A", "B"])
@pytest.mark.parametrize("case", [(False, 3, 2), (False, 24, 40), (True, 17, 40), (True, 64, 64)],
                         ids=lambda c: "%s_%dx%d" % ("c64" if c[0] else "r64", c[1], c[2]))
def test_small_rows_before_large_ones(sp, case, big, slices):
    """16 rows of order 1, then 112 rows in which one operand is of order 2^50
    and the other zero: the first 16 rows are the whole product."""
    import torch
    cplx, M, N = case
    K, op = 200003, "C" if cplx else "T"
    rng = np.random.default_rng(M + N)
    A, B = _data("normal", rng, K, M, cplx), _data("normal", rng, K, N, cplx)
    (A if big == "A" else B)[16:128] *= 2.0 ** 50
    (B if big == "A" else A)[16:] = 0.0
    got = sp.tsmttsm_split(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), op=op, slices=slices).cpu().numpy()
    assert sp.status() == 0
    assert _err(got, np.ascontiguousarray(A[:16]), np.ascontiguousarray(B[:16]), op) <= 32 * 2.0 ** -(8 * slices - 1)


@pytest.mark.parametrize("slices", [5, 6])
@pytest.mark.parametrize("shape", [(3, 2), (24, 40), (64, 64), (128, 128)], ids=lambda s: "%dx%d" % s)
def test_values_above_the_exponent(sp, shape, slices):
    """Steps of 16 rows whose values are all 127, with some of 254 and 255
    among them: 127 sets e, 254 exceeds 2^e by just less than the digits
    allow, 255 by too much.  All of one sign, so that the tile's sums reach
    their bounds; at random, and as a run.
    (Widths above 64 as the two parts of complex data.)"""
    import torch
    M, N = shape
    K = 16 * 3001
    rng = np.random.default_rng(M * N + slices)

    def steps(w, p):
        x = np.where(rng.random((K // 16, 1, w)) < p, 254.0, 127.0)
        x = np.where(rng.random((K // 16, 1, w)) < 0.002, 255.0, x)
        if p == 0.0:
            x = np.full((K // 16, 1, w), 127.0)
            x[15:26] = 254.0
        return np.ascontiguousarray(np.broadcast_to(x, (K // 16, 16, w)).reshape(K, w))

    for p in (0.0, 0.02, 0.3):
        A, B = steps(M, p), steps(N, p)
        if M <= 64:
            got = sp.tsmttsm_split(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), slices=slices).cpu().numpy()
            assert np.array_equal(got, A.T @ B)
        else:
            a, b = A.view(np.complex128), B.view(np.complex128)
            got = sp.tsmttsm_split(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), op="C",
                                   slices=slices).cpu().numpy()
            assert np.array_equal(got, a.conj().T @ b)
    assert sp.status() == 0


@pytest.mark.parametrize("kind", ["normal", "loguniform", "growing", "zeros_first", "spikes"])
@pytest.mark.parametrize("case", SHAPES, ids=lambda c: "%s_%dx%d" % ("c64" if c[0] else "r64", c[1], c[2]))
def test_five_slices(sp, case, kind):
    import torch
    cplx, M, N = case
    K, op = 9001 if M * N > 1000 else 40009, "C" if cplx else "T"
    rng = np.random.default_rng(M * 100 + N)
    A, B = _data(kind, rng, K, M, cplx), _data(kind, rng, K, N, cplx)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    got = [sp.tsmttsm_split(dA, dB, op=op, slices=5).cpu().numpy() for _ in range(4)]
    assert sp.status() == 0
    assert _err(got[0], A, B, op) <= 32 * 2.0 ** -39
    for g in got[1:]:
        assert np.array_equal(g, got[0])
