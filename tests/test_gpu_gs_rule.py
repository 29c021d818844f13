"""Both sides of the line between the fused Gram-Schmidt step and the two
products: the automatic choice, the fused kernel and the two products give the
oracle's C and B (normwise 1e-12 of the larger term), on padded rows."""

import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


@pytest.mark.parametrize("cplx,M,N", [(False, 4, 4), (True, 33, 20), (False, 43, 17), (False, 13, 1), (True, 2, 30),
                                      (False, 1, 9), (True, 64, 64)])
def test_step_on_both_sides_of_the_line(tsm, cplx, M, N):
    import torch
    for K in (800, 801, 1501, 3001, 8001, 32769):
        A = synth.block_vector(1, K, M, ld=M + 1, complex_=cplx)
        B0 = synth.block_vector(2, K, N, ld=N + 2, complex_=cplx)
        a, b = np.ascontiguousarray(A[:, :M]), np.ascontiguousarray(B0[:, :N])
        C = oracle.gram(a, b, "C" if cplx else "T")
        want = b - a @ C
        dA = torch.from_numpy(A).cuda()[:, :M]
        for mode in ("auto", "fused", "two_products"):
            B = torch.from_numpy(B0).cuda()
            got = tsm.gs_step(dA, B[:, :N], mode=mode).cpu().numpy()
            out = B.cpu().numpy()
            scale = np.linalg.norm(a @ C)
            assert oracle.rel_fro(got, C) <= TOL, (K, mode)
            assert np.linalg.norm(out[:, :N] - want) <= TOL * scale, (K, mode)
            assert np.array_equal(out[:, N:], B0[:, N:]), (K, mode)
