"""Short products back to back on one stream: their kernels start early at any
grid, and so does the final reduction, so that several launches of a chain
overlap.  As in the tests of the long products, every chain runs once drained
after each call and once without any synchronisation, with all outputs
allocated before, and the results must agree bit for bit; the drained ones are
checked against the oracle on the values the chain had at that point."""

import os

import numpy as np
import pytest

import oracle
from test_gpu_pdl import TOL, _dev, _run_twice

pytestmark = pytest.mark.gpu

SHAPES = [(False, 8, 8, 16000), (True, 16, 16, 2000), (False, 37, 53, 1500), (True, 33, 20, 1000), (False, 3, 3, 100000),
          (False, 25, 25, 60000)]
ids = ["%s_%dx%d_%d" % ("c64" if s[0] else "r64", *s[1:]) for s in SHAPES]
N_STEPS = 12


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


def _step(drain):
    if drain:
        import torch
        torch.cuda.synchronize()


@pytest.mark.parametrize("shape", SHAPES, ids=ids)
def test_fresh_output_is_read(tsm, shape):
    """V = A C_i, then G_i = op(A)^T V: V has other values at every step, and
    is overwritten while the reduction of the step before may still run."""
    import torch
    cplx, M, N, K = shape
    names = {v["index"]: v["name"] for v in tsm.variants(tsm.KIND_TSMTTSM)}
    assert names[tsm.choose(tsm.KIND_TSMTTSM, int(cplx), M, N, K)[0]].endswith("_row")
    A, op = _dev(tsm, K, M, cplx, 1), "C" if cplx else "T"
    Cs = [_dev(tsm, M, N, cplx, 50 + i) for i in range(N_STEPS)]
    V = torch.empty((K, N), dtype=A.dtype, device="cuda")

    def chain(drain):
        Gs = [torch.zeros((M, N), dtype=A.dtype, device="cuda") for _ in Cs]
        torch.cuda.synchronize()
        for Ci, G in zip(Cs, Gs):
            tsm.tsmm(A, Ci, V, 1.0, 0.0)
            _step(drain)
            tsm.tsmttsm(A, V, G, op=op)
            _step(drain)
        return Gs
    res = _run_twice(chain)
    Ah = A.cpu().numpy()
    for i in (0, N_STEPS - 1):
        assert oracle.rel_fro(res[i], oracle.gram(Ah, oracle.apply(Ah, Cs[i].cpu().numpy()), op)) <= TOL


@pytest.mark.parametrize("shape", SHAPES, ids=ids)
def test_small_matrix_goes_round(tsm, shape):
    """C = op(A)^T B, B += C-dependent update, C accumulated: each call reads
    what the one before it wrote, and writes what the one before it read."""
    import torch
    cplx, M, N, K = shape
    A, B0, op = _dev(tsm, K, M, cplx, 3), _dev(tsm, K, N, cplx, 4), "C" if cplx else "T"
    C = torch.zeros((M, N), dtype=A.dtype, device="cuda")

    def chain(drain):
        B = B0.clone()
        C.zero_()
        torch.cuda.synchronize()
        for _ in range(N_STEPS):
            tsm.tsmttsm(A, B, C, 1.0 / K, 0.5, op=op)
            _step(drain)
            tsm.tsmm(A, C, B, -0.25, 1.0)
            _step(drain)
        torch.cuda.synchronize()
        return [B, C.clone()]
    B, C_got = _run_twice(chain)
    a, b, c = A.cpu().numpy(), B0.cpu().numpy(), np.zeros((M, N), dtype=B0.cpu().numpy().dtype)
    for _ in range(N_STEPS):
        c = oracle.gram(a, b, op, 1.0 / K, 0.5, c)
        b = oracle.apply(a, c, -0.25, 1.0, b)
    assert oracle.rel_fro(C_got, c) <= TOL and oracle.rel_fro(B, b) <= TOL


@pytest.mark.parametrize("shape", SHAPES, ids=ids)
def test_inputs_changed_by_other_kernels(tsm, shape):
    """A kernel of another library writes an input between two products."""
    import torch
    cplx, M, N, K = shape
    A0, B, op = _dev(tsm, K, M, cplx, 5), _dev(tsm, K, N, cplx, 6), "C" if cplx else "T"

    def chain(drain):
        A = A0.clone()
        Gs = [torch.zeros((M, N), dtype=A.dtype, device="cuda") for _ in range(N_STEPS)]
        torch.cuda.synchronize()
        for G in Gs:
            tsm.tsmttsm(A, B, G, op=op)
            _step(drain)
            A.mul_(-0.5)
            _step(drain)
        return Gs
    res = _run_twice(chain)
    want = oracle.gram(A0.cpu().numpy(), B.cpu().numpy(), op)
    for i, G in enumerate(res):
        assert oracle.rel_fro(G, want * (-0.5) ** i) <= TOL


def test_independent_products_of_several_shapes(tsm):
    """Products that share nothing, short ones between longer ones: the early
    reads of one overlap the reductions of two others."""
    import torch
    jobs = []
    for i, (cplx, M, N, K) in enumerate(SHAPES * 2):
        A, B = _dev(tsm, K, M, cplx, 70 + i), _dev(tsm, K, N, cplx, 90 + i)
        jobs.append((A, B, torch.zeros((M, N), dtype=A.dtype, device="cuda"), "C" if cplx else "T"))

    def chain(drain):
        for A, B, G, op in jobs:
            G.zero_()
        torch.cuda.synchronize()
        for _ in range(5):
            for A, B, G, op in jobs:
                tsm.tsmttsm(A, B, G, 1.0, 1.0, op=op)
                _step(drain)
        torch.cuda.synchronize()
        return [G.clone() for _, _, G, _ in jobs]
    for got, (A, B, _, op) in zip(_run_twice(chain), jobs):
        assert oracle.rel_fro(got, 5.0 * oracle.gram(A.cpu().numpy(), B.cpu().numpy(), op)) <= TOL
