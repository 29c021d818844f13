"""Instances without rows in a batched launch: a TSMM with K = 0 takes no
work item (its A and C may be null and nothing is written), a TSMTTSM with
K = 0 still applies beta to its output, alone and among other instances."""

import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bt():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import batched, build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return batched


def _empty(bt, kind, M, N, out, beta):
    """Descriptor of an instance with K = 0 and null inputs."""
    import torch
    d = bt.desc(kind, torch.empty((0, M), dtype=torch.complex128, device="cuda"),
                torch.empty((0 if kind == bt.TSMTTSM else M, N), dtype=torch.complex128, device="cuda"), out, 1.5, beta)
    assert d.K == 0
    d.A = d.B = None
    d.lda, d.ldb = M, N
    return d


@pytest.mark.parametrize("config", [0, 10 << 8], ids=["default", "1024_rows"])
@pytest.mark.parametrize("among", [False, True], ids=["alone", "among_others"])
def test_instances_without_rows(bt, among, config):
    import torch
    rows = np.ascontiguousarray(synth.block_vector(1, 4, 64, complex_=True, dist="smallint"))
    small = synth.small_matrix(2, 5, 7, complex_=True, dist="smallint")
    B_out, C_out = torch.from_numpy(rows).cuda(), torch.from_numpy(small).cuda()
    descs = [_empty(bt, bt.TSMM, 64, 64, B_out, 0.5), _empty(bt, bt.TSMTTSM, 5, 7, C_out, 3.0)]
    for d in descs:
        d.config = config
    want = None
    if among:
        A = synth.block_vector(3, 3001, 6, complex_=False, dist="smallint")
        X = synth.block_vector(4, 3001, 9, complex_=False, dist="smallint")
        dA, dX = torch.from_numpy(A).cuda(), torch.from_numpy(X).cuda()
        G = torch.zeros((6, 9), dtype=torch.float64, device="cuda")
        descs.insert(1, bt.desc(bt.TSMTTSM, dA, dX, G, config=config))
        want = oracle.gram(A, X, "T")
    batch = bt.Batch(descs)
    if not among:
        assert batch.info()[0] == 1  # the TSMTTSM's empty item
    for n in (1, 2):
        batch.run()
        torch.cuda.synchronize()
        assert np.array_equal(C_out.cpu().numpy(), small * 3.0 ** n)
        assert np.array_equal(B_out.cpu().numpy(), rows)
        if among:
            assert np.array_equal(G.cpu().numpy(), want)


def test_plan_without_any_item(bt):
    import torch
    out = torch.ones((3, 4), dtype=torch.complex128, device="cuda")
    batch = bt.Batch([_empty(bt, bt.TSMM, 64, 4, out, 2.0)] * 2)
    assert batch.info()[0] == 0
    batch.run()
    batch.run_direct()
    torch.cuda.synchronize()
    assert bool((out == 1).all())
