"""The batched launch's split and its two-level reduction where they change
form: one item, one group (up to 16 items), just over one group, a last
group of one item, many groups; and the default split from one row to
instances far larger than the rest of the batch.  Small integers, so every
sum is exact in any order and must equal the oracle bit for bit."""

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


def _check(bt, insts, config):
    import torch
    descs, want, outs, keep = [], [], [], []
    for i, (kind, cplx, M, N, K) in enumerate(insts):
        A = synth.block_vector(10 + i, K, M, complex_=cplx, dist="smallint")
        B = (synth.block_vector if kind == 0 else synth.small_matrix)(
            60 + i, K if kind == 0 else M, N, complex_=cplx, dist="smallint")
        O = np.zeros((M, N) if kind == 0 else (K, N), dtype=A.dtype)
        op = ("C" if cplx else "T") if kind == 0 else "N"
        dA, dB, dO = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A, B, O))
        descs.append(bt.desc(kind, dA, dB, dO, op=op, config=config))
        want.append(oracle.gram(A, B, op) if kind == 0 else oracle.apply(A, B))
        outs.append(dO)
        keep.append((dA, dB))
    batch = bt.Batch(descs)
    for _ in range(2):  # the tickets are back at zero for the second run
        for o in outs:
            o.zero_()
        batch.run()
        torch.cuda.synchronize()
        for inst, o, w in zip(insts, outs, want):
            assert np.array_equal(o.cpu().numpy(), w), inst


@pytest.mark.parametrize("items", [1, 16, 17, 18, 26, 101])
def test_items_per_instance(bt, items):
    K = 1024 * (items - 1) + 700
    _check(bt, [(0, False, 3, 2, K), (0, True, 5, 7, K), (0, False, 20, 13, K)], 10 << 8)


@pytest.mark.parametrize("insts", [
    [(0, True, 64, 64, 1), (1, True, 64, 64, 1), (0, False, 1, 1, 1)],
    [(0, False, 64, 64, 2900), (0, False, 2, 2, 3), (1, False, 9, 6, 5)],
    [(0, True, 17, 31, 40007), (1, True, 31, 17, 30011), (0, False, 1, 1, 200003), (1, False, 1, 1, 200003)],
], ids=["one_row", "one_large", "mixed"])
def test_default_split(bt, insts):
    _check(bt, insts, 0)
