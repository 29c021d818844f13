"""Two plans of the batched launch whose shared-memory needs differ, both above
the 48 KB every kernel may use: making the smaller one must leave the larger
one runnable, without the graph (which holds the limit of its capture) too."""

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


def test_smaller_plan_after_a_larger_one(bt):
    import torch
    plans = []
    for w in (64, 60):  # C of 65536 and 57600 bytes
        A = synth.block_vector(w, 501, w, complex_=True, dist="smallint")
        C = synth.small_matrix(w + 1, w, w, complex_=True, dist="smallint")
        dA, dC = torch.from_numpy(A).cuda(), torch.from_numpy(C).cuda()
        out = torch.zeros((501, w), dtype=torch.complex128, device="cuda")
        plans.append((bt.Batch([bt.desc(bt.TSMM, dA, dC, out)]), out, oracle.apply(A, C), dA, dC))
    for batch, out, want, *_ in plans:
        for run in (batch.run_direct, batch.run):
            out.zero_()
            run()
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), want)
