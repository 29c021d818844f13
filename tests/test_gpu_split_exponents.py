"""The split path's running exponents: data whose column maxima keep growing
(normal, log-uniform, growing along K, zeros first), at the widths where
the stacking of X's slices and the column chunks change, must be as exact as
the slices allow, and repeat bit for bit (the exponents depend on the data
alone, not on which warp came first).

Tolerance: 32 * 2^-(8S-1), the normwise bound of the slice-count test.
"""

import os

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [(False, 1, 1), (False, 32, 3), (False, 33, 40), (True, 16, 16), (True, 17, 40), (True, 32, 41), (True, 64, 64)]


@pytest.fixture(scope="module")
def sp():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib, split
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return split


def _data(kind, rng, K, w, cplx):
    x = rng.standard_normal((K, w)) + (1j * rng.standard_normal((K, w)) if cplx else 0.0)
    if kind == "loguniform":
        x = x * np.exp2(rng.uniform(-20, 20, (K, w)))
    if kind == "growing":
        x = x * np.exp2(np.arange(K) / 500.0)[:, None]
    if kind == "zeros_first":
        x[: K // 3] = 0.0
    if kind == "spikes":  # a value in 300 exceeds the others by 8
        x = x * np.where(rng.random((K, w)) < 1 / 300, 8.0, 1.0)
    return np.ascontiguousarray(x)


@pytest.mark.parametrize("slices", [4, 6])
@pytest.mark.parametrize("kind", ["normal", "loguniform", "growing", "zeros_first", "spikes"])
@pytest.mark.parametrize("case", SHAPES, ids=lambda c: "%s_%dx%d" % ("c64" if c[0] else "r64", c[1], c[2]))
def test_growing_exponents(sp, case, kind, slices):
    import torch
    cplx, M, N = case
    K = 9001 if M * N > 1000 else 40009
    rng = np.random.default_rng(M * 100 + N)
    A, B = _data(kind, rng, K, M, cplx), _data(kind, rng, K, N, cplx)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    op = "C" if cplx else "T"
    got = [sp.tsmttsm_split(dA, dB, op=op, slices=slices).cpu().numpy() for _ in range(4)]
    assert sp.status() == 0
    err = oracle.rel_fro(got[0], oracle.gram(A, B, op))
    # relative to the norms of the columns: a sum of signs may cancel
    scale = np.linalg.norm(np.linalg.norm(A, axis=0)[:, None] * np.linalg.norm(B, axis=0)[None, :])
    err *= np.linalg.norm(got[0]) / scale
    assert err <= 32 * 2.0 ** -(8 * slices - 1), (kind, err)
    for g in got[1:]:
        assert np.array_equal(g, got[0])
