"""The tiled network kernels at the edges of their sample tiles (32), unit
padding (64 units, 32 inputs) and tile loop (more tiles than CTAs), against
the float64 oracle.

Tolerances: an activation is a chain of at most 64 FP32 FMAs into a tanh
(slope <= 1) of inputs below 1, so its error is below 64 * 2^-24 * 64 * 0.3
per layer, under 1e-4 of the output scale in the worst case and about 1e-6
for random signs; 1e-5 is the bar of the other network tests.  A gradient
entry sums n terms of such error: 1e-4 of the largest entry, as there.
"""

import os

import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

CASES = [(1, 1, 1), (5, 8, 31), (17, 64, 32), (32, 64, 33), (3, 63, 64), (31, 61, 97), (17, 64, 10007)]


@pytest.fixture(scope="module")
def M():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib, mlp
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return mlp


@pytest.mark.parametrize("D,H,n", CASES)
def test_values_and_gradient_at_tile_edges(M, D, H, n):
    import torch
    rng = np.random.default_rng(100 * D + H + n)
    p = rng.uniform(-0.3, 0.3, omlp.param_count(D, H)).astype(np.float32)
    X = rng.uniform(-1, 1, (n, D)).astype(np.float32)
    t = rng.uniform(-1, 1, n).astype(np.float32)
    net = M.Mlp(D, H, max_batch=n)
    net.set_params(p)
    dX, dt = torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda()
    y = net.forward(dX).cpu().numpy()
    ref = omlp.forward(p, X, D, H)
    assert np.max(np.abs(y - ref)) <= 1e-5 * max(1.0, np.max(np.abs(ref)))
    loss = float(net.backward(dX, dt).item())
    want = omlp.loss(p, X, t, D, H)
    assert abs(loss - want) <= 1e-5 * max(1.0, want)
    g = net.grads()
    g_ref = omlp.grad(p, X, t, D, H)
    assert np.max(np.abs(g - g_ref)) <= 1e-4 * np.max(np.abs(g_ref))
    net.backward(dX, dt)
    assert np.array_equal(net.grads(), g)
