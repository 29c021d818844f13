"""The network on streams other than the default one: the copies to and from
the host wait for the calls before them on any stream, and what they write is
there for the calls after them, without a synchronisation by the caller."""

import os

import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu
D, H, N = 9, 40, 3000


@pytest.fixture(scope="module")
def M():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib, mlp
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return mlp


@pytest.fixture
def data():
    import torch
    rng = np.random.default_rng(11)
    p = [rng.uniform(-0.3, 0.3, omlp.param_count(D, H)).astype(np.float32) for _ in range(2)]
    X = rng.uniform(-1, 1, (N, D)).astype(np.float32)
    t = rng.uniform(-1, 1, N).astype(np.float32)
    return p, X, t, torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda()


def _late(stream):
    """Half a second of other work before what follows on the stream."""
    import torch
    with torch.cuda.stream(stream):
        torch.cuda._sleep(1_000_000_000)


def test_copies_wait_for_side_streams(M, data):
    import torch
    p, X, t, dX, dt = data
    net = M.Mlp(D, H, max_batch=N)
    net.set_params(p[0])
    torch.cuda.synchronize()
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    _late(side)
    _late(other)
    y = net.forward(dX, stream=other)
    net.backward(dX, dt, stream=side)
    g = net.grads()
    ref = omlp.grad(p[0], X, t, D, H)
    assert np.max(np.abs(g - ref)) <= 1e-4 * np.max(np.abs(ref))
    net.adam(stream=side)
    net.set_params(p[1])  # after the step, and after the other stream's read
    assert np.array_equal(net.params(), p[1])
    other.synchronize()
    want = omlp.forward(p[0], X, D, H)
    assert np.max(np.abs(y.cpu().numpy() - want)) <= 1e-5 * max(1.0, np.max(np.abs(want)))


def test_side_streams_see_what_was_set(M, data):
    import torch
    p, X, t, dX, dt = data
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    _late(torch.cuda.default_stream())
    net = M.Mlp(D, H, max_batch=N, seed=5)
    first = net.forward(dX, stream=side)
    side.synchronize()
    own = net.params()
    net.set_params(p[1])
    y = net.forward(dX, stream=side)
    side.synchronize()
    for got, q in ((first, own), (y, p[1])):
        want = omlp.forward(q, X, D, H)
        assert np.max(np.abs(got.cpu().numpy() - want)) <= 1e-5 * max(1.0, np.max(np.abs(want)))
