"""The first product on a new stream while the default stream is busy: its
workspace's tickets and error words must be zero before its kernels run, on
whatever stream those run.  The memory the workspace gets is filled with ones
first, so tickets that are cleared too late are seen: the last CTA would not
be recognised and the output stay as it was, or the split kernel's error word
would turn it into NaN."""

import ctypes
import os

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tsm():
    import paper_1905_03136_gb300 as t
    from paper_1905_03136_gb300 import build, _lib
    if not os.path.exists(_lib.LIB_PATH):
        build.build()
    t.load()
    return t


def _fill_free_memory(size, count):
    """`count` device blocks of `size` bytes, set to ones and freed again."""
    import torch
    cudart = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    blocks = []
    for _ in range(count):
        p = ctypes.c_void_p()
        assert cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        assert cudart.cudaMemset(p, 0xFF, ctypes.c_size_t(size)) == 0
        blocks.append(p)
    assert cudart.cudaDeviceSynchronize() == 0
    for p in blocks:
        assert cudart.cudaFree(p) == 0


@pytest.mark.parametrize("path", ["last_cta", "fused_step", "split"])
def test_first_call_on_a_side_stream(tsm, path):
    import torch
    from paper_1905_03136_gb300 import split
    A = torch.randint(-3, 4, (700, 4), device="cuda").to(torch.float64)
    B = torch.randint(-3, 4, (700, 4), device="cuda").to(torch.float64)
    C = torch.full((4, 4), 7.0, dtype=torch.float64, device="cuda")
    want = A.T @ B
    direct = [v["index"] for v in tsm.variants(tsm.KIND_TSMTTSM) if v["name"] == "tsmttsm_r64_direct_t1x1_u4"][0]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    tsm._lib.call("tsm_release")
    _fill_free_memory(256, 32)
    torch.cuda._sleep(1_000_000_000)  # half a second on the default stream
    if path == "last_cta":
        tsm.tsmttsm(A, B, C, variant=direct, grid=152, stream=side)
    elif path == "fused_step":
        tsm.gs_step(A, B, C, stream=side, mode="fused")
    else:
        split.tsmttsm_split(A, B, C, stream=side)
    side.synchronize()
    got = C.cpu()  # (waits for the default stream)
    assert torch.equal(got, want.cpu())


def test_batch_made_while_the_default_stream_is_busy(tsm):
    """A batch's plan (items, instances, tickets) is in place when create
    returns: run on a side stream while the default stream has work queued."""
    import torch
    from paper_1905_03136_gb300 import batched
    A = torch.randint(-3, 4, (30000, 5), device="cuda").to(torch.float64)
    B = torch.randint(-3, 4, (30000, 3), device="cuda").to(torch.float64)
    G = torch.full((5, 3), 7.0, dtype=torch.float64, device="cuda")
    want = A.T @ B
    descs = [batched.desc(batched.TSMTTSM, A, B, G, config=10 << 8)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for size in (256, 512, 1024, 4096):
        _fill_free_memory(size, 16)
    torch.cuda._sleep(1_000_000_000)
    batch = batched.Batch(descs)
    batch.run(stream=side)
    side.synchronize()
    assert torch.equal(G.cpu(), want.cpu())
