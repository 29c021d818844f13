"""Threads that launch one kernel with different amounts of shared memory at
the same time, all above the 48 KB every kernel may use: the limit is state of
the kernel function, so no launch may set it below what another one needs."""

import os
import threading

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


@pytest.mark.parametrize("path", ["tsmm_c64_smemc_tpr4_npt16_u1", "tsmm_c64_rt_npt4_u2", "fused_step"])
def test_threads(tsm, path):
    import torch
    index = {v["name"]: v["index"] for v in tsm.variants(tsm.KIND_TSMM)}
    errors = []

    def work(w):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                g = torch.Generator(device="cuda").manual_seed(w)
                A, C, B0 = (torch.complex(*(torch.randint(-3, 4, (2, n, w), generator=g, device="cuda").double()))
                            for n in (200, w, 200))
                B = torch.empty_like(B0)
                for _ in range(200):
                    if path == "fused_step":
                        B.copy_(B0)
                        tsm.gs_step(A, B, mode="fused")
                    else:
                        tsm.tsmm(A, C, B, 1.0, 0.0, variant=index[path])
                want = B0 - A @ (A.mH @ B0) if path == "fused_step" else A @ C
                st.synchronize()
                if not torch.equal(B, want):
                    errors.append((w, "values"))
        except Exception as e:
            errors.append((w, repr(e)))

    threads = [threading.Thread(target=work, args=(w,)) for w in (64, 60, 62, 58)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
