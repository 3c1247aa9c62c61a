"""A thread whose first CUDA call is a product: same bits as the main thread's."""
import ctypes
import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("splits", [1, 4])
def test_first_cuda_call_of_a_thread(splits):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import load, tc_gemm
    build.build()
    g = torch.Generator(device="cuda").manual_seed(2)
    A = torch.randn(256, 512, generator=g, device="cuda").bfloat16()
    B = torch.randn(64, 512, generator=g, device="cuda").bfloat16()
    want, C = tc_gemm(A, B, splits=splits), torch.zeros(256, 64, device="cuda")
    torch.cuda.synchronize()
    a, b, c, rc, vp, L = A.data_ptr(), B.data_ptr(), C.data_ptr(), [], ctypes.c_void_p, load()
    t = threading.Thread(target=lambda: rc.append(L.mgmc_tc_gemm(vp(a), 512, vp(b), 512, vp(c), 256, 64, 512, splits, 0, None, None)))
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert rc == [0] and torch.equal(C, want)
