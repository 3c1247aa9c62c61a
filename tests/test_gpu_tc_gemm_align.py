"""Products into a C that starts at any element: the bits of the product into an aligned C, nothing
written beside it; a C or bias between elements is refused."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

MGMC_ERR_ARG = 1


# widths with and without 16-byte rows, full and partial tiles
@pytest.mark.parametrize("M,N,K,splits", [(200, 32, 72, 1), (300, 64, 128, 1), (256, 264, 200, 1), (130, 36, 320, 3)])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 5, 8])
def test_any_element_offset(M, N, K, splits, bf16, shift):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import EPI_BF16, tc_gemm, tc_gemm_status
    build.build()
    if bf16:
        splits = 1
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    epi = EPI_BF16 if bf16 else 0
    want = tc_gemm(A, B, splits=splits, epilogue=epi)
    room = torch.full((shift + M * N + 8,), 7.0, dtype=want.dtype, device="cuda")
    tc_gemm(A, B, out=room[shift:shift + M * N].view(M, N), splits=splits, epilogue=epi)
    tc_gemm_status()
    assert torch.equal(room[shift:shift + M * N].view(M, N), want)
    assert bool((room[:shift] == 7.0).all()) and bool((room[shift + M * N:] == 7.0).all())


def test_an_address_between_elements_is_refused():
    import torch
    from paper_2407_12149_gb300.mgmc import load
    A = torch.zeros(128, 64, dtype=torch.bfloat16, device="cuda")
    C = torch.zeros(128 * 128 + 4, device="cuda")
    vp = ctypes.c_void_p

    def call(c, epi, bias):
        return load().mgmc_tc_gemm(vp(A.data_ptr()), 64, vp(A.data_ptr()), 64, vp(c), 128, 128, 64, 1, epi, vp(bias), None)

    assert call(C.data_ptr() + 2, 0, 0) == MGMC_ERR_ARG
    assert call(C.data_ptr() + 1, 4, 0) == MGMC_ERR_ARG
    assert call(C.data_ptr(), 1, C.data_ptr() + 2) == MGMC_ERR_ARG
    assert call(C.data_ptr(), 0, 0) == 0
    torch.cuda.synchronize()
