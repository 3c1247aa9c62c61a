"""The two GEMM kernels on both sides of the rule between them (a wide tile per multiprocessor): a
product of few tiles has the bits of the same rows and columns in a product of many, in every
tile width, with ragged edges, and agrees with the FP64 product of the same BF16 values."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(8, 72), (32, 2_304), (64, 200), (100, 1_304), (128, 64), (256, 648), (512, 328), (1_000, 40)])
@pytest.mark.parametrize("few", [1, 129, 2_000])
def test_few_rows_have_the_bits_of_many(N, K, few):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import EPI_BF16, EPI_BIAS, EPI_RELU, tc_gemm, tc_gemm_status
    build.build()
    g = torch.Generator(device="cuda").manual_seed(N + K)
    A = torch.randn(40_000, K, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    bias = torch.randn(N, generator=g, device="cuda")
    many = tc_gemm(A, B)
    part = tc_gemm(A[:few], B)
    assert torch.equal(part, many[:few])
    # FP32 accumulation of K products of BF16 values (|a b| <~ 10): rounding ~ K 2^-24 10
    assert (part.double() - A[:few].double() @ B.double().T).abs().max().item() <= 1e-5 * K + 1e-5
    kw = dict(epilogue=EPI_BIAS | EPI_RELU | EPI_BF16, bias=bias)
    assert torch.equal(tc_gemm(A[:few], B, **kw), tc_gemm(A, B, **kw)[:few])
    tc_gemm_status()


@pytest.mark.parametrize("M,N,K,splits", [(64, 24, 4_096, 64), (300, 512, 6_400, 100), (2_000, 256, 2_304, 12)])
def test_splits_on_both_sides(M, N, K, splits):
    import torch
    from paper_2407_12149_gb300.mgmc import tc_gemm
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    ref = A.double() @ B.double().T
    assert (tc_gemm(A, B, splits=splits).double() - ref).abs().max().item() <= 1e-5 * K + 1e-5
