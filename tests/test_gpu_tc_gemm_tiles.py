"""The BF16 GEMM where a CTA takes several tiles, in every tile width: more tiles than
multiprocessors, ragged last tiles along M, N and K, an incomplete group of M tiles, K splits."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,splits", [(40_000, 24, 40, 1), (20_001, 64, 72, 1), (40_100, 100, 136, 1),
                                          (20_200, 130, 648, 1), (2_500, 2_300, 200, 1), (2_177, 1_032, 1_304, 3),
                                          (128, 8, 64 * 400, 400)])
@pytest.mark.parametrize("relu_bf16", [False, True])
def test_many_tiles(M, N, K, splits, relu_bf16):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import EPI_BF16, EPI_BIAS, EPI_RELU, tc_gemm
    build.build()
    if relu_bf16 and splits > 1:
        pytest.skip("K splits store FP32")
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    ref = A.double() @ B.double().T
    if not relu_bf16:
        err = (tc_gemm(A, B, splits=splits).double() - ref).abs().max().item()
        # FP32 accumulation of K products of BF16 values (|a b| <~ 10): rounding ~ K 2^-24 10
        assert err <= 1e-5 * K + 1e-5, err
        return
    bias = torch.randn(N, generator=g, device="cuda")
    out = tc_gemm(A, B, epilogue=EPI_BIAS | EPI_RELU | EPI_BF16, bias=bias).double()
    ref = (ref + bias.double()).clamp(min=0.0)
    # BF16 rounding 2^-8 and the accumulation's
    assert ((out - ref).abs() <= 2.0 ** -8 * ref + 1e-5 * K).all()
