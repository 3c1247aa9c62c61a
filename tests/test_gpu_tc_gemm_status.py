"""A tensor-core product whose bounded waits give up: the query after it reports the time-out, no
part of C is written that is not whole (a warp stores 32 rows of a tile), and the next product
is right.  A negative bound makes the part that issues the products give up while the copies of
its operands are in flight and the epilogue waits for its accumulator; a bound of some
nanoseconds lets some tiles through."""
import pytest

pytestmark = pytest.mark.gpu

MGMC_ERR_TIMEOUT = 5


def _data(M, N, K):
    import torch
    from paper_2407_12149_gb300 import build
    build.build()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    return (torch.randn(M, K, generator=g, device="cuda").bfloat16(),
            torch.randn(N, K, generator=g, device="cuda").bfloat16())


# less than a wave of tiles and several tiles per CTA, one and several K blocks, every tile width
@pytest.mark.parametrize("M,N,K", [(300, 24, 64), (40_000, 64, 200), (2_000, 128, 1_024), (20_001, 256, 648)])
@pytest.mark.parametrize("wait_ns", [-2_000_000, -1, 1, 3_000])
def test_no_partial_sums_and_the_time_out_is_reported(M, N, K, wait_ns):
    import torch
    from paper_2407_12149_gb300.mgmc import MGMCError, tc_gemm, tc_gemm_status
    A, B = _data(M, N, K)
    good = tc_gemm(A, B)
    tc_gemm_status()
    C = torch.full((M, N), 12345.0, device="cuda")
    tc_gemm(A, B, out=C, wait_ns=wait_ns)
    gave_up = False
    try:
        tc_gemm_status()
    except MGMCError as e:
        assert e.code == MGMC_ERR_TIMEOUT
        gave_up = True
    tc_gemm_status()                       # reported once
    whole = (C == good)
    untouched = C == 12345.0
    for m0 in range(0, M, 32):
        w, u = whole[m0:m0 + 32], untouched[m0:m0 + 32]
        assert bool(w.all()) or bool(u.all())
    if wait_ns < 0:
        assert gave_up and bool(untouched.all())
    if not gave_up:
        assert bool(whole.all())
    assert torch.equal(tc_gemm(A, B), good)
    tc_gemm_status()
