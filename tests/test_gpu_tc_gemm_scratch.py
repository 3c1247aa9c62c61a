"""The scratch that a stream keeps for its split products: growing and shrinking products, two
threads on one stream, more streams than scratches are kept for, streams that come and go -- every
result has the bits of the same product run alone."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def _product(seed, M, N, K, splits):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import tc_gemm
    build.build()
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    B = torch.randn(N, K, generator=g, device="cuda").bfloat16()
    want = tc_gemm(A, B, splits=splits)
    torch.cuda.synchronize()
    return A, B, splits, want


def test_sizes_that_grow_and_shrink_on_one_stream():
    import torch
    from paper_2407_12149_gb300.mgmc import tc_gemm
    jobs = [_product(i, *s) for i, s in enumerate([(64, 8, 256, 2), (700, 300, 2_048, 8), (128, 64, 512, 3), (900, 512, 4_096, 30)])]
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        out = [tc_gemm(A, B, splits=s) for _ in range(3) for A, B, s, _ in jobs]
    torch.cuda.synchronize()
    for k, o in enumerate(out):
        assert torch.equal(o, jobs[k % len(jobs)][3])


def test_two_threads_on_one_stream():
    import torch
    from paper_2407_12149_gb300.mgmc import tc_gemm
    jobs = [_product(10 + i, 512, 256, 4_096, 16) for i in range(2)]
    side, got = torch.cuda.Stream(), [[], []]

    def work(i):
        A, B, s, _ = jobs[i]
        with torch.cuda.stream(side):
            got[i].extend(tc_gemm(A, B, splits=s) for _ in range(40))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    torch.cuda.synchronize()
    for i in range(2):
        assert len(got[i]) == 40 and all(torch.equal(o, jobs[i][3]) for o in got[i])


def test_more_streams_than_scratches():
    import ctypes

    import torch
    from paper_2407_12149_gb300.mgmc import load
    A, B, splits, want = _product(20, 300, 72, 4_096, 20)
    L, vp, rt = load(), ctypes.c_void_p, torch.cuda.cudart()
    for _ in range(2):               # the second round's streams are new ones
        streams = [vp() for _ in range(70)]
        for s in streams:
            assert int(rt.cudaStreamCreate(ctypes.addressof(s))) == 0
        outs = [torch.zeros(300, 72, device="cuda") for _ in streams]
        torch.cuda.synchronize()
        for _ in range(2):
            for s, C in zip(streams, outs):
                assert L.mgmc_tc_gemm(vp(A.data_ptr()), A.stride(0), vp(B.data_ptr()), B.stride(0), vp(C.data_ptr()), 300, 72,
                                      4_096, splits, 0, None, s) == 0
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in outs)
        for s in streams:
            assert int(rt.cudaStreamDestroy(s.value)) == 0
