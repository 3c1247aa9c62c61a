"""Split-K products on several streams, from several threads and in a captured graph: each has its
own partial sums, so each result has the bits of the same product run alone."""
import threading

import pytest

pytestmark = pytest.mark.gpu

# (M, N, K, splits): few enough tiles that two products run at the same time
SHAPES = [(512, 256, 4_096, 16), (300, 72, 8_192, 40)]


def _operands(seed, M, N, K):
    import torch
    from paper_2407_12149_gb300 import build
    build.build()
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(M, K, generator=g, device="cuda").bfloat16(),
            torch.randn(N, K, generator=g, device="cuda").bfloat16())


def _products(jobs, stream, rounds):
    """`rounds` products of every job on `stream`; the outputs."""
    import torch
    from paper_2407_12149_gb300.mgmc import tc_gemm
    with torch.cuda.stream(stream):
        return [tc_gemm(A, B, splits=s) for _ in range(rounds) for A, B, s in jobs]


def _jobs(seed):
    return [(*_operands(seed + i, M, N, K), s) for i, (M, N, K, s) in enumerate(SHAPES)]


@pytest.mark.parametrize("threads", [False, True])
def test_two_streams_do_not_share_partial_sums(threads):
    import torch
    sets = [_jobs(1), _jobs(11)]
    alone = []
    for jobs in sets:
        alone.append(_products(jobs, torch.cuda.current_stream(), 1))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in sets]
    rounds, got = 20, [None, None]

    def work(i, n):
        got[i] = (got[i] or []) + _products(sets[i], streams[i], n)

    if threads:
        ts = [threading.Thread(target=work, args=(i, rounds)) for i in range(2)]
        [t.start() for t in ts]
        [t.join() for t in ts]
    else:
        for _ in range(rounds):
            work(0, 1)
            work(1, 1)
    torch.cuda.synchronize()
    for i in range(2):
        assert len(got[i]) == rounds * len(SHAPES)
        for k, out in enumerate(got[i]):
            assert torch.equal(out, alone[i][k % len(SHAPES)])


def test_split_product_in_a_graph_beside_a_larger_one():
    import torch
    from paper_2407_12149_gb300.mgmc import tc_gemm
    (A, B, s), (A2, B2, _) = _jobs(3)[0], _jobs(5)[0]
    alone = tc_gemm(A, B, splits=s)
    out = torch.empty_like(alone)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        tc_gemm(A, B, out=out, splits=s)
    side = torch.cuda.Stream()
    for _ in range(5):
        out.zero_()
        with torch.cuda.stream(side):
            tc_gemm(A2, B2, splits=64)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, alone)
