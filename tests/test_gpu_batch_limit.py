"""The largest batch mgmc_create_batch accepts, 65 536 chains: every chain advances and writes its
QoI series, and chains at both ends and in the middle repeat their solo runs bit for bit."""
import pytest

from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_65536_chains():
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import BatchSampler, Sampler
    build.build()
    p = inputs.make_problem("limit", 2, 3, kappa2_const=10.0, m=0, qoi_cells=2)
    n, steps = 65_536, 2
    b = BatchSampler([p] * n, precision="fp32", use_torch_allocator=False)
    q = torch.full((n, steps), float("nan"), dtype=torch.float64, device="cuda")
    b.sample(None, steps, 17, qoi=q)
    b.check_status()
    assert bool(torch.isfinite(q).all())
    s = Sampler(p, precision="fp32", coarse_max_n=31)
    for c in (0, 1, 32_768, 65_534, 65_535):
        x, qs = s.zeros(), torch.zeros(steps, dtype=torch.float64, device="cuda")
        s.sample(x, steps, 17, chain=c, qoi=qs)
        assert torch.equal(qs, q[c])
        assert torch.equal(b.get_state(c, s.zeros()), x)
    s.close()
    b.close()
