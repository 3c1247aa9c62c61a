"""Low-rank steps of the streamed grids whose rows of G take several CTAs (one cluster per
chain): every CTA reads the state at the observation entries that others update, so the result
must not depend on their timing.  A chain and a mixed batch repeat bit for bit, and the chain
agrees with the FP64 oracle at the FP32 tolerance (2e-4 of the rms)."""
import numpy as np
import pytest

import oracle
from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,ball", [(16, None), (37, None), (3, 0.06)])
def test_many_rows_of_g(m, ball):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import BatchSampler, Sampler
    build.build()
    p = inputs.make_problem("lr", 2, 255, kappa2_seed=3, m=m, obs_seed=5, qoi_cells=16, ball_radius=ball)
    o = oracle.Oracle(p.dim, p.n, p.n_levels, kappa2=p.kappa2, obs_site=p.obs_site, obs_w=p.obs_w, Gamma=p.Gamma, y=p.y,
                      qoi_site=p.qoi_site, qoi_w=p.qoi_w)
    xo, _ = o.sample(2, 13)
    s = Sampler(p, precision="fp32", coarse_max_n=31)
    first = None
    for _ in range(20):
        x = s.zeros()
        s.sample(x, 2, 13)
        first = x.clone() if first is None else first
        assert torch.equal(x, first)
    rms = np.sqrt(np.mean(xo ** 2))
    assert np.abs(first.double().cpu().numpy() - xo).max() <= 2e-4 * rms
    small = inputs.make_problem("lr2", 2, 127, kappa2_seed=4, m=2, obs_seed=6, qoi_cells=8)
    b = BatchSampler([p, small, p], precision="fp32")
    ref = None
    for _ in range(10):
        xs = b.zeros()
        b.sample(xs, 2, 13)
        ref = [v.clone() for v in xs] if ref is None else ref
        assert all(torch.equal(u, v) for u, v in zip(xs, ref))
    assert torch.equal(ref[0], first)
