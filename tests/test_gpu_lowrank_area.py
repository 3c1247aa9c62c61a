"""Low-rank steps of area observations (FP32): thousands of rows of G, several per thread of a
chain's cluster.  The chain agrees with the FP64 oracle at the FP32 tolerance (2e-4 of the rms),
repeats bit for bit, has the same bits whichever kernels run the grids below the finest (the
streaming ones leave the state, the tile ones partial sums for the low-rank step), and in a batch
with a chain of few rows both have the bits of their solo runs."""
import numpy as np
import pytest

import oracle
from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu


# rows of G: just above one per thread on the finest grid; far above it on two grids, a full
# Gamma; more observations than a thread keeps coefficients of in registers
@pytest.mark.parametrize("n,m,ball,full", [(255, 3, 0.06, False), (511, 5, 0.05, True), (255, 20, 0.05, False)])
def test_area_observations(n, m, ball, full):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import BatchSampler, Sampler
    build.build()
    p = inputs.make_problem("area", 2, n, kappa2_seed=3, m=m, obs_seed=5, qoi_cells=16, ball_radius=ball)
    if full:
        a = np.random.default_rng(5).normal(size=(m, m))
        p.Gamma = 1e-4 * (np.eye(m) + 0.1 * a @ a.T / m)
    o = oracle.Oracle(p.dim, p.n, p.n_levels, kappa2=p.kappa2, obs_site=p.obs_site, obs_w=p.obs_w, Gamma=p.Gamma, y=p.y,
                      qoi_site=p.qoi_site, qoi_w=p.qoi_w)
    xo, qo = o.sample(2, 13)
    s = Sampler(p, precision="fp32", coarse_max_n=31, band_min_n=127)
    q = torch.zeros(2, dtype=torch.float64, device="cuda")

    def run(step_seed=13):
        x = s.zeros()
        s.sample(x, 2, step_seed, qoi=q)
        return x

    first = run()
    rms = np.sqrt(np.mean(xo ** 2))
    assert np.abs(first.double().cpu().numpy() - xo).max() <= 2e-4 * rms
    assert np.abs(q.cpu().numpy() - qo).max() <= 2e-4 * rms
    for _ in range(10):
        assert torch.equal(run(), first)
    for band in (1 << 20, 63):
        s.set_band_min_n(band)
        assert torch.equal(run(), first)
    few = inputs.make_problem("few", 2, n, kappa2_seed=4, m=2, obs_seed=6, qoi_cells=8)
    t = Sampler(few, precision="fp32", coarse_max_n=31)
    xf = t.zeros()
    t.sample(xf, 2, 13, chain=1)
    b = BatchSampler([p, few], precision="fp32", band_min_n=127)
    xs = b.zeros()
    b.sample(xs, 2, 13)
    assert torch.equal(xs[0], first) and torch.equal(xs[1], xf)
