"""The QoI series against the oracle's, with one CTA per chain and with several (from 1025 sites on),
on every path that ends in the QoI launch: Gibbs handles, the coarse kernel alone, the fused
2D cycle, the general path, batches of chains with different numbers of sites.  The QoI is an
average of the state, so the tolerances are the states' (FP64 1e-11, FP32 2e-4 of the rms)."""
import numpy as np
import pytest

import oracle
from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 2e-4}
STEPS = 4


def _series(p, gibbs=False, chain=0):
    o = oracle.Oracle(p.dim, p.n, p.n_levels, kappa2=p.kappa2, kappa2_const=p.kappa2_const, disc=p.disc,
                      obs_site=p.obs_site, obs_w=p.obs_w, Gamma=p.Gamma, y=p.y, qoi_site=p.qoi_site, qoi_w=p.qoi_w)
    x, q = o.sample(STEPS, 21, chain=chain, gibbs=gibbs) if gibbs else o.sample(STEPS, 21, chain=chain)
    return np.sqrt(np.mean(x ** 2)), q


# (cells + 1)^dim QoI sites: 9 (one CTA), 1089 (two), 4913 and 66 049 (the most, 16)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,n,m,cells,disc,gibbs", [(2, 255, 8, 32, 1, True), (2, 511, 4, 256, 0, True),
                                                      (2, 31, 5, 2, 0, False), (2, 63, 5, 32, 0, False),
                                                      (2, 511, 8, 256, 0, False), (3, 31, 4, 16, 0, False)])
def test_series_of_a_chain(dim, n, m, cells, disc, gibbs, precision):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    p = inputs.make_problem("q", dim, n, kappa2_seed=None if disc else 5, kappa2_const=100.0, m=m, obs_seed=4, disc=disc,
                            qoi_cells=cells)
    rms, want = _series(p, gibbs)
    s = Sampler(p, precision=precision, gibbs=gibbs)
    q = torch.full((STEPS,), float("nan"), dtype=torch.float64, device="cuda")
    s.sample(s.zeros(), STEPS, 21, qoi=q)
    assert np.abs(q.cpu().numpy() - want).max() <= TOL[precision] * rms
    s.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_series_of_a_batch(precision):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import BatchSampler
    build.build()
    ps = [inputs.make_problem("q", 2, n, kappa2_seed=5 + c, m=4, obs_seed=4 + c, qoi_cells=cells)
          for c, (n, cells) in enumerate([(63, 2), (255, 128), (127, 32), (31, 16)])]
    b = BatchSampler(ps, precision=precision)
    q = torch.full((len(ps), STEPS), float("nan"), dtype=torch.float64, device="cuda")
    b.sample(b.zeros(), STEPS, 21, qoi=q)
    for c, p in enumerate(ps):
        rms, want = _series(p, chain=c)
        assert np.abs(q[c].cpu().numpy() - want).max() <= TOL[precision] * rms
    b.close()
