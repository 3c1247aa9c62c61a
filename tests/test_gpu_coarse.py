"""The one-CTA coarse-grid kernel at the edges of its plan, per site against the FP64 oracle:
every chain below runs (almost) all its grids inside that kernel.

Covered: coarsest grids on both sides of the gain-matrix limit (1, 9, 49, 225 unknowns), one
grid only, observation counts around the four lanes per observation and the register rows of
G (0, 1, 5, 17, 37), a full Gamma, several sweeps per grid (normals drawn inside the phase) and
none, a 63^2 FP32 grid (the two sweeps share the normals' place), Q1 grids, 3D.  Tolerances as
in the parity tests: FP64 1e-11 of max(|x|, rms) per site, FP32 2e-4 of the rms.
"""
import numpy as np
import pytest

import oracle
from paper_2407_12149_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    # dim, n, n_levels, m, nu1, nu2, disc, full Gamma
    (2, 31, 5, 5, 1, 1, 0, False),
    (2, 31, 4, 0, 1, 1, 0, False),
    (2, 31, 3, 17, 1, 1, 0, True),
    (2, 31, 2, 37, 1, 1, 0, False),
    (2, 15, 1, 5, 1, 1, 0, True),
    (2, 3, 2, 1, 1, 1, 0, False),
    (2, 63, 6, 17, 1, 1, 0, False),
    (2, 63, 4, 5, 2, 1, 0, True),
    (2, 31, 4, 5, 0, 2, 0, False),
    (2, 31, 5, 5, 3, 0, 1, False),
    (3, 7, 3, 5, 1, 1, 0, False),
    (3, 15, 3, 17, 1, 1, 0, False),
    (3, 7, 2, 37, 2, 2, 0, True),
]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(v) for v in c))
def test_coarse_kernel_matches_oracle(case, precision):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    dim, n, levels, m, nu1, nu2, disc, full = case
    p = inputs.make_problem("coarse", dim, n, n_levels=levels, kappa2_seed=None if disc else 3, m=m, obs_seed=4,
                            qoi_cells=2, disc=disc)
    if full:
        a = np.random.default_rng(5).normal(size=(m, m))
        p.Gamma = 1e-4 * (np.eye(m) + 0.1 * a @ a.T / m)
    o = oracle.Oracle(p.dim, p.n, p.n_levels, nu1=nu1, nu2=nu2, kappa2=p.kappa2, kappa2_const=p.kappa2_const,
                      obs_site=p.obs_site, obs_w=p.obs_w, Gamma=p.Gamma, y=p.y, qoi_site=p.qoi_site, qoi_w=p.qoi_w,
                      disc=p.disc)
    xo, qo = o.sample(3, 11)
    s = Sampler(p, precision=precision, nu1=nu1, nu2=nu2)
    x = s.zeros()
    q = torch.zeros(3, dtype=torch.float64, device="cuda")
    s.sample(x, 3, 11, qoi=q)
    s.check_status()
    xg = x.double().cpu().numpy()
    rms = np.sqrt(np.mean(xo ** 2))
    err = np.abs(xg - xo)
    if precision == "fp64":
        assert np.all(err <= 1e-11 * np.maximum(np.abs(xo), rms)), err.max() / rms
        assert np.allclose(q.cpu().numpy(), qo, rtol=1e-11, atol=1e-11 * rms)
    else:
        assert err.max() <= 2e-4 * rms, err.max() / rms
    s.close()
