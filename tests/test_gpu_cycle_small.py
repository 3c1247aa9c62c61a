"""The one-CTA kernel of a W-cycle's small grids where its plan changes: FP32 handles, coarsest grids
of 1, 9, 49 and 225 unknowns (gain matrix in shared memory, in global memory, triangular solves), as many
observations as a handle takes (the normals drawn at the start run out, so that phases of one
visit use both sources), several sweeps.  Against the FP64 oracle at the parity tolerances (FP32
2e-4 of the rms; FP64 as derived in test_gpu_wcycle.py)."""
import numpy as np
import pytest

from paper_2407_12149_gb300 import inputs
from tests.test_gpu_parity import _check32, _check64, _run_gpu
from tests.test_gpu_wcycle import _tol

import oracle

pytestmark = pytest.mark.gpu


def _oracle(p, nu, steps, **kw):
    o = oracle.Oracle(p.dim, p.n, p.n_levels, kappa2=p.kappa2, kappa2_const=p.kappa2_const, nu1=nu, nu2=nu,
                      obs_site=p.obs_site, obs_w=p.obs_w, Gamma=p.Gamma, y=p.y, qoi_site=p.qoi_site, qoi_w=p.qoi_w,
                      disc=p.disc, gamma=2)
    return o.sample(steps, 31, **kw)


# disc, n, coarsest n, m, nu
FP32 = [(0, 31, 1, 5, 1), (0, 63, 3, 16, 1), (0, 127, 7, 0, 1), (0, 63, 15, 64, 1), (0, 31, 3, 9, 2), (1, 63, 1, 8, 1)]
FP64 = [(2, 63, 3, 8, 1), (2, 63, 7, 8, 1), (2, 63, 1, 64, 1), (2, 31, 15, 5, 1), (0, 63, 7, 64, 1), (0, 127, 1, 64, 2)]


@pytest.mark.parametrize("precision,disc,n,coarsest,m,nu", [("fp32", *c) for c in FP32] + [("fp64", *c) for c in FP64])
def test_small_grids_match_oracle(precision, disc, n, coarsest, m, nu):
    import torch
    from paper_2407_12149_gb300 import build
    from paper_2407_12149_gb300.mgmc import Sampler
    build.build()
    p = inputs.make_problem("s", 2, n, n_levels=inputs.levels_for(n, coarsest), kappa2_seed=None if disc else 3,
                            kappa2_const=100.0, m=m, obs_seed=4, disc=disc, sigma2=1e-4 if disc == 0 else 1.5e-6,
                            qoi_cells=(n + 1) // 4)
    steps = 3
    xo, qo = _oracle(p, nu, steps, chain=2)
    s = Sampler(p, precision=precision, gamma=2, nu1=nu, nu2=nu)
    xg, qg = _run_gpu(torch, s, p, steps, 31, chain=2)
    if precision == "fp32":
        _check32(xg, xo)
        assert np.abs(qg - qo).max() <= 2e-4 * np.sqrt(np.mean(xo ** 2))
    else:
        _check64(xg, xo, _tol(p))
        _check64(qg, qo, _tol(p))
    s.check_status()
    s.close()
